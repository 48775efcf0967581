"""rbffd_apply at the edges of its tiles (32 rows of n entries; even and odd n, eight entries
at a time), with a partial last tile, past the tiles' largest n and at views that start off a
16-byte boundary, against the oracle's sums."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_12878_gb300 import build as nvbuild
    nvbuild.build()
    import paper_2502_12878_gb300 as m
    m.lib()
    return m


@pytest.mark.parametrize("n", [1, 3, 8, 9, 12, 16, 17, 31, 32, 33, 57, 64, 71, 128, 146, 586, 587])
@pytest.mark.parametrize("rows", [1, 31, 33, 4 * 32 + 5, 5000])
@pytest.mark.parametrize("skip", [0, 1])
def test_apply_tiles(rb, orc, rows, n, skip):
    rng = np.random.default_rng(rows * 1000 + n)
    N = rows + 40
    # skip = 1: the call gets the array from its second row on, which starts off a 16-byte
    # boundary unless n is a multiple of 4
    w = rng.standard_normal((rows + 1, n))
    idx = rng.integers(0, N, (rows + 1, n)).astype(np.int32)
    u = rng.standard_normal(N)
    W, X = torch.from_numpy(w).cuda(), torch.from_numpy(idx).cuda()
    got = rb.rbffd_apply(W[skip:], X[skip:], torch.from_numpy(u).cuda()).cpu().numpy()
    ref = orc.apply(np.ascontiguousarray(w[skip:]), np.ascontiguousarray(idx[skip:]), u)
    scale = np.maximum(np.abs(ref), (np.abs(w[skip:]) * np.abs(u[idx[skip:]])).sum(1))
    assert np.all(np.abs(got - ref) <= 1e-12 * scale)


@pytest.mark.parametrize("n", [196, 197, 199, 200, 301, 400])
def test_long_rows_by_either_kernel(rb, n):
    """Rows of a length of which few tiles fit an SM go to one kernel or the other by their
    number: each row's chain, and so its bits, are the same."""
    g = torch.Generator("cuda").manual_seed(n)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    fit = (227 * 1024) // (32 * n * 12 + 1024)
    for rows in (16 * 5 * sms * fit // 32 * 32, 16 * 5 * sms * fit // 32 * 32 + 1, 40000):
        w = torch.randn((rows, n), generator=g, device="cuda", dtype=torch.float64)
        idx = torch.randint(0, rows, (rows, n), generator=g, device="cuda", dtype=torch.int32)
        u = torch.randn(rows, generator=g, device="cuda", dtype=torch.float64)
        cut = rows // 64 * 32
        parts = [rb.rbffd_apply(w[a:b], idx[a:b], u) for a, b in ((0, cut), (cut, rows))]
        assert torch.equal(rb.rbffd_apply(w, idx, u), torch.cat(parts))
