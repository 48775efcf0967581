"""Supports where the FP32-ordered search can go wrong, against the oracle's kd-tree
(bit-exact, as every support test): ties that only FP64 keys and indices decide, near-ties
below FP32 resolution, cells too dense for a warp's arrays, balls that grow past the node
set, thin and coarse grids, n at its limits, and candidate masks."""
import numpy as np
import pytest

import rbffd_inputs as gen

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


def _points(kind):
    rng = np.random.default_rng(5)
    if kind == "grid2":          # every distance tied many times
        return gen.grid_points(33, 2)
    if kind == "grid3":
        return gen.grid_points(11, 3)
    if kind == "near_ties":      # a grid moved by less than FP32 can tell
        return gen.grid_points(40, 2) + rng.uniform(-1, 1, (2, 1600)) * 1e-10
    if kind == "uniform2":
        return gen.random_points(3001, 2, 7)
    if kind == "uniform3":
        return gen.random_points(4003, 3, 8)
    if kind == "line":           # 1D, and a 2D set on a line
        return gen.random_points(2500, 1, 9)
    if kind == "long_line":      # more cells an axis than FP32 coordinates allow
        return gen.random_points(40000, 1, 10)
    if kind == "collinear2":
        x = np.sort(rng.uniform(0, 1, 700))
        return np.stack([x, 3.0 * x])
    if kind == "clusters":       # thousands of nodes in a few cells, and a sparse rest
        c = rng.uniform(0, 1, (2, 900)) * 1e-4 + 0.5
        return np.concatenate([c, gen.random_points(300, 2, 11)], axis=1)
    if kind == "duplicates":
        p = gen.random_points(400, 2, 12)
        return np.concatenate([p, p, p], axis=1)
    if kind == "thin":           # 3D, one axis a hundredth of the others
        p = gen.random_points(5000, 3, 13)
        p[1] *= 0.01
        return p
    assert kind == "shifted"     # far from the origin: FP64 coordinates lose bits
    return gen.random_points(2000, 2, 14) * 1e-3 + 1e4


@pytest.mark.parametrize("n", [1, 2, 13, 31, 70, 128])
@pytest.mark.parametrize("kind", ["grid2", "grid3", "near_ties", "uniform2", "uniform3", "line",
                                  "long_line", "collinear2", "clusters", "duplicates", "thin",
                                  "shifted"])
def test_supports_equal_the_kdtree(rb, orc, kind, n):
    xyz = np.ascontiguousarray(_points(kind))
    N = xyz.shape[1]
    centres = np.random.default_rng(n).permutation(N)[:1500].astype(np.int32)
    ref = orc.knn_kdtree(xyz, centres, n)
    X, C = torch.from_numpy(xyz).cuda(), torch.from_numpy(centres).cuda()
    assert np.array_equal(rb.rbffd_knn(X, C, n).cpu().numpy(), ref)
    mask = (np.arange(N) % 3 != 0).astype(np.uint8)
    ref = orc.knn_kdtree(xyz, centres, n, cand=mask)
    got = rb.rbffd_knn_masked(X, torch.from_numpy(mask).cuda(), C, n)
    assert np.array_equal(got.cpu().numpy(), ref)


@pytest.mark.parametrize("d,N", [(1, 1), (2, 3), (3, 128), (2, 129)])
def test_supports_of_the_whole_set(rb, orc, d, N):
    n = min(N, 128)
    xyz = gen.random_points(N, d, N)
    centres = np.arange(N, dtype=np.int32)
    got = rb.rbffd_knn(torch.from_numpy(xyz).cuda(), torch.from_numpy(centres).cuda(), n)
    assert np.array_equal(got.cpu().numpy(), orc.knn_kdtree(xyz, centres, n))


def test_too_few_candidates_are_refused(rb):
    xyz = torch.from_numpy(gen.random_points(50, 2, 3)).cuda()
    mask = torch.zeros(50, dtype=torch.uint8, device="cuda")
    mask[:5] = 1
    with pytest.raises(rb.RbffdError):
        rb.rbffd_knn_masked(xyz, mask, torch.arange(50, dtype=torch.int32, device="cuda"), 7)
