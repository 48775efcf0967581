"""Reverse steps over columns of every length around the load phases (full
phases and one shorter one): within 1e-12 of the oracle's adjoint, and the same
bits with int32 rows and with 16-bit row codes."""
import numpy as np
import pytest

from oracle_problem import build

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


def T(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# columns hold about n entries, more and fewer near the boundary: the lengths of
# one plan run over several remainders of phases of 8, 10, 12 and 16
@pytest.mark.parametrize("d,Kg,n", [(2, 9, 2), (2, 30, 3), (2, 30, 7), (2, 41, 9), (2, 30, 11),
                                    (2, 30, 15), (2, 23, 17), (2, 41, 24), (2, 23, 37),
                                    (3, 11, 51)])
def test_column_lengths(rb, orc, d, Kg, n):
    p = build(orc, d, Kg, 2, seed=n)
    g = np.random.default_rng(n)
    idx = orc.knn_kdtree(p.xyz, p.interior, n)
    w = g.standard_normal(idx.shape) / n
    dLdu = g.standard_normal(p.N)
    K, dt = 13, 0.37
    gf, gg, l0 = orc.adjoint(w, idx, p.interior, p.N, dLdu, K, dt)
    got = []
    for pack in (0, rb.RBFFD_PACK_IDX32):
        plan = rb.Plan(T(p.xyz), T(p.is_bnd), T(p.interior), T(idx), T(w), pack)
        got.append([t.cpu().numpy() for t in plan.adjoint(T(dLdu), K, dt)])
        plan.destroy()
    for a, b, o in zip(got[0], got[1], (gf, gg, l0)):
        assert np.array_equal(a, b)
        assert np.max(np.abs(a - o)) <= 1e-12 * max(np.max(np.abs(o)), 1e-300)
