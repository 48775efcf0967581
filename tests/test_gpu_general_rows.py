"""Steps of stencil sizes that no kernel is compiled for: every length of the last
load phase, in the tuned launch, one launch a step, the persistent and the batched
launch, FP64 within 1e-12 max|u| of the oracle and the launches bit for bit alike."""
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


@pytest.mark.parametrize("pack32", [False, True])
@pytest.mark.parametrize("d,Kg,n", [(2, 9, 2), (2, 40, 5), (2, 23, 14), (2, 40, 15), (2, 40, 16),
                                    (2, 40, 17), (2, 23, 29), (2, 23, 33), (2, 23, 44),
                                    (2, 23, 47), (3, 11, 63)])
def test_general_rows(rb, orc, d, Kg, n, pack32):
    p = build(orc, d, Kg, 2, seed=n)
    g = np.random.default_rng(n)
    idx = orc.knn_kdtree(p.xyz, p.interior, n)
    # diagonally dominant rows, so the steps stay bounded
    w = 0.5 * g.random(idx.shape) / n
    w[:, 0] = -1.0
    f = g.standard_normal(p.NI)
    u0 = g.standard_normal(p.N)
    K, dt = 41, 0.8
    ou = orc.solve_explicit(w, idx, p.interior, f, u0, dt, K, 0.0)[0]
    pack = rb.RBFFD_PACK_IDX32 if pack32 else 0
    got = []
    for flags in (pack | rb.RBFFD_LAUNCH_AUTO, pack, pack | rb.RBFFD_LAUNCH_PERSISTENT):
        plan = rb.Plan(T(p.xyz), T(p.is_bnd), T(p.interior), T(idx), T(w), flags)
        u = T(u0)
        plan.solve_explicit(T(f), u, dt, K)
        got.append(u.cpu().numpy())
    batch = rb.Batch([plan])
    for shape in ((1, 1, 1024), (1, 1, 256), (2, 2, 512)):
        batch.set_shape(*shape)
        us = [T(u0)]
        batch.solve([T(f)], us, [dt], [K], [0.0])
        got.append(us[0].cpu().numpy())
    batch.destroy()
    plan.destroy()
    for a in got:
        assert np.max(np.abs(a - ou)) <= 1e-12 * np.max(np.abs(ou))
        assert np.array_equal(a, got[0])
