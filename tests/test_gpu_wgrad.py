"""The weight gradient accumulated over groups of up to eight steps, at every group length and
remainder (segments of 1, 7, 8, 9, 17 and K steps; K = 0), for stencil sizes with and without a
compiled replay, 16-bit and 32-bit indices and one partial slice, against the oracle; every
spacing gives the same bits."""
import numpy as np
import pytest

import rbffd_inputs as gen
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


def T(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("d,Kg,m,n,flags", [(2, 40, 2, 12, 0), (2, 30, 4, 30, 32),
                                            (2, 70, 4, 31, 64), (2, 4, 1, 6, 0),
                                            (3, 10, 4, 70, 2)])
def test_weight_gradient_for_every_spacing(rb, orc, d, Kg, m, n, flags):
    p = build(orc, d, Kg, m, seed=23, n=n)
    plan = rb.Plan(T(p.xyz), T(p.is_bnd), T(p.interior), T(p.idx), T(p.w), flags, 3)
    dt = 0.5 * 2.0 / np.abs(p.w).sum(1).max()
    dLdu = gen.random_vector(p.N, 8)
    for K in (0, 1, 19):
        # u^0, u^1, ... by the plan itself (their parity is tested elsewhere)
        us = [p.u0.copy()]
        for _ in range(K):
            u = T(us[-1])
            plan.solve_explicit(T(p.f), u, dt, 1)
            us.append(u.cpu().numpy())
        ref = orc.adjoint_w(p.w, p.idx, p.interior, p.f, p.u0, dLdu, K, dt)
        first = None
        for every in (1, 2, 7, 8, 9, 17, max(K, 1)):
            ckpt = np.stack(us[0:max(K, 1):every])
            got = plan.adjoint_w(T(p.f), T(ckpt), every, T(dLdu), K, dt)
            for a, b in zip(got[:3], ref[:3]):
                scale = np.max(np.abs(b)) if np.any(b) else 1.0
                assert np.max(np.abs(a.cpu().numpy() - b)) <= 1e-12 * scale
            if first is None:
                first = got
            assert all(torch.equal(a, b) for a, b in zip(got, first)), (K, every)
