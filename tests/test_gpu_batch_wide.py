"""Teams of many blocks at 64 registers a thread (one 1024-thread block or two
512-thread blocks per SM): the iterate gathered through L1 between the other
blocks' writes.  The columns are those of the 256-thread blocks, bit for bit
(the same fma chain per row), and the oracle's to 1e-12 max|u|."""
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


def T(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# (d, Kg, m): stencils of 12, 30 and 56, of another size (20 in 3D), and a
# domain with fewer slices than one block has warps
@pytest.mark.parametrize("d,Kg,m", [(2, 70, 2), (2, 61, 4), (2, 66, 6), (3, 13, 2), (2, 9, 4)])
def test_wide_teams(rb, orc, d, Kg, m):
    p = build(orc, d, Kg, m, seed=5)
    dt = 0.9 * orc.stable_dt(p.w, p.idx, p.interior, p.N, gen.random_vector(p.NI, 3), 200)
    plan = rb.Plan(T(p.xyz), T(p.is_bnd), T(p.interior), T(p.idx), T(p.w))
    batch = rb.Batch([plan])
    ref = None
    for shape in ((1, 1, 256), (1, 1, 1024), (2, 2, 512), (2, 1, 512)):
        batch.set_shape(*shape)
        us = [T(p.u0)]
        batch.solve([T(p.f)], us, [dt], [301], [0.0])
        got = us[0].cpu().numpy()
        if ref is None:
            ref = got
            ou = orc.solve_explicit(p.w, p.idx, p.interior, p.f, p.u0, dt, 301, 0.0)[0]
            assert np.max(np.abs(got - ou)) <= 1e-12 * np.max(np.abs(ou))
        assert np.array_equal(got, ref)
    batch.destroy()
    plan.destroy()
