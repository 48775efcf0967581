"""The power iteration's launches (plans without Neumann nodes: one persistent launch, or linked
ones of up to 64 iterations) against the oracle's iteration: one, two and many iterations, about
a launch's 64 too (the norms come from different kernels), stencil sizes
with and without a compiled kernel, node orders, int32 indices, one partial slice; vectors with
no direction or with NaN are refused."""
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


@pytest.mark.parametrize("d,Kg,m,n,flags", [(2, 60, 2, 12, 0), (2, 45, 4, 30, 64),
                                            (2, 45, 4, 31, 2), (2, 30, 4, 30, 32),
                                            (2, 100, 2, 12, 64), (2, 160, 4, 31, 64),
                                            (2, 40, 6, 56, 0), (3, 12, 4, 70, 0),
                                            (3, 12, 4, 70, 64), (2, 4, 1, 6, 0)])
def test_radius_equals_the_oracles(rb, orc, d, Kg, m, n, flags):
    p = build(orc, d, Kg, m, seed=17, n=n)
    plan = rb.Plan(T(p.xyz), T(p.is_bnd), T(p.interior), T(p.idx), T(p.w), flags, 3)
    v0 = gen.random_vector(p.NI, 5)
    # each iteration's sums of n + N terms round within (n + N) 2^-53 of the exact ones and
    # the radius is stationary to first order; the repository's bound is 1e-9
    for iters in (1, 2, 3, 63, 65, 200):
        rho = orc.power_rho(p.w, p.idx, p.interior, p.N, v0, iters)
        for scale in (1.0, 1e-100, 1e100):
            got = plan.stable_dt(T(v0 * scale), iters, 1.05)[1]
            assert abs(got - rho) <= 1e-9 * rho
    # no direction: zero, NaN, squares that underflow or overflow
    for bad in (np.zeros(p.NI), np.full(p.NI, np.nan), v0 * 1e-200, v0 * 1e200):
        with pytest.raises(rb.RbffdError):
            plan.stable_dt(T(bad), 5)


@pytest.mark.parametrize("n,flags", [(12, 0), (12, 64), (17, 64), (30, 128)])
def test_waits_that_run_out_do_not_change_the_radius(rb, orc, n, flags):
    """Withheld arrivals and decisions, and limits about as long as a wait takes, so that any
    launch of the linked form may fall short: the radius is the same."""
    p = build(orc, 2, 100, 2 if n < 30 else 4, seed=17, n=n)
    plan = rb.Plan(T(p.xyz), T(p.is_bnd), T(p.interior), T(p.idx), T(p.w), flags, 3)
    v0 = gen.random_vector(p.NI, 5)
    for iters in (1, 2, 65, 200):
        rho = orc.power_rho(p.w, p.idx, p.interior, p.N, v0, iters)
        waits = [(20.0, 1), (0.0, 0)] + [(ms, 0) for ms in (2e-4, 5e-4, 1e-3, 2e-3, 4e-3) * 4]
        for wait in waits:
            plan.set_wait(*wait)
            assert abs(plan.stable_dt(T(v0), iters, 1.05)[1] - rho) <= 1e-9 * rho, wait


@pytest.mark.parametrize("flags", [0, 64, 2])
@pytest.mark.parametrize("big", [1e3, 1e5, 1e8, 1e40])
def test_radius_far_below_the_row_sums(rb, orc, flags, big):
    """A huge weight on a boundary node leaves W_II, and so the radius, as it was, but not the
    largest row sum, by which the linked launch scales its iterations."""
    p = build(orc, 2, 60, 2, seed=17, n=12)
    row = next(r for r in range(p.NI) if p.is_bnd[p.idx[r]].any())
    w = p.w.copy()
    j = int(np.nonzero(p.is_bnd[p.idx[row]])[0][0])
    w[row, j] = big * np.abs(p.w).sum(1).max()
    plan = rb.Plan(T(p.xyz), T(p.is_bnd), T(p.interior), T(p.idx), T(w), flags, 3)
    v0 = gen.random_vector(p.NI, 5)
    for iters in (2, 8, 64, 128, 200, 256):
        rho = orc.power_rho(p.w, p.idx, p.interior, p.N, v0, iters)
        assert abs(plan.stable_dt(T(v0), iters, 1.05)[1] - rho) <= 1e-9 * rho
