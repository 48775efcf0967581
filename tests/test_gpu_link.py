"""The linked launch (blocks exchange rows and decisions through tagged words, no grid barrier)
against graph-replayed steps, bit for bit, and against its own stop rule: shares of one, two and
more slices than warps, fewer slices than SMs, one partial slice, every way a run can end and
how many steps after the start, both block sizes, both arithmetics, and tags that start over."""
import numpy as np
import pytest

import rbffd_inputs as gen
from oracle_problem import build

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda"


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
    return torch.from_numpy(np.ascontiguousarray(x)).to(DEV)


def _plans(rb, p, threads, order=0):
    ref = rb.Plan(T(p.xyz), T(p.is_bnd), T(p.interior), T(p.idx), T(p.w), order, 3)
    lnk = rb.Plan(T(p.xyz), T(p.is_bnd), T(p.interior), T(p.idx), T(p.w),
                  order | rb.RBFFD_LAUNCH_RESIDENT, 3)
    lnk.set_block(threads)
    return ref, lnk


def _linked(shape):
    return shape[1] == -1 and shape[0] >= 8


# d, Kg, m, n, order: 9 rows; 2 blocks of one slice; fewer slices than SMs; 2-3 slices a block;
# 8; 18 (more than 512 threads have warps for); 3D; a random order (every support scattered)
CASES = [(2, 4, 1, 6, 0), (2, 9, 2, 12, 0), (2, 60, 2, 13, 0), (2, 100, 2, 12, 0),
         (2, 200, 4, 30, 0), (2, 300, 4, 30, 0), (2, 120, 6, 56, 0), (3, 22, 4, 70, 0),
         (2, 90, 2, 17, 0), (2, 70, 4, 31, 2)]


@pytest.mark.parametrize("threads", [512, 1024])
@pytest.mark.parametrize("d,Kg,m,n,order", CASES)
def test_same_bits_as_graph_steps(rb, orc, d, Kg, m, n, order, threads):
    p = build(orc, d, Kg, m, seed=7, n=n)
    ref, lnk = _plans(rb, p, threads, order)
    f, u0 = T(p.f), T(p.u0)
    dt = 0.5 * 2.0 / np.abs(p.w).sum(1).max()
    try:
        lnk.solve_explicit(f, u0.clone(), dt, 1)
    except rb.RbffdError as e:     # a block size not compiled for this n
        assert e.code == rb.RBFFD_ERR_CAPACITY and threads == 1024
        return
    for K in (1, 2, 5, 6, 7, 40, 333):
        a, b = u0.clone(), u0.clone()
        ra = ref.solve_explicit(f, a, dt, K)
        rl = lnk.solve_explicit(f, b, dt, K)
        assert ra == rl and torch.equal(a, b), K
    # stops by tolerance: at the first step, within and beyond the steps a block may be ahead
    hist = []
    u = u0.clone()
    for k in range(12):
        hist.append(ref.solve_explicit(f, u, dt, 1)[2])
    for k in (0, 1, 3, 4, 5, 6, 9, 11):
        tol = np.nextafter(hist[k], np.inf)
        a, b = u0.clone(), u0.clone()
        ra = ref.solve_explicit(f, a, dt, 5_000_000_000 if k == 9 else 200, tol)
        rl = lnk.solve_explicit(f, b, dt, 5_000_000_000 if k == 9 else 200, tol)
        assert ra == rl and torch.equal(a, b), k
    # defect correction: FP32 inner steps, stopped by the cap and by rho_in
    for K_in, rho in ((7, 0.0), (400, 0.9)):
        a, b = u0.clone(), u0.clone()
        ra = ref.solve_dc(f, a, dt, 1e-12, 3, K_in, rho)
        rl = lnk.solve_dc(f, b, dt, 1e-12, 3, K_in, rho)
        assert ra == rl and torch.equal(a, b)
    assert _linked(lnk.stats()[3]) or threads == 512 and n >= 56


@pytest.mark.parametrize("d,Kg,m,n", [(2, 9, 2, 12), (2, 30, 1, 6), (2, 75, 2, 12), (2, 110, 1, 6)])
def test_thousands_of_stops(rb, orc, d, Kg, m, n):
    """Blocks learn of a stop at their own times, and a block that is a step further than its
    neighbours waits for rows that are never written: it has to find the stop instead of running
    out of its wait.  Short steps (small n, FP32 too) on 2 to 152 blocks, stopped some 2,000 times
    by tolerance and 500 by rho_in at every distance from the start."""
    p = build(orc, d, Kg, m, seed=7, n=n)
    ref, lnk = _plans(rb, p, 0)
    f, u0 = T(p.f), T(p.u0)
    dt = 0.5 * 2.0 / np.abs(p.w).sum(1).max()
    hist, its = [], []
    u = u0.clone()
    for k in range(40):
        hist.append(ref.solve_explicit(f, u, dt, 1)[2])
        its.append(u.clone())
    # the steps whose residual is the smallest so far: where a tolerance above it stops
    stops = [k for k in range(40) if all(hist[k] < r for r in hist[:k])]
    v = torch.empty_like(u0)
    for rep in range(-(-2000 // len(stops))):
        for k in stops:
            v.copy_(u0)
            got = lnk.solve_explicit(f, v, dt, 100000, np.nextafter(hist[k], np.inf))
            assert got == (rb.RBFFD_OK, k + 1, hist[k])
            assert torch.equal(v, its[k])
    assert _linked(lnk.stats()[3])
    for rho in np.linspace(0.999, 0.5, 25):
        v.copy_(u0)
        want = ref.solve_dc(f, v, dt, 0.0, 2, 3000, rho)
        for rep in range(10):
            w = u0.clone()
            assert lnk.solve_dc(f, w, dt, 0.0, 2, 3000, rho) == want
            assert torch.equal(v, w)


def test_nonfinite_and_diverging_runs_end(rb, orc):
    p = build(orc, 2, 80, 2, seed=9)
    ref, lnk = _plans(rb, p, 0)
    dt = 0.5 * 2.0 / np.abs(p.w).sum(1).max()
    bad = p.f.copy()
    bad[1234] = np.nan
    for plan in (ref, lnk):
        with pytest.raises(rb.RbffdError) as e:
            plan.solve_explicit(T(bad), T(p.u0), dt, 100)
        assert e.value.code == rb.RBFFD_ERR_NONFINITE
        with pytest.raises(rb.RbffdError) as e:
            plan.solve_explicit(T(p.f), T(p.u0), 60 * dt, 4000)
        assert e.value.code == rb.RBFFD_ERR_DIVERGED
    a, b = T(p.u0), T(p.u0)      # and the plan solves on
    assert ref.solve_explicit(T(p.f), a, dt, 50) == lnk.solve_explicit(T(p.f), b, dt, 50)
    assert torch.equal(a, b)


@pytest.mark.parametrize("flag", ["RBFFD_LAUNCH_RESIDENT", "RBFFD_LAUNCH_FAR"])
def test_limits_shorter_than_the_copies(rb, orc, flag):
    """A wait limit below what the planes' copies into shared memory take: a block that gives up
    still waits for them before it leaves.  Each solve ends with its result or as timed out."""
    p = build(orc, 2, 120, 4, seed=11)
    dt = 0.5 * 2.0 / np.abs(p.w).sum(1).max()
    f, u0 = T(p.f), T(p.u0)
    plan = rb.Plan(T(p.xyz), T(p.is_bnd), T(p.interior), T(p.idx), T(p.w), getattr(rb, flag), 3)
    want = u0.clone()
    plan.solve_explicit(f, want, dt, 50)
    out = 0
    for ms in (1e-5, 1e-4, 1e-3, 3e-3, 1e-2) * 6:
        plan.set_wait(ms)
        u = u0.clone()
        try:
            plan.solve_explicit(f, u, dt, 50)
            assert torch.equal(u, want)
        except rb.RbffdError as e:
            assert e.code == rb.RBFFD_ERR_TIMEOUT
            out += 1
    assert out > 0
    plan.set_wait()
    u = u0.clone()
    plan.solve_explicit(f, u, dt, 50)
    assert torch.equal(u, want)


def test_plans_of_different_sizes_share_kernels(rb, orc):
    """A launch's dynamic shared memory is limited by an attribute of the kernel: a smaller
    plan tuned later must not lower it below what a larger plan of the same kernel needs."""
    sizes = {rb.RBFFD_LAUNCH_RESIDENT: (200, 90), rb.RBFFD_LAUNCH_FAR: (180, 90),
             rb.RBFFD_LAUNCH_SPLIT: (330, 110)}
    for flag, kgs in sizes.items():
        plans = []
        for kg in kgs:
            xyz, bnd = rb.rbffd_nodes(2, 0, kg, 0.3, 5)
            inter = rb.rbffd_interior(bnd)
            idx = rb.rbffd_knn(xyz, inter, 30)
            w, _ = rb.rbffd_weights(xyz, idx, 4)
            f = torch.ones(inter.numel(), dtype=torch.float64, device=DEV)
            u = torch.zeros(xyz.shape[1], dtype=torch.float64, device=DEV)
            dt = 0.5 * 2.0 / float(w.abs().sum(1).max())
            plan = rb.Plan(xyz, bnd, inter, idx, w, flag)
            plan.solve_explicit(f, u.clone(), dt, 3)
            plans.append((plan, f, u, dt))
        for plan, f, u, dt in plans + plans[::-1]:
            a = u.clone()
            assert plan.solve_explicit(f, a, dt, 20)[1] == 20
            assert torch.isfinite(a).all()
