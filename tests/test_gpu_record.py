"""Recorded runs (rbffd_solve_record) against solves of one segment after another, bit for bit:
every launch family, segments that divide K or not, records of every step or of segments, none at
all; the same divergence verdict; plans with Neumann nodes; and the differentiable solve through
either."""
import numpy as np
import pytest

import rbffd_inputs as gen
from oracle_problem import build, build_mixed

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


# graph, persistent, linked, far lists (resident with a barrier)
@pytest.mark.parametrize("flags", [0, 16, 128, 2048])
@pytest.mark.parametrize("Kg,m", [(60, 2), (110, 4), (4, 1)])
def test_record_equals_segment_solves(rb, orc, Kg, m, flags):
    p = build(orc, 2, Kg, m, seed=31)
    plan = rb.Plan(T(p.xyz), T(p.is_bnd), T(p.interior), T(p.idx), T(p.w), flags)
    dt = 0.5 * 2.0 / np.abs(p.w).sum(1).max()
    f = T(p.f)
    for K, seg in ((1, 1), (20, 5), (21, 4), (7, 9), (30, 1)):
        u, kept = T(p.u0), []
        for k in range(K):
            kept.append(u.clone())
            plan.solve_explicit(f, u, dt, 1)
        kept = torch.stack(kept)
        for rows in (None, -(-K // seg), K):
            v = T(p.u0)
            ck = None if rows is None else torch.full((rows, p.N), 7.0, dtype=torch.float64,
                                                      device="cuda")
            every = plan.solve_record(f, v, dt, K, seg, ck)
            assert torch.equal(u, v)
            assert every in (1, seg) and (every == seg or rows == K)
            if ck is not None:
                assert torch.equal(ck[:-(-K // every)], kept[::every])
    # a growing run: refused by the same segment lengths as one solve after another
    u0 = T(gen.random_vector(p.N, 4))
    for seg in (3, 40):
        got = []
        for how in range(2):
            u = u0.clone()
            try:
                if how:
                    plan.solve_record(f, u, 40 * dt, 40, seg, None)
                else:
                    for k in range(0, 40, seg):
                        plan.solve_explicit(f, u, 40 * dt, min(seg, 40 - k))
                got.append(0)
            except rb.RbffdError as e:
                got.append(e.code)
        assert got[0] == got[1]


@pytest.mark.parametrize("flags", [0, 64])
def test_record_with_neumann_nodes(rb, orc, flags):
    mp = build_mixed(orc, 2, 24, 2, seed=3)
    p = mp.base
    plan = rb.Plan(T(p.xyz), T(p.is_bnd), T(p.interior), T(p.idx), T(p.w), flags)
    plan.set_neumann(T(mp.nnode), T(mp.nidx), T(mp.nw), T(mp.g + 0.25))
    dt = 0.5 * 2.0 / np.abs(p.w).sum(1).max()
    f = T(p.f)
    for K, seg, scale in ((20, 5, 1), (21, 4, 1), (1, 3, 1), (30, 7, 1e6)):
        u, v, kept, code = T(p.u0), T(p.u0), [], [0, 0]
        rows = -(-K // seg)
        ck = torch.zeros((rows, p.N), dtype=torch.float64, device="cuda")
        try:
            for k in range(0, K, seg):
                kept.append(u.clone())
                plan.solve_explicit(f, u, scale * dt, min(seg, K - k))
        except rb.RbffdError as e:
            code[0] = e.code
        try:
            assert plan.solve_record(f, v, scale * dt, K, seg, ck) == seg
        except rb.RbffdError as e:
            code[1] = e.code
        assert code[0] == code[1] and (scale == 1 or code[0] != 0)
        assert torch.equal(u, v)
        assert torch.equal(ck[:len(kept)], torch.stack(kept))


def test_differentiable_solve_keeps_its_bits(rb, orc):
    p = build(orc, 2, 70, 4, seed=33)
    dt = 0.5 * 2.0 / np.abs(p.w).sum(1).max()
    bnd = p.is_bnd.astype(bool)
    res = []
    for flags, every, keep in ((0, None, None), (64, None, None), (64, None, 0), (64, 3, 0)):
        s = rb.ExplicitSolver(T(p.xyz), T(p.is_bnd), T(p.interior), T(p.idx), 23, dt, every,
                              flags)
        f, g, w = (T(a).requires_grad_(True) for a in (p.f, p.u0[bnd], p.w))
        old = rb.KEEP_ITERATES
        rb.KEEP_ITERATES = old if keep is None else keep
        try:
            u = s(f, g, w)
            grads = torch.autograd.grad(u, (f, g, w), torch.ones_like(u))
            (gf,) = torch.autograd.grad(s(f, g, w.detach()), (f,), torch.ones_like(u))
        finally:
            rb.KEEP_ITERATES = old
        res.append([u.detach(), *grads, gf])
    for r in res[1:]:
        assert all(torch.equal(a, b) for a, b in zip(r, res[0]))


def test_memory_of_a_differentiable_solve(rb, orc):
    """A caller's spacing bounds the iterates kept; so does a plan that cannot keep them all."""
    p = build(orc, 2, 70, 4, seed=33)
    dt = 0.5 * 2.0 / np.abs(p.w).sum(1).max()
    bnd = p.is_bnd.astype(bool)
    K = 23
    for flags, every, rows in ((0, None, 5), (0, 4, 6), (64, 4, 6), (64, 1, K), (64, None, K)):
        s = rb.ExplicitSolver(T(p.xyz), T(p.is_bnd), T(p.interior), T(p.idx), K, dt, every, flags)
        f, g, w = (T(a).requires_grad_(True) for a in (p.f, p.u0[bnd], p.w))
        u = s(f, g, w)
        kept = u.grad_fn.saved_tensors[1]
        assert kept.shape == (rows, p.N)
        assert kept.untyped_storage().nbytes() == rows * p.N * 8
