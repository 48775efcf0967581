"""The work a user of this framework has it do, as measurable cases.

Every case is one call (or one short chain of calls) of the public binding on a
node set of the kinds this repository is used with: jittered grids of the unit
square and cube at the spacings of its workload table (1/100, 1/300, 1/1000;
cubes to 1/100), monomial orders m = 2, 4, 6 with the support sizes n = 2M or
2M + 1 that go with them, and the Poisson-disc fill.

Inputs - node sets, supports, weights, fields - are built here with plain torch
from the seed alone, so they do not depend on the library under measurement;
only plans and batches, the handles a program keeps, are the library's.
"""
from __future__ import annotations

import itertools
import math
import random

import torch

import paper_2502_12878_gb300 as rb

DEV = "cuda"
F64 = torch.float64


# ------------------------------------------------------------------- the cases
def listed():
    return [
        # residual of a given field with stencils in the caller's layout (Eq. 1): the
        # check a program makes of an iterate that is not the solver's own
        dict(name="apply_square_1m_m4", kind="apply", d=2, kg=1000, m=4, n=30),
        # supports of a large node set, the first setup call of every problem (here in 3D,
        # with the larger stencils that dimension needs)
        dict(name="knn_cube_1m_n70", kind="knn", d=3, kg=100, n=70),
        # stencil weights of a large 2D node set, the longest setup call
        dict(name="weights_square_1m_m4", kind="weights", d=2, kg=1000, m=4, n=30),
        # weights in 3D: local systems of 105 unknowns
        dict(name="weights_cube_69k_m4", kind="weights", d=3, kg=40, m=4, n=70),
        # everything a new small node set costs before its first step: supports,
        # weights, plan, stable time step (launches and allocations count here)
        dict(name="setup_square_10k_m2", kind="setup", d=2, kg=100, m=2, n=12, flags="auto"),
        # the small whole problem: thousands of steps of a few microseconds
        dict(name="solve_square_10k_m2", kind="solve", d=2, kg=100, m=2, n=12, steps=2000,
             flags="auto"),
        # the headline workload: FP64 sweeps of a million rows
        dict(name="solve_square_1m_m4", kind="solve", d=2, kg=1000, m=4, n=30, steps=100,
             flags="auto"),
        # FP32 inner sweeps inside FP64 defect correction, at the size where time to
        # accuracy is measured
        dict(name="dc_square_90k_m4", kind="dc", d=2, kg=300, m=4, n=30, k_in=1000, outer=2,
             flags="auto"),
        # gradients with respect to source and Dirichlet data of a large problem
        dict(name="adjoint_square_1m_m4", kind="adjoint", d=2, kg=1000, m=4, n=30, steps=100,
             flags="auto"),
        # a differentiable solve with weight gradients: forward and backward
        dict(name="train_square_90k_m4", kind="train", d=2, kg=300, m=4, n=30, steps=64,
             flags="auto"),
        # many independent domains of uneven sizes and orders solved in one call
        dict(name="batch_20_domains", kind="batch", domains=20, mix=4, kg_lo=70, kg_hi=330,
             steps=200),
        # node placement by the Poisson-disc fill
        dict(name="pds_square_218k", kind="pds", d=2, kg=500),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _stencil(rng, d, orders):
    m = rng.choice(orders)
    return m, 2 * math.comb(m + d, d) + rng.choice([0, 0, 1])


def draw(rng):
    kind = rng.choice(["apply", "knn", "knn", "weights", "weights", "setup", "solve", "solve",
                       "solve", "dc", "adjoint", "train", "batch", "pds"])
    if kind == "batch":
        return dict(kind=kind, domains=rng.randint(3, 20), mix=rng.randrange(1000), kg_lo=50,
                    kg_hi=_log(rng, 100, 330), steps=_log(rng, 20, 200))
    # dimension 3 where the path is used in 3D at all
    d = 3 if kind in ("knn", "weights", "solve", "pds") and rng.random() < 0.3 else 2
    c = dict(kind=kind, d=d)
    if kind == "pds":
        c["kg"] = _log(rng, 20, 500) if d == 2 else _log(rng, 8, 40)
        return c
    if kind == "knn":
        c["n"] = rng.randint(6, 57) if d == 2 else rng.randint(10, 71)
        c["kg"] = _log(rng, 30, 1000) if d == 2 else _log(rng, 14, 90)
        return c
    c["m"], c["n"] = _stencil(rng, d, (2, 4, 6) if d == 2 else (2, 4))
    # local systems cost (n + M)^3: larger ones on smaller sets
    top = {2: 1000, 4: 700, 6: 400}[c["m"]] if d == 2 else {2: 60, 4: 36}[c["m"]]
    c["kg"] = _log(rng, 30, top) if d == 2 else _log(rng, 14, top)
    if kind in ("solve", "adjoint", "train", "dc", "setup"):
        c["flags"] = rng.choice(["auto", "auto", "auto", "default"])
    rows = c["kg"] ** d
    if kind in ("solve", "adjoint", "dc"):
        k = max(20, min(_log(rng, 20, 2000), int(3e9 / (rows * c["n"]))))
        if kind == "dc":
            c["k_in"], c["outer"] = max(10, k // 2), 2
        else:
            c["steps"] = k
    if kind == "train":
        c["kg"] = min(c["kg"], 300)
        c["steps"] = _log(rng, 4, 64)
    return c


def _domains(case):
    """The batch's domains: spacings log-uniform in [1/kg_hi, 1/kg_lo], orders mixed."""
    rng = random.Random(case["mix"])
    out = []
    for _ in range(case["domains"]):
        m = rng.choice((2, 4, 6))
        out.append(dict(d=2, kg=_log(rng, case["kg_lo"], case["kg_hi"]), m=m,
                        n=2 * math.comb(m + 2, 2)))
    return out


# --------------------------------------------------------------------- inputs
def _nodes(case, seed):
    """Jittered grid of the unit square or cube: boundary nodes on the grid, interior
    ones moved by up to 0.3 h along each axis.  (xyz [d, N], is_bnd [N], interior [NI])."""
    d, kg = case["d"], case["kg"]
    g = torch.Generator(device=DEV).manual_seed(seed)
    h = 1.0 / kg
    ax = torch.arange(kg + 1, device=DEV)
    ij = torch.stack([t.reshape(-1) for t in torch.meshgrid(*([ax] * d), indexing="ij")])
    bnd = ((ij == 0) | (ij == kg)).any(0)
    jit = (torch.rand(ij.shape, generator=g, device=DEV, dtype=F64) * 2 - 1) * (0.3 * h)
    xyz = ij.to(F64) / kg + torch.where(bnd, torch.zeros_like(jit), jit)
    return xyz.contiguous(), bnd.to(torch.uint8), torch.nonzero(~bnd).flatten().to(torch.int32)


def _supports(case, xyz, interior):
    """The n nearest nodes of every interior node, itself first, from a window of grid
    neighbours wide enough for nodes beside an edge."""
    d, kg, n = case["d"], case["kg"], case["n"]
    rad = math.sqrt(2 * n / math.pi) if d == 2 else (1.5 * n / math.pi) ** (1 / 3)
    side = min(2 * math.ceil(rad + 0.8) + 1, kg + 1)
    offs = torch.tensor(list(itertools.product(range(side), repeat=d)), device=DEV)
    strides = torch.tensor([(kg + 1) ** (d - 1 - a) for a in range(d)], device=DEV)
    off = (offs * strides).sum(1)
    out = torch.empty((interior.numel(), n), dtype=torch.int32, device=DEV)
    chunk = max(1, (1 << 26) // off.numel())
    for b in range(0, interior.numel(), chunk):
        c = interior[b:b + chunk].long()
        start = torch.zeros_like(c)
        for a in range(d):
            ia = (c // strides[a]) % (kg + 1)
            start += (ia - side // 2).clamp(0, kg + 1 - side) * strides[a]
        cand = start[:, None] + off[None]
        d2 = torch.zeros(cand.shape, dtype=F64, device=DEV)
        for a in range(d):
            d2 += (xyz[a][cand] - xyz[a][c][:, None]) ** 2
        near = torch.topk(d2, n, dim=1, largest=False, sorted=True).indices
        out[b:b + chunk] = torch.gather(cand, 1, near).to(torch.int32)
    return out


def _monomials(d, m):
    return sorted((e for e in itertools.product(range(m + 1), repeat=d) if sum(e) <= m),
                  key=lambda e: (sum(e), [-x for x in e]))


def _plain_weights(case, xyz, idx):
    """RBF-FD Laplacian weights (r^3 and monomials to degree m) by batched dense solves."""
    d, m, n = case["d"], case["m"], idx.shape[1]
    ex = _monomials(d, m)
    M = len(ex)
    s = n + M
    rhs_p = torch.tensor([2.0 if max(e) == 2 and sum(e) == 2 else 0.0 for e in ex], device=DEV,
                         dtype=F64)
    out = torch.empty(idx.shape, dtype=F64, device=DEV)
    chunk = max(1, (1 << 28) // (s * s))
    for b in range(0, idx.shape[0], chunk):
        x = xyz[:, idx[b:b + chunk].long()]
        x = x - x[:, :, :1]
        sig = x.square().sum(0).sqrt().amax(1)
        x = x / sig[None, :, None]
        G = torch.zeros((x.shape[1], s, s), dtype=F64, device=DEV)
        r2 = torch.zeros((x.shape[1], n, n), dtype=F64, device=DEV)
        for a in range(d):
            r2 += (x[a][:, :, None] - x[a][:, None, :]) ** 2
        G[:, :n, :n] = r2 * r2.sqrt()
        for k, e in enumerate(ex):
            p = torch.ones_like(x[0])
            for a in range(d):
                for _ in range(e[a]):
                    p = p * x[a]
            G[:, :n, n + k] = p
            G[:, n + k, :n] = p
        rhs = torch.empty((x.shape[1], s, 1), dtype=F64, device=DEV)
        rhs[:, :n, 0] = 3.0 * (d + 1) * x.square().sum(0).sqrt()
        rhs[:, n:, 0] = rhs_p
        out[b:b + chunk] = torch.linalg.solve(G, rhs)[:, :n, 0] / (sig * sig)[:, None]
    return out


def _fields(xyz, bnd, interior):
    """Manufactured u = prod sin(pi x): its source at the interior nodes, and the start
    iterate (its values on the boundary, 0 inside)."""
    ua = torch.sin(math.pi * xyz).prod(0)
    f = (-math.pi ** 2 * xyz.shape[0]) * ua[interior.long()]
    u0 = torch.where(bnd.bool(), ua, torch.zeros_like(ua))
    return f, u0


def _problem(case, seed):
    xyz, bnd, interior = _nodes(case, seed)
    idx = _supports(case, xyz, interior)
    w = _plain_weights(case, xyz, idx)
    f, u0 = _fields(xyz, bnd, interior)
    # inside the stability bound for every node set: |eigenvalues| <= max row sum
    dt = 0.9 * 2.0 / w.abs().sum(1).max().item()
    return dict(xyz=xyz, bnd=bnd, interior=interior, idx=idx, w=w, f=f, u0=u0, dt=dt)


def _vector(count, seed, k):
    g = torch.Generator(device=DEV).manual_seed(seed * 8 + k)
    return torch.randn(count, generator=g, device=DEV, dtype=F64)


def _misfit(p, seed):
    """dL/du of a misfit observed at one node in a hundred (all kinds of nodes)."""
    v = _vector(p["u0"].numel(), seed, 1)
    g = torch.Generator(device=DEV).manual_seed(seed * 8 + 2)
    return torch.where(torch.rand(v.shape, generator=g, device=DEV) < 0.01, v,
                       torch.zeros_like(v))


def _flags(case):
    return rb.RBFFD_LAUNCH_AUTO if case["flags"] == "auto" else 0


def _plan(case, p):
    return rb.Plan(p["xyz"], p["bnd"], p["interior"], p["idx"], p["w"], _flags(case))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "pds":
        # node arrays of a fixed capacity: how many nodes the fill places varies by seed
        cap = 2 * (case["kg"] + 2) ** case["d"]
        return dict(case=case, seed=seed, xyz=torch.zeros((case["d"], cap), dtype=F64, device=DEV),
                    bnd=torch.zeros(cap, dtype=torch.uint8, device=DEV))
    if kind in ("knn", "setup"):
        xyz, bnd, interior = _nodes(case, seed)
        return dict(case=case, xyz=xyz, bnd=bnd, interior=interior,
                    v0=_vector(interior.numel(), seed, 3))
    if kind == "weights":
        xyz, _, interior = _nodes(case, seed)
        return dict(case=case, xyz=xyz, idx=_supports(case, xyz, interior))
    if kind == "batch":
        ps = [_problem(c, seed * 64 + i) for i, c in enumerate(_domains(case))]
        p = dict(case=case, fs=[q["f"] for q in ps], u0s=[q["u0"] for q in ps],
                 dts=[q["dt"] for q in ps],
                 plans=[rb.Plan(q["xyz"], q["bnd"], q["interior"], q["idx"], q["w"])
                        for q in ps])
        p["batch"] = rb.Batch(p["plans"])
        # one 1024-thread block per SM, the domains' costs measured by a short probe
        p["batch"].set_shape(1, 1, 1024)
        p["batch"].calibrate(p["fs"], [u.clone() for u in p["u0s"]], p["dts"], 50)
        return p
    p = _problem(case, seed)
    p["case"] = case
    if kind == "apply":
        # a field that is not the solution: its residual is not all cancellation
        p["u"] = p["u0"] + 0.1 * _vector(p["u0"].numel(), seed, 4)
    elif kind == "solve":
        p["plan"] = _plan(case, p)
        p["plan"].solve_explicit(p["f"], p["u0"].clone(), p["dt"], 2)
    elif kind == "dc":
        p["plan"] = _plan(case, p)
        p["plan"].solve_dc(p["f"], p["u0"].clone(), p["dt"], 0.0, 1, 2, 1e-3)
    elif kind == "adjoint":
        p["dLdu"] = _misfit(p, seed)
        p["plan"] = _plan(case, p)
        p["plan"].adjoint(p["dLdu"], 1, p["dt"])
    elif kind == "train":
        p["g"] = p["u0"][p["bnd"].bool()]
        p["dLdu"] = _misfit(p, seed)
        p["solver"] = rb.ExplicitSolver(p["xyz"], p["bnd"], p["interior"], p["idx"],
                                        case["steps"], p["dt"], flags=_flags(case))
        for k in ("f", "g", "w"):
            p[k].requires_grad_(True)
        _train(p)
    return p


# ------------------------------------------------------------------- one pass
def _train(p):
    u = p["solver"](p["f"], p["g"], p["w"])
    gf, gg, gw = torch.autograd.grad(u, (p["f"], p["g"], p["w"]), p["dLdu"])
    return u.detach(), gf, gg, gw


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "apply":
        return rb.rbffd_apply(state["w"], state["idx"], state["u"])
    if kind == "knn":
        return rb.rbffd_knn(state["xyz"], state["interior"], case["n"])
    if kind == "weights":
        return rb.rbffd_weights(state["xyz"], state["idx"], case["m"])
    if kind == "setup":
        idx = rb.rbffd_knn(state["xyz"], state["interior"], case["n"])
        w, status = rb.rbffd_weights(state["xyz"], idx, case["m"])
        plan = rb.Plan(state["xyz"], state["bnd"], state["interior"], idx, w, _flags(case))
        dt, rho = plan.stable_dt(state["v0"])
        plan.destroy()
        return idx, w, status, dt, rho
    if kind == "solve":
        u = state["u0"].clone()
        _, steps, res = state["plan"].solve_explicit(state["f"], u, state["dt"], case["steps"])
        return u, steps, res
    if kind == "dc":
        u = state["u0"].clone()
        _, outer, inner, res = state["plan"].solve_dc(state["f"], u, state["dt"], 1e-10,
                                                      case["outer"], case["k_in"], 1e-3)
        return u, outer, inner, res
    if kind == "adjoint":
        return state["plan"].adjoint(state["dLdu"], case["steps"], state["dt"])
    if kind == "train":
        return _train(state)
    if kind == "batch":
        us = [u.clone() for u in state["u0s"]]
        nd = len(us)
        _, steps, res, _ = state["batch"].solve(state["fs"], us, state["dts"],
                                                [case["steps"]] * nd, [0.0] * nd)
        return us, steps, res
    assert kind == "pds"
    xyz, bnd, generations = rb.rbffd_nodes_pds(0, case["kg"], state["seed"], d=case["d"])
    state["xyz"][:, :bnd.numel()] = xyz
    state["bnd"][:bnd.numel()] = bnd
    return state["xyz"], state["bnd"], bnd.numel(), generations


# ----------------------------------------------------------------- necessities
def work(case):
    """Bytes and operations of one pass.  Sweeps count each stencil entry's weight (8, or
    4 in FP32) and a 2-byte neighbour index once per step when the stencils are larger than
    the 126 MB L2, once per pass otherwise."""
    kind = case["kind"]
    if kind == "batch":
        each = [work(dict(c, kind="solve", steps=case["steps"])) for c in _domains(case)]
        return {k: sum(e[k] for e in each) for k in ("bytes", "flops")}
    d, kg = case["d"], case["kg"]
    N, NI = (kg + 1) ** d, (kg - 1) ** d
    if kind == "pds":   # the spacing-1/kg fill holds about 0.87 (2D) / 0.82 (3D) nodes per h^d
        nodes = (0.87 if d == 2 else 0.82) * N
        K = 15 if d == 2 else 50
        return dict(bytes=nodes * (8 * d + 1), flops=nodes * K * (3 * d - 1) * 2)
    n = case["n"]
    dist = NI * n * (3 * d - 1)
    if kind == "knn":
        return dict(bytes=8 * d * N + 4 * NI + 4 * NI * n, flops=dist)
    s = n + math.comb(case["m"] + d, d)
    solve_flops = NI * (2 * s ** 3 / 3 + 2 * s * s)
    if kind == "weights":
        return dict(bytes=8 * d * N + NI * (12 * n + 1), flops=solve_flops)
    if kind == "apply":
        return dict(bytes=NI * (12 * n + 8) + 8 * N, flops=2 * NI * n)
    sweep = NI * (2 * n + 3)
    if kind == "setup":
        return dict(bytes=8 * d * N + NI * (24 * n + 1), flops=dist + solve_flops + 200 * sweep)

    def stream(entry, row, steps):
        per = NI * (entry * n + row)
        return per * (steps if NI * entry * n > 126e6 else 1)
    if kind == "solve":
        return dict(bytes=stream(10, 24, case["steps"]) + 16 * N, flops=sweep * case["steps"])
    if kind == "dc":
        inner = case["outer"] * case["k_in"]
        return dict(bytes=stream(6, 12, inner) + (case["outer"] + 1) * NI * (10 * n + 24),
                    flops=sweep * (inner + case["outer"] + 1))
    if kind == "adjoint":
        return dict(bytes=stream(10, 32, case["steps"]) + 24 * N, flops=sweep * case["steps"])
    # train: the forward steps, the replayed ones, the reverse ones, the weight gradient
    return dict(bytes=stream(10, 32, 3 * case["steps"]) + NI * (20 * n + 8) + 24 * N,
                flops=sweep * 4 * case["steps"])


# ------------------------------------------------------------- 64-bit values
def _apply(p, u):
    """W u, summed over chunks of rows."""
    out = torch.empty(p["idx"].shape[0], dtype=F64, device=DEV)
    for b in range(0, out.numel(), 1 << 18):
        out[b:b + (1 << 18)] = (p["w"][b:b + (1 << 18)] * u[p["idx"][b:b + (1 << 18)].long()]).sum(1)
    return out


def _forward(p, steps, keep=False):
    """u^steps of the explicit iteration, the last step's residual max-norm, and the
    iterates u^0 .. u^{steps-1} if kept."""
    u, rows, res, all_u = p["u0"].clone(), p["interior"].long(), 0.0, []
    for _ in range(steps):
        if keep:
            all_u.append(u.clone())
        r = _apply(p, u) - p["f"]
        u[rows] += p["dt"] * r
        res = r.abs().max()
    return u, float(res), all_u


def _transpose(p):
    """W^T [N, NI] as a sparse matrix."""
    NI, n = p["idx"].shape
    rows = torch.arange(NI, device=DEV).repeat_interleave(n)
    at = torch.stack([p["idx"].long().reshape(-1), rows])
    N = p["u0"].numel()
    return torch.sparse_coo_tensor(at, p["w"].reshape(-1), (N, NI)).coalesce().to_sparse_csr()


def _reverse(p, dLdu, steps, dt, at_step=None):
    """Reverse sweep: gradients to the source and the boundary values, and lambda^0;
    at_step(k, lambda^{k+1}) is called for k = steps-1 .. 0."""
    rows = p["interior"].long()
    WT = _transpose(p)
    lam = dLdu[rows].clone()
    S = torch.zeros_like(lam)
    for k in range(steps - 1, -1, -1):
        if at_step:
            at_step(k, lam)
        S += lam
        lam = lam + dt * (WT @ lam)[rows]
    gg = torch.where(p["bnd"].bool(), dt * (WT @ S) + dLdu, torch.zeros_like(dLdu))
    return -dt * S, gg, lam


def exact(case, seed):
    kind = case["kind"]
    if kind in ("knn", "pds"):
        # supports are whole numbers; the fill is a sequential walk whose nodes are the
        # outcome of exact comparisons, hours of plain numpy at these sizes
        return None
    if kind == "weights":
        xyz, _, interior = _nodes(case, seed)
        return _plain_weights(case, xyz, _supports(case, xyz, interior)), None
    if kind == "setup":
        xyz, bnd, interior = _nodes(case, seed)
        idx = _supports(case, xyz, interior)
        p = dict(idx=idx, w=_plain_weights(case, xyz, idx))
        y = _vector(interior.numel(), seed, 3)
        v = torch.zeros(xyz.shape[1], dtype=F64, device=DEV)
        for _ in range(200):
            v[interior.long()] = y / y.norm()
            y = _apply(p, v)
        rho = float(y.norm())
        return None, p["w"], None, 2.0 / (1.05 * rho), rho
    if kind == "batch":
        us, rs = [], []
        for i, c in enumerate(_domains(case)):
            u, r, _ = _forward(_problem(c, seed * 64 + i), case["steps"])
            us.append(u)
            rs.append(r)
        return us, [None] * len(us), rs
    if kind == "solve" and case["steps"] * case["kg"] ** case["d"] * case["n"] > 8e9:
        return None
    p = _problem(case, seed)
    if kind == "apply":
        return _apply(p, p["u0"] + 0.1 * _vector(p["u0"].numel(), seed, 4))
    if kind == "solve":
        u, res, _ = _forward(p, case["steps"])
        return u, None, res
    if kind == "dc":
        u, rows, r = p["u0"].clone(), p["interior"].long(), None
        for _ in range(case["outer"]):
            r = _apply(p, u) - p["f"]
            e = torch.zeros_like(u)
            for _ in range(case["k_in"]):
                rho = _apply(p, e) + r
                e[rows] += p["dt"] * rho
                if float(rho.abs().max()) < 1e-3 * float(r.abs().max()):
                    break
            u += e
        return u, None, None, float((_apply(p, u) - p["f"]).abs().max())
    dLdu = _misfit(p, seed)
    if kind == "adjoint":
        return _reverse(p, dLdu, case["steps"], p["dt"])
    u, _, us = _forward(p, case["steps"], keep=True)
    gw = torch.zeros_like(p["w"])
    at = p["idx"].long()

    def add(k, lam):
        gw.add_(p["dt"] * lam[:, None] * us[k][at])
    gf, gg, _ = _reverse(p, dLdu, case["steps"], p["dt"], add)
    return u, gf, gg[p["bnd"].bool()], gw
