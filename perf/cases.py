"""The calls a user of this package makes, at the sizes such a user has.

Every case is one call (or one training pass, or one corrector step) through
the package's public entry points on a seeded synthetic mesh: jittered
triangular lattices numbered row by row, and lattices with bisected sides
numbered along a Morton curve, whose cell graph has odd cycles as that of an
unstructured Delaunay mesh has.  Fields and right-hand sides follow the
workloads of the benchmark (porous block, channel with an anisotropic block,
random-Fourier ensemble members, log-permeability fields).

``work`` counts the arrays a call gets and gives back, each once: what an
iterative solve has to move per iteration depends on the method it takes.
``exact`` computes the same results with plain torch operations in FP64,
Krylov solves refined to the FP64 floor included.
"""
import math

import torch

import paper_2309_03543_gb300 as cps

NU, DT, GRAIN = 1.5e-5, 0.225, 1e-3
F64 = torch.float64
_CTX = []
_KEPT = []


def _ctx():
    """One library context per process, as a program keeps one."""
    if not _CTX:
        _CTX.append(cps.Context(0))
    return _CTX[0]


def _keep(*handles):
    """A program keeps the systems it solves with for its whole run."""
    _KEPT.extend(handles)


# ------------------------------------------------------------------- cases

def listed():
    return [
        # one corrector solve on a small mesh, the size of a quick test or of
        # a coarse run: bound by latency
        {"name": "solve_block_n64", "op": "solve", "n": 64, "mesh": "lattice", "fields": "block",
         "pc": "jacobi", "precision": "fp64"},
        # a mid-size corrector solve: does not fit one cluster, does not fill HBM
        {"name": "solve_channel_n301", "op": "solve", "n": 301, "mesh": "lattice",
         "fields": "channel", "pc": "jacobi", "precision": "fp64"},
        # the benchmark's solve: 2.09M cells, anisotropic block in a channel
        {"name": "solve_channel_n1024", "op": "solve", "n": 1024, "mesh": "lattice",
         "fields": "channel", "pc": "jacobi", "precision": "fp64"},
        # a mesh that two colours cannot colour, numbered along a space-filling
        # curve (the unstructured meshes of the scheme)
        {"name": "solve_defect_n451", "op": "solve", "n": 451, "mesh": "defect",
         "fields": "ensemble", "pc": "jacobi", "precision": "fp64"},
        # the paper's preconditioner, incomplete Cholesky, on a large lattice
        {"name": "ic0_channel_n700", "op": "solve", "n": 700, "mesh": "lattice",
         "fields": "channel", "pc": "ic0", "precision": "fp64"},
        # binary32 iterations inside FP64 refinement
        {"name": "mixed_channel_n400", "op": "solve", "n": 400, "mesh": "lattice",
         "fields": "channel", "pc": "jacobi", "precision": "mixed"},
        # an uneven ensemble in one call (uncertainty runs)
        {"name": "batch_48", "op": "batch", "count": 48, "lo": 2000, "hi": 120000,
         "precision": "fp64"},
        # assembly of the 2.09M-cell matrix, done for every parameter value
        {"name": "assemble_n1024", "op": "assemble", "n": 1024, "mesh": "lattice",
         "fields": "channel"},
        # a training pass: chained solves, checkpointed, with their adjoints
        {"name": "chain_logk_n129", "op": "chain", "n": 129, "steps": 3, "every": 2},
        # the pressure corrector step: two solves, the second one warm, and the
        # flux and velocity kernels around them
        {"name": "cp2_channel_n384", "op": "cp2", "n": 384, "mesh": "lattice",
         "fields": "channel", "pc": "jacobi"},
        # the viscous corrector step: x and y systems coupled by the tensor
        {"name": "cp1_channel_n1024", "op": "cp1", "n": 1024, "mesh": "lattice",
         "fields": "channel", "precision": "fp64"},
        # the assembled operator applied to a field of 8.4M cells
        {"name": "matvec_n2048", "op": "matvec", "n": 2048, "mesh": "lattice",
         "fields": "channel"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["solve", "solve", "solve", "solve", "batch", "assemble", "chain", "cp2",
                     "cp1", "matvec"])
    lattice = {"mesh": rng.choice(["lattice", "lattice", "defect"]),
               "fields": rng.choice(["block", "channel", "ensemble"])}
    if op == "solve":
        pc, precision = rng.choice([("jacobi", "fp64"), ("jacobi", "fp64"), ("ic0", "fp64"),
                                    ("reduced", "fp64"), ("jacobi", "mixed"),
                                    ("ic0", "mixed")])
        if pc == "reduced":
            lattice["mesh"] = "lattice"
        n = _log_int(rng, 24, 400 if precision == "mixed" else 900)
        return {"op": op, "n": n, "pc": pc, "precision": precision, **lattice}
    if op == "batch":
        lo = _log_int(rng, 500, 4000)
        return {"op": op, "count": rng.randint(3, 48), "lo": lo, "hi": _log_int(rng, 8000, 120000),
                "precision": rng.choice(["fp64", "fp64", "mixed"])}
    if op == "chain":
        return {"op": op, "n": _log_int(rng, 17, 129), "steps": rng.randint(1, 3),
                "every": rng.randint(1, 2)}
    if op == "cp2":
        pc = rng.choice(["jacobi", "jacobi", "ic0"])
        return {"op": op, "n": _log_int(rng, 20, 384), "pc": pc, **lattice}
    if op == "cp1":
        return {"op": op, "n": _log_int(rng, 40, 1024), "precision": rng.choice(["fp64", "mixed"]),
                **lattice, "mesh": "lattice"}
    if op == "assemble":
        return {"op": op, "n": _log_int(rng, 600, 1024), **lattice}
    return {"op": op, "n": _log_int(rng, 100, 2048), **lattice}


# ------------------------------------------------------------------- meshes

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1 + 7919 * int(seed))
    return g


def _morton(c):
    lo, hi = c.min(0).values, c.max(0).values
    q = ((c - lo) / (hi - lo) * 65535.0).to(torch.int64)
    key = torch.zeros(c.shape[0], dtype=torch.int64, device=c.device)
    for b in range(16):
        for d in range(2):
            key |= ((q[:, d] >> b) & 1) << (2 * b + d)
    return key


def _mesh(n, kind, g):
    """xy [nv, 2], tri [nt, 3] counter-clockwise, Dirichlet sides (tri * 3 +
    local side) on the right edge."""
    j, i = torch.meshgrid(torch.arange(n, device="cuda"), torch.arange(n, device="cuda"),
                          indexing="ij")
    xy = torch.stack([(i + 0.5 * (j % 2)).reshape(-1), (j * (math.sqrt(3.0) / 2)).reshape(-1)],
                     1).to(F64)
    r = 0.05 * torch.sqrt(torch.rand(n * n, generator=g, device="cuda", dtype=F64))
    phi = 2 * math.pi * torch.rand(n * n, generator=g, device="cuda", dtype=F64)
    inner = ((i > 0) & (i < n - 1) & (j > 0) & (j < n - 1)).reshape(-1)
    xy = xy + torch.where(inner, r, torch.zeros_like(r))[:, None] * \
        torch.stack([torch.cos(phi), torch.sin(phi)], 1)
    right = (i == n - 1).reshape(-1)
    b = (j * n + i)[:-1, :-1]
    t = b + n
    even = (j[:-1, :-1] % 2) == 0
    up = torch.stack([b, b + 1, torch.where(even, t, t + 1)], -1)
    down = torch.stack([t, torch.where(even, b + 1, b), t + 1], -1)
    if kind == "defect":
        # bisect the side shared by the up and the down cell of one column at
        # spaced places away from the boundary (about 0.2% of the cells, at least one)
        step = 16
        off = int(torch.randint(2, 6, (1,), generator=g, device="cuda"))
        m = n - 1
        rows = torch.arange(off, m - 2, step, device="cuda")
        jj, ii = torch.meshgrid(rows, rows, indexing="ij")
        jj, ii = jj.reshape(-1), ii.reshape(-1)
        u, d = up[jj, ii], down[jj, ii]
        ev = (jj % 2 == 0)
        p = torch.where(ev, u[:, 1], u[:, 0])       # the shared side p -> q
        q = u[:, 2]
        mid = n * n + torch.arange(jj.numel(), device="cuda")
        xy = torch.cat([xy, 0.5 * (xy[p] + xy[q])])
        right = torch.cat([right, torch.zeros(jj.numel(), dtype=torch.bool, device="cuda")])
        cu = torch.where(ev, u[:, 0], u[:, 1])      # the vertices opposite it
        cd = torch.where(ev, d[:, 2], d[:, 0])
        # counter-clockwise halves: side p -> q in the up cell, q -> p in the down cell
        first = torch.where(ev[:, None], torch.stack([p, mid, cu], 1), torch.stack([q, mid, cu], 1))
        second = torch.where(ev[:, None], torch.stack([mid, q, cu], 1),
                             torch.stack([mid, p, cu], 1))
        third = torch.where(ev[:, None], torch.stack([q, mid, cd], 1), torch.stack([p, mid, cd], 1))
        fourth = torch.where(ev[:, None], torch.stack([mid, p, cd], 1),
                             torch.stack([mid, q, cd], 1))
        up, down = up.clone(), down.clone()
        up[jj, ii], down[jj, ii] = first, third
        tri = torch.cat([torch.stack([up, down], 2).reshape(-1, 3), second, fourth])
        a, bb, c = xy[tri[:, 0]], xy[tri[:, 1]], xy[tri[:, 2]]
        cross = (bb[:, 0] - a[:, 0]) * (c[:, 1] - a[:, 1]) - (bb[:, 1] - a[:, 1]) * (c[:, 0] - a[:, 0])
        tri = torch.where((cross < 0)[:, None], tri[:, [0, 2, 1]], tri)
        tri = tri[torch.argsort(_morton(xy[tri].mean(1)), stable=True)]
    else:
        tri = torch.stack([up, down], 2).reshape(-1, 3)
    on = right[tri[:, [1, 2, 0]]] & right[tri[:, [2, 0, 1]]]
    e, s = torch.nonzero(on, as_tuple=True)
    return xy, tri.to(torch.int32).contiguous(), (e * 3 + s).to(torch.int32)


def _fourier(p, g, modes=32, kmax=8):
    """Standardised sum of random cosines with integer wave vectors."""
    k = torch.randint(-kmax, kmax + 1, (modes, 2), generator=g, device="cuda").to(F64)
    k = torch.where((k == 0).all(1, keepdim=True), torch.ones_like(k), k)
    a = torch.randn(modes, generator=g, device="cuda", dtype=F64)
    ph = 2 * math.pi * torch.rand(modes, generator=g, device="cuda", dtype=F64)
    k = (2 * math.pi) * k / (p.max(0).values - p.min(0).values)
    f = torch.zeros(p.shape[0], dtype=F64, device="cuda")
    for m in range(modes):
        f += a[m] * torch.cos(p @ k[m] + ph[m])
    return (f - f.mean()) / f.std()


def _box(p, lo, hi):
    """Signed distance to a box, positive outside."""
    c = torch.tensor([0.5 * (lo[0] + hi[0]), 0.5 * (lo[1] + hi[1])], dtype=F64, device="cuda")
    h = torch.tensor([0.5 * (hi[0] - lo[0]), 0.5 * (hi[1] - lo[1])], dtype=F64, device="cuda")
    q = (p - c).abs() - h
    return q.clamp(min=0).norm(dim=1) + q.max(1).values.clamp(max=0)


def _kozeny(eps):
    return 180.0 * (1.0 - eps) ** 2 / (GRAIN * GRAIN * eps ** 3)


def _iso(k):
    return torch.stack([k, torch.zeros_like(k), k], 1)


def _fields(xy, n, kind, g):
    """Nodal porosity and inverse permeability tensor (xx, xy, yy)."""
    W, H = n - 1.0, (n - 1.0) * math.sqrt(3.0) / 2
    if kind == "block":
        w = 0.5 * (1 - torch.tanh(_box(xy, (W / 4, H / 4), (3 * W / 4, 3 * H / 4)) / 0.75))
        eps = 1.0 - 0.6 * w
        return eps, _iso(_kozeny(eps))
    f = _fourier(xy, g)
    if kind == "ensemble":
        eps = (0.65 + 0.175 * f).clamp(0.3, 1.0)
        return eps, _iso(_kozeny(eps))
    blk = (0.45 + 0.1 * f).clamp(0.3, 0.6)
    w = 0.5 * (1 - torch.tanh(_box(xy, (W / 3, -H), (2 * W / 3, 0.8 * H)) / 0.75))
    eps = 1.0 + (blk - 1.0) * w
    k, c, s = _kozeny(eps), math.cos(math.pi / 6), math.sin(math.pi / 6)
    l1, l2 = 100.0 * k, k
    return eps, torch.stack([c * c * l1 + s * s * l2, c * s * (l1 - l2),
                             s * s * l1 + c * c * l2], 1)


def _areas(xy, tri):
    t = tri.long()
    a, b, c = xy[t[:, 0]], xy[t[:, 1]], xy[t[:, 2]]
    return 0.5 * ((b[:, 0] - a[:, 0]) * (c[:, 1] - a[:, 1])
                  - (b[:, 1] - a[:, 1]) * (c[:, 0] - a[:, 0]))


def _normal(m, g):
    return torch.randn(m, generator=g, device="cuda", dtype=F64)


def _velocity(xy, tri, g, mean, scale):
    c = xy[tri.long()].mean(1)
    m = torch.tensor(mean, dtype=F64, device="cuda")[:, None]
    return m + scale * torch.stack([_fourier(c, g), _fourier(c, g)])


def _problem(case, seed):
    g = _gen(seed)
    xy, tri, dirichlet = _mesh(case["n"], case.get("mesh", "lattice"), g)
    eps, kinv = _fields(xy, case["n"], case["fields"], g)
    return g, xy, tri, dirichlet, eps, kinv


def _walls(tri):
    """Every boundary side (no-slip walls)."""
    nbr, _ = _neighbours(tri)
    e, s = torch.nonzero(nbr < 0, as_tuple=True)
    return (e * 3 + s).to(torch.int32)


def _members(case, seed):
    """Sizes (vertices per side) of an ensemble, log-uniform in cells: the
    same for every seed, as the members' fields and right-hand sides are what
    a user redraws."""
    k = case["count"]
    f = [(i + 0.5) / k for i in range(k)]
    cells = [case["lo"] * (case["hi"] / case["lo"]) ** v for v in f]
    return [max(3, 1 + round(math.sqrt(c / 2))) for c in cells]


# --------------------------------------------------------- prepare and run

RTOL = 1e-10          # the solves' tolerance (the entry points' default)
PC = {"jacobi": cps.PC_JACOBI, "ic0": cps.PC_IC0, "reduced": cps.PC_REDUCED}
PREC = {"fp64": cps.FP64, "mixed": cps.MIXED}


def prepare(case, seed):
    ctx = _ctx()
    op = case["op"]
    if op == "batch":
        g = _gen(seed)
        systems, bs = [], []
        for n in _members(case, seed):
            xy, tri, d = _mesh(n, "lattice", g)
            eps, kinv = _fields(xy, n, "ensemble", g)
            systems.append(ctx.assemble(xy, tri, d, eps, kinv, cps.PER_VERTEX, cps.KIND_CP2,
                                        NU, DT))
            bs.append(_areas(xy, tri) * _normal(tri.shape[0], g))
        _keep(*systems)
        return {"case": case, "systems": systems, "bs": bs}
    if op == "chain":
        g, xy, tri, dirichlet, eps, theta, bs, targets = _chain_inputs(case, seed)
        model = cps.LogPermeabilityCorrector(ctx, xy, tri, dirichlet, eps, NU, DT,
                                             rtol=RTOL)
        _keep(model)
        return {"case": case, "model": model, "theta": theta, "bs": bs, "targets": targets}
    g, xy, tri, dirichlet, eps, kinv = _problem(case, seed)
    state = {"case": case}
    if op == "assemble":
        state["args"] = (xy, tri, dirichlet, eps, kinv, cps.PER_VERTEX, cps.KIND_CP2, NU, DT)
        return state
    if op == "cp1":
        walls = _walls(tri)
        sx, sy = (ctx.assemble(xy, tri, walls, eps, kinv, cps.PER_VERTEX, k, NU, DT)
                  for k in (cps.KIND_CP1_X, cps.KIND_CP1_Y))
        cps.cp1_setup(sx, sy, xy, tri, eps, kinv)
        _keep(sx, sy)
        state.update(sx=sx, sy=sy, du=_velocity(xy, tri, g, (0.05, 0.01), 0.02))
        return state
    s = ctx.assemble(xy, tri, dirichlet, eps, kinv, cps.PER_VERTEX, cps.KIND_CP2, NU, DT)
    state["sys"] = s
    _keep(s)
    if op == "matvec":
        state["x"] = _normal(tri.shape[0], g)
        return state
    if case["pc"] != "jacobi":
        s.set_precond(PC[case["pc"]])
    if op == "cp2":
        s.cp2_setup(xy, tri, eps, kinv)
        state.update(u=_velocity(xy, tri, g, (0.05, 0.01), 0.02),
                     g_k=_velocity(xy, tri, g, (0.0, 0.0), 1e-3))
        return state
    state["b"] = _areas(xy, tri) * _normal(tri.shape[0], g)
    return state


def _chain_inputs(case, seed):
    g = _gen(seed)
    xy, tri, dirichlet = _mesh(case["n"], "lattice", g)
    theta = -math.log(float(_kozeny(torch.tensor(0.4, dtype=F64)))) + \
        _fourier(xy[tri.long()].mean(1), g)
    eps = torch.full_like(theta, 0.4)
    area = _areas(xy, tri)
    bs = [area * _normal(area.numel(), g) for _ in range(case["steps"])]
    # noisy observations at scattered sensors, about one in 64 cells (none: NaN)
    seen = torch.rand(area.numel(), generator=g, device="cuda") < 1 / 64
    seen[:1] = True
    nothing = torch.full_like(area, math.nan)
    targets = [torch.where(seen, 3e5 * _normal(area.numel(), g), nothing)
               for _ in range(case["steps"])]
    return g, xy, tri, dirichlet, eps, theta, bs, targets


def _loss(xs, targets):
    return sum((torch.where(t.isnan(), 0.0, x - t) ** 2).sum() for x, t in zip(xs, targets))


def run(state):
    case = state["case"]
    op = case["op"]
    if op == "solve":
        x, _ = state["sys"].solve(state["b"], rtol=RTOL, precision=PREC[case["precision"]])
        return x
    if op == "batch":
        xs = [torch.zeros_like(b) for b in state["bs"]]
        cps.solve_batch(state["systems"], state["bs"], xs, rtol=RTOL,
                        precision=PREC[case["precision"]])
        return xs
    if op == "assemble":
        s = _ctx().assemble(*state["args"])
        out = s.export_matrix()
        s.free()
        return out
    if op == "chain":
        theta = state["theta"].detach().clone().requires_grad_(True)
        bs = [b.detach().clone().requires_grad_(True) for b in state["bs"]]
        xs = cps.chained_solve(state["model"], theta, bs, checkpoint_every=case["every"],
                               normalized=True)
        _loss(xs, state["targets"]).backward()
        return {"x": [x.detach() for x in xs], "dtheta": theta.grad, "db": [b.grad for b in bs]}
    if op == "cp2":
        out = state["sys"].cp2_step(state["u"], state["g_k"], rtol=RTOL)
        return {k: out[k] for k in ("eta_tilde", "eta", "u_next", "g_next", "flux")}
    if op == "cp1":
        du, _ = cps.cp1_step(state["sx"], state["sy"], state["du"],
                             precision=PREC[case["precision"]])
        return du
    return state["sys"].matvec(state["x"])


def _cells(case):
    n = case["n"]
    cells = 2 * (n - 1) ** 2
    if case.get("mesh") == "defect":
        cells += 2 * len(range(4, n - 3, 16)) ** 2
    return cells


def work(case):
    op = case["op"]
    # matrix rows: three values, three columns, the diagonal
    if op == "batch":
        cells = sum(2 * (n - 1) ** 2 for n in _members(case, 0))
        return {"bytes": cells * (44 + 16), "flops": cells * 8}
    c = _cells(case)
    if op == "assemble":        # xy, tri, eps and Kinv in; diagonal, columns and values out
        return {"bytes": c * (8 + 12 + 16) + c * 44, "flops": c * 150}
    if op == "chain":           # per step b, x, target in or out, and dtheta, db
        return {"bytes": c * (44 + 16 + case["steps"] * 32), "flops": c * 16 * case["steps"]}
    if op == "cp2":             # matrix, u and g in, two etas, u, g and fluxes out
        return {"bytes": c * (44 + 32 + 16 + 32 + 24), "flops": c * 150}
    if op == "cp1":             # both matrices, mass terms, du in and out
        return {"bytes": c * (2 * 44 + 24 + 32), "flops": c * 40}
    return {"bytes": c * (44 + 16), "flops": c * 8}


# ------------------------------------------------------- the same in 64 bits

def _neighbours(tri):
    """(cell across each local side or -1, that cell's local side)."""
    t = tri.long()
    nt = t.shape[0]
    a, b = t[:, [1, 2, 0]], t[:, [2, 0, 1]]
    key = (torch.minimum(a, b) * (int(t.max()) + 1) + torch.maximum(a, b)).reshape(-1)
    srt, order = torch.sort(key, stable=True)
    same = srt[1:] == srt[:-1]
    l, r = order[:-1][same], order[1:][same]
    other = torch.full((3 * nt,), -1, dtype=torch.int64, device=t.device)
    other[l], other[r] = r, l
    other = other.reshape(nt, 3)
    return torch.where(other >= 0, other // 3, other), torch.where(other >= 0, other % 3, other)


class _Geometry:
    def __init__(self, xy, tri):
        t = tri.long()
        self.tri = t
        self.nbr, self.side = _neighbours(tri)
        p = xy[t]
        a, b, c = p[:, 0], p[:, 1], p[:, 2]
        self.area = _areas(xy, tri)
        ba, ca = b - a, c - a
        b2, c2 = (ba * ba).sum(1), (ca * ca).sum(1)
        d = 4.0 * self.area
        cc = a + torch.stack([ca[:, 1] * b2 - ba[:, 1] * c2, ba[:, 0] * c2 - ca[:, 0] * b2],
                             1) / d[:, None]
        v, w = p[:, [1, 2, 0]], p[:, [2, 0, 1]]
        tv = w - v
        self.len = tv.norm(dim=2)
        self.nrm = torch.stack([tv[..., 1], -tv[..., 0]], 2) / self.len[..., None]
        self.inner = self.nbr >= 0
        far = torch.where(self.inner[..., None], cc[self.nbr.clamp(min=0)], 0.5 * (v + w))
        self.dist = ((far - cc[:, None, :]) * self.nrm).sum(2)


def _dirichlet_mask(nt, dirichlet):
    m = torch.zeros(3 * nt, dtype=torch.bool, device="cuda")
    m[dirichlet.long()] = True
    return m.reshape(nt, 3)


def _xi(eps, kinv):
    c = NU * eps * DT
    m00, m01, m11 = 1 + c * kinv[:, 0], c * kinv[:, 1], 1 + c * kinv[:, 2]
    det = m00 * m11 - m01 * m01
    return (eps * DT / det)[:, None] * torch.stack([m11, -m01, m00], 1)


def _cp2_sides(geo, dirichlet, xi_node):
    """T per side for nodal tensors: l n.Xi n / d, zero on a no-flux side."""
    t = geo.tri
    x = 0.5 * (xi_node[t[:, [1, 2, 0]]] + xi_node[t[:, [2, 0, 1]]])
    nx, ny = geo.nrm[..., 0], geo.nrm[..., 1]
    T = geo.len * (nx * nx * x[..., 0] + 2 * nx * ny * x[..., 1] + ny * ny * x[..., 2]) / geo.dist
    return torch.where(geo.inner | _dirichlet_mask(t.shape[0], dirichlet), T, torch.zeros_like(T))


class _Operator:
    """diag + off-diagonals -T on interior sides, and solves with it."""

    def __init__(self, geo, T, mass=None):
        e = torch.arange(T.shape[0], device="cuda")[:, None].expand(-1, 3)
        self.col = torch.where(geo.inner, geo.nbr, e).contiguous()
        self.off = torch.where(geo.inner, -T, torch.zeros_like(T)).contiguous()
        self.diag = T.sum(1) + (0 if mass is None else mass)

    def mul(self, x):
        return self.diag * x + (self.off * x[self.col]).sum(1)

    def solve(self, b, x0=None, tol=2e-15, rounds=4):
        """Jacobi-PCG rounds, each on the true residual of the one before."""
        x = torch.zeros_like(b) if x0 is None else x0.clone()
        nb = float(b.norm())
        if nb == 0.0:
            return torch.zeros_like(b)
        inv = 1.0 / self.diag
        last = math.inf
        for k in range(rounds):
            res = b - self.mul(x)
            rel = float(res.norm()) / nb
            if rel <= tol or rel > 0.3 * last:
                break
            last = rel
            x = x + self._pcg(res, inv, max(1e-13, 0.1 * tol / max(rel, tol)))
        return x

    def _pcg(self, b, inv, rtol):
        x, r = torch.zeros_like(b), b.clone()
        z = inv * r
        p, rho = z.clone(), torch.dot(r, z)
        stop = (rtol * b.norm()) ** 2
        for k in range(40000):
            q = self.mul(p)
            alpha = rho / torch.dot(p, q)
            x.addcmul_(p, alpha)
            r.addcmul_(q, -alpha)
            z = inv * r
            new = torch.dot(r, z)
            p = torch.addcmul(z, p, new / rho)
            rho = new
            # a mass-dominated system is solved in a handful of iterations
            if (k % 64 == 63 or (k < 64 and k % 2 == 1)) and not bool(torch.dot(r, r) > stop):
                break
        return x


class _ExactSolve(torch.autograd.Function):
    """x = A(T)^-1 b for side coefficients T, with its adjoint."""

    @staticmethod
    def forward(ctx, T, b, geo):
        op = _Operator(geo, T)
        x = op.solve(b)
        ctx.op, ctx.geo, ctx.x = op, geo, x
        return x

    @staticmethod
    def backward(ctx, g):
        lam, geo, x = ctx.op.solve(g), ctx.geo, ctx.x
        n = geo.nbr.clamp(min=0)
        far = torch.where(geo.inner, x[n], torch.zeros_like(geo.len))
        fl = torch.where(geo.inner, lam[n], torch.zeros_like(geo.len))
        # each interior side's coefficient appears once in either cell's row
        dT = torch.where(geo.inner, -lam[:, None] * (x[:, None] - far),
                         -lam[:, None] * x[:, None])
        return dT, lam, None


def _exact_chain(case, seed):
    g, xy, tri, dirichlet, eps, theta, bs, targets = _chain_inputs(case, seed)
    geo = _Geometry(xy, tri)
    theta = theta.clone().requires_grad_(True)
    bs = [b.clone().requires_grad_(True) for b in bs]
    xi = eps * DT / (1 + NU * eps * DT * torch.exp(-theta))
    far = torch.where(geo.inner, xi[geo.nbr.clamp(min=0)], xi[:, None].expand(-1, 3))
    live = geo.inner | _dirichlet_mask(tri.shape[0], dirichlet)
    T = torch.where(live, geo.len * 0.5 * (xi[:, None] + far) / geo.dist,
                    torch.zeros_like(geo.len))
    xs, prev = [], None
    for b in bs:
        rhs = b if prev is None else b + 0.1 * (torch.linalg.vector_norm(b) /
                                                torch.linalg.vector_norm(prev)) * prev
        prev = _ExactSolve.apply(T, rhs, geo)
        xs.append(prev)
    _loss(xs, targets).backward()
    return {"x": [x.detach() for x in xs], "dtheta": theta.grad, "db": [b.grad for b in bs]}


def _exact_cp1(case, seed):
    g, xy, tri, _, eps, kinv = _problem(case, seed)
    du = _velocity(xy, tri, g, (0.05, 0.01), 0.02)
    geo = _Geometry(xy, tri)
    T = NU * geo.len / geo.dist          # no-slip walls: every boundary side carries nu l / delta
    c = NU * eps * DT
    m = torch.stack([(1 + c * kinv[:, 0]) / DT, c * kinv[:, 1] / DT, (1 + c * kinv[:, 2]) / DT], 1)
    m = m[geo.tri].mean(1) * geo.area[:, None]
    ops = [_Operator(geo, T, m[:, 0]), _Operator(geo, T, m[:, 2])]
    lap = _Operator(geo, T)
    base = [-lap.mul(du[k]) for k in range(2)]
    x = [ops[k].solve(base[k]) for k in range(2)]
    for sweep in range(1000):
        new = [ops[k].solve(base[k] - m[:, 1] * x[1 - k], x0=x[k]) for k in range(2)]
        err = [float((new[k] - x[k]).norm() / x[k].norm()) for k in range(2)]
        x = new
        if min(err) <= 1e-4:
            break
    return torch.stack(x)


def exact(case, seed):
    op = case["op"]
    if op == "chain":
        return _exact_chain(case, seed)
    if op == "cp1":
        return _exact_cp1(case, seed)
    if op == "batch":
        g, xs = _gen(seed), []
        for n in _members(case, seed):
            xy, tri, d = _mesh(n, "lattice", g)
            eps, kinv = _fields(xy, n, "ensemble", g)
            b = _areas(xy, tri) * _normal(tri.shape[0], g)
            geo = _Geometry(xy, tri)
            xs.append(_Operator(geo, _cp2_sides(geo, d, _xi(eps, kinv))).solve(b))
        return xs
    g, xy, tri, dirichlet, eps, kinv = _problem(case, seed)
    geo = _Geometry(xy, tri)
    T = _cp2_sides(geo, dirichlet, _xi(eps, kinv))
    A = _Operator(geo, T)
    if op == "assemble":
        return A.diag, None, A.off.t().contiguous()
    if op == "matvec":
        return A.mul(_normal(tri.shape[0], g))
    if op == "cp2":
        # the first solution only: its right-hand side is the mean side flux
        u = _velocity(xy, tri, g, (0.05, 0.01), 0.02)
        un = (u[0][:, None] * geo.nrm[..., 0] + u[1][:, None] * geo.nrm[..., 1])
        n = geo.nbr.clamp(min=0)
        far, af = un[n, geo.side.clamp(min=0)], geo.area[n]
        a = geo.area[:, None]
        f = torch.where(geo.inner, (un * af - far * a) / (a + af), un) * geo.len
        f = torch.where(geo.inner | _dirichlet_mask(tri.shape[0], dirichlet), f,
                        torch.zeros_like(f))
        return {"eta_tilde": A.solve(f.sum(1)), "eta": None, "u_next": None, "g_next": None,
                "flux": None}
    return A.solve(_areas(xy, tri) * _normal(tri.shape[0], g))
