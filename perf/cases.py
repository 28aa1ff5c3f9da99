"""The workloads that this library is timed on: its public calls (Solver.solve, solve_host, apply, apply_T,
Group.solve and the differentiable solve) on the domains and sizes of its benchmark and tests.

Every state is a fresh set-up of its domain with seeded inputs: u* is the exact cell averages of a sum of plane
waves (closed form on pure cells, the library's cut-cell quadrature on the others), g the boundary averages of the
same function, and f = L u* + N g evaluated in 64 bits by plain torch from the stencil's weights and the fitted
rows of the set-up handle.  The discrete solution of (f, g) is then u* itself, and f is the manufactured
right-hand side up to the discretisation's truncation error."""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2504_00724_gb300 as ccm
from paper_2504_00724_gb300 import autograd

CIRCLE, ELLIPSE, STAR, POLYGON = 1, 2, 3, 4

MAX_CYCLES = 200

# the grids of the many-geometry workload, mixed in one group
GROUP_GRIDS = (128, 256, 512, 1024)


# ---------------------------------------------------------------- the cases

def listed():
    return [
        # the smallest benchmark configuration: Poisson outside a disk, FP64 V-cycles; one call is all latency
        dict(name="disk64_fp64", op="solve", domain="disk", n=64, precision="fp64", rtol=1e-10, coarsest=16),
        # the star configuration at its smallest grid, the default mixed form: a solve inside a user's loop
        dict(name="star256_mixed", op="solve", domain="star", n=256, precision="mixed", rtol=1e-10, coarsest=16),
        # the paper's Problem 3 (ii), a rotated box on a 3n/2 grid: a ragged size, a polygon and a mixed derivative
        dict(name="box960_mixed", op="solve", domain="box", n=960, precision="mixed", rtol=1e-10, coarsest=16),
        # the headline configuration: one large solve in the mixed form
        dict(name="star4096_mixed", op="solve", domain="star", n=4096, precision="mixed", rtol=1e-10, coarsest=64),
        # the same star in plain FP64, for users who do not want FP32 cycles
        dict(name="star1024_fp64", op="solve", domain="star", n=1024, precision="fp64", rtol=1e-10, coarsest=64),
        # Neumann data on three holes, the GMRES-corrected mixed form
        dict(name="ellipses1024_gmres", op="solve", domain="ellipses", n=1024, precision="mixed", rtol=1e-10,
             coarsest=32, krylov=2),
        # many right-hand sides on one geometry, advanced together
        dict(name="disk512_batch64", op="solve", domain="disk", n=512, precision="mixed", rtol=1e-10, coarsest=16,
             nrhs=64),
        # many geometries of uneven grid sizes in one graph launch
        dict(name="group12", op="group", domain="mix", n=1024, precision="mixed", rtol=1e-10, coarsest=32, count=12),
        # data fitting: the differentiable solve forward and backward (gradients to f and g), FP64
        dict(name="star1024_adjoint", op="adjoint", domain="star", n=1024, b=0.3, c=1.0, precision="fp64",
             rtol=1e-10, coarsest=16),
        # f, g and u in pinned host memory, through the host-buffer call
        dict(name="star2048_host", op="host", domain="star", n=2048, precision="mixed", rtol=1e-10, coarsest=64),
        # the operator alone, as a residual check or inside a user's own iteration
        dict(name="star4096_apply", op="apply", domain="star", n=4096, precision="mixed", coarsest=64, nrhs=1),
        # its transpose on several vectors, Poisson on a grid that is not a power of two
        dict(name="disk1408_applyT", op="apply_T", domain="disk", n=1408, precision="mixed", coarsest=16, nrhs=4),
    ]


def _odd_grid(rng, lo, hi):
    """A grid size in [lo, hi], spread over its logarithm, that halves down to 10 - 16 cells (on 9, 12 and 14 cells
    the disk's coarsest level is degenerate and the set-up refuses it)."""
    n = lo * (hi / lo) ** rng.random()
    sizes = [m * 2 ** k for k in range(9) for m in (10, 11, 13, 15, 16)]
    return min((m for m in sizes if lo <= m <= hi), key=lambda m: abs(m - n))


def draw(rng):
    op = rng.choice(["solve"] * 6 + ["batch", "group", "adjoint", "host", "apply", "apply_T"])
    if op == "group":
        return dict(op="group", domain="mix", n=1024, precision="mixed", rtol=1e-10, coarsest=32,
                    count=rng.randint(2, 12), first=rng.randint(1, 1000))
    domain = rng.choice(["disk", "star", "box"])
    c = dict(op="solve" if op == "batch" else op, domain=domain, precision=rng.choice(["mixed", "mixed", "fp64"]),
             rtol=10.0 ** rng.uniform(-11, -9), coarsest=16)
    if op == "adjoint":
        c["n"] = _odd_grid(rng, 64, 1024)
        c.update(precision="fp64", rtol=1e-10)
    elif op == "batch":
        c["n"] = _odd_grid(rng, 64, 512)
        c.update(precision="mixed", nrhs=max(2, min(64, round(64 ** rng.random() * (512 / c["n"]) ** 0.5))))
    elif op in ("apply", "apply_T"):
        c["n"] = _odd_grid(rng, 64, 2048)
        c["nrhs"] = rng.randint(1, 4)
    else:
        c["n"] = _odd_grid(rng, 64, 3072 if c["precision"] == "mixed" else 1024)
        if op == "solve" and domain == "disk" and c["precision"] == "mixed" and rng.random() < 0.4:
            c.update(domain="ellipses", krylov=2, n=_odd_grid(rng, 256, 1024))
    if domain == "star":
        c.update(r0=round(rng.uniform(0.25, 0.32), 4), amp=round(rng.uniform(0.05, 0.08), 4), k=rng.randint(3, 5))
    if c["n"] >= 1024:
        c["coarsest"] = 64
    if rng.random() < 0.3 and c["domain"] in ("disk", "star"):
        c["a"], c["b"], c["c"] = 1.0, round(rng.uniform(-0.5, 0.5), 3), round(rng.uniform(0.8, 2.0), 3)
    return c


# ---------------------------------------------------------------- domains

def _curve(kind, params, orient, bc):
    return SimpleNamespace(kind=kind, params=params, orient=orient, bc=bc, robin=(1.0, 0.0))


def _problem(a, b, c, x0, h, n, box_bc, curves):
    return SimpleNamespace(a=a, b=b, c=c, x0=x0, y0=x0, h=h, nx=n, ny=n, box_bc=box_bc, curves=curves)


def _domain(case):
    """The problem of a case: the unit square minus a disk of radius 0.2, the interior of a star, the unit box
    rotated by pi/6, or the unit square minus three ellipses."""
    d, n = case["domain"], int(case["n"])
    a = case.get("a", 1.0)
    if d == "disk":
        return _problem(a, case.get("b", 0.0), case.get("c", 1.0), 0.0, 1.0 / n, n, ccm.CCM_DIRICHLET,
                        [_curve(CIRCLE, (0.5, 0.5, 0.2), -1, ccm.CCM_DIRICHLET)])
    if d == "star":
        p = (0.5, 0.5, case.get("r0", 0.3), case.get("amp", 0.08), float(case.get("k", 5)))
        return _problem(a, case.get("b", 0.5), case.get("c", 2.0), 0.0, 1.0 / n, n, ccm.CCM_NONE,
                        [_curve(STAR, p, +1, ccm.CCM_DIRICHLET)])
    if d == "box":
        # n cells a side of the square [-1/4, 5/4]^2 that holds the rotated unit box
        co, si, pts = math.cos(math.pi / 6), math.sin(math.pi / 6), []
        for x, y in ((-0.5, -0.5), (0.5, -0.5), (0.5, 0.5), (-0.5, 0.5)):
            pts += [0.5 + co * x - si * y, 0.5 + si * x + co * y]
        return _problem(1.25, -math.sqrt(3.0) / 2, 1.75, -0.25, 1.5 / n, n, ccm.CCM_NONE,
                        [_curve(POLYGON, tuple(pts), +1, ccm.CCM_DIRICHLET)])
    if d == "ellipses":
        e = [(0.27, 0.3, 0.10, 0.06, 0.4), (0.73, 0.33, 0.08, 0.08, 0.0), (0.48, 0.72, 0.12, 0.05, 2.1)]
        return _problem(1.0, 0.0, 1.0, 0.0, 1.0 / n, n, ccm.CCM_DIRICHLET,
                        [_curve(ELLIPSE, p, -1, ccm.CCM_NEUMANN) for p in e])
    raise ValueError(d)


def _members(case):
    """The members of a group: grids, kinds and shapes spread over the many-geometry workload's ranges."""
    out = []
    for k in range(int(case["count"])):
        r = np.random.default_rng([int(case.get("first", 0)), k])
        n = int(GROUP_GRIDS[(k + int(case.get("first", 0))) % 4])
        if r.integers(0, 2) == 0:
            m = dict(domain="star", n=n, coarsest=64, r0=float(r.uniform(0.25, 0.32)), amp=float(r.uniform(0.05, 0.08)),
                     k=int(r.integers(3, 6)))
        else:
            m = dict(domain="ellipses", n=n, coarsest=32, krylov=2)
        out.append(dict(m, precision="mixed", rtol=case["rtol"]))
    return out


def _solver(case):
    kw = dict(precision=ccm.CCM_FP64 if case["precision"] == "fp64" else ccm.CCM_MIXED, rtol=case.get("rtol", 1e-10),
              max_iter=MAX_CYCLES, coarsest=int(case["coarsest"]), krylov=int(case.get("krylov", 0)))
    if case["op"] == "solve" and case.get("nrhs", 1) > 1:
        kw["batch"] = int(case["nrhs"])
    return ccm.Solver(_domain(case), **kw)


# ---------------------------------------------------------------- inputs

def _waves(seed, k):
    """Amplitude, wave numbers and phase of six plane waves."""
    r = np.random.default_rng([int(seed), int(k)])
    return [(r.normal(), r.uniform(0.3, 4) * math.pi, r.uniform(-4, 4) * math.pi, r.uniform(0, 2 * math.pi))
            for _ in range(6)]


def _geometry(s):
    """What the inputs need of a set-up handle, on the GPU."""
    st, _, rg, _ = s.cell_map()
    cell, cols, beta, nb, seg = s.level_rows(0)
    cq, cxy, cw, sq, bxy, bw, bn = s.quadrature()
    cq_cells, cq = np.unique(cq, return_inverse=True)
    dev = lambda x: torch.as_tensor(x, device="cuda")  # noqa: E731
    return SimpleNamespace(
        p=s.prob, nseg=s.nseg, live=dev(st != 0), reg=dev(rg != 0), cell=dev(cell.astype(np.int64)),
        cols=dev(cols.astype(np.int64)), beta=dev(beta), nb=dev(nb), seg=dev(seg.astype(np.int64)),
        gam=dev(s.boundary_operator()), cq=dev(cq), cq_cells=dev(cq_cells.astype(np.int64)), cxy=dev(cxy), cw=dev(cw), sq=dev(sq.astype(np.int64)),
        bxy=dev(bxy), bw=dev(bw), bn=dev(bn))


def _sums(at, values, n):
    """values summed by their index, in a fixed order (on the host: the same inputs from the same seed)."""
    return torch.as_tensor(np.bincount(at.cpu().numpy(), values.cpu().numpy(), n), device="cuda")


def _averages(G, waves):
    """(u, g): cell averages of the waves over the cells (0 on empty ones), boundary averages over the segments."""
    p, h = G.p, G.p.h
    x = p.x0 + h * (torch.arange(p.nx, dtype=torch.float64, device="cuda") + 0.5)
    y = p.y0 + h * (torch.arange(p.ny, dtype=torch.float64, device="cuda") + 0.5)
    u = torch.zeros((p.ny, p.nx), dtype=torch.float64, device="cuda")
    val, dx, dy, fq = (torch.zeros(n, dtype=torch.float64, device="cuda") for n in (len(G.bw), len(G.bw), len(G.bw), len(G.cw)))
    for am, kx, ky, ph in waves:
        si = am * np.sinc(kx * h / 2 / math.pi) * np.sinc(ky * h / 2 / math.pi)
        ax, ay = kx * x, ky * y + ph
        u += si * (torch.sin(ax)[None, :] * torch.cos(ay)[:, None] + torch.cos(ax)[None, :] * torch.sin(ay)[:, None])
        fq += am * torch.sin(kx * G.cxy[:, 0] + ky * G.cxy[:, 1] + ph)
        t = kx * G.bxy[:, 0] + ky * G.bxy[:, 1] + ph
        val += am * torch.sin(t)
        dx += am * kx * torch.cos(t)
        dy += am * ky * torch.cos(t)
    u *= G.live
    u.view(-1)[G.cq_cells] = _sums(G.cq, fq * G.cw, len(G.cq_cells)) / _sums(G.cq, G.cw, len(G.cq_cells))
    gam = G.gam[G.sq]
    gn = G.bw * (gam[:, 0] * val + gam[:, 1] * (dx * G.bn[:, 0] + dy * G.bn[:, 1]))
    return u, _sums(G.sq, gn, G.nseg) / _sums(G.sq, G.bw, G.nseg)


def _weights(p):
    """The regular stencil's weights [dj + 2][di + 2] times h^2 (eq. stdLap along x and y, eq. stdGrad twice)."""
    lap = np.array([-1.0, 16.0, -30.0, 16.0, -1.0]) / 12
    gra = np.array([1.0, -8.0, 0.0, 8.0, -1.0]) / 12
    w = p.b * np.outer(gra, gra)
    w[2, :] += p.a * lap
    w[:, 2] += p.c * lap
    return w


def _apply64(G, u, g):
    """L u + N g by plain torch in 64 bits."""
    p, w = G.p, _weights(G.p)
    pad = torch.nn.functional.pad(u, (2, 2, 2, 2))
    out = torch.zeros_like(u)
    for dj in range(5):
        for di in range(5):
            if w[dj, di] != 0:
                out += w[dj, di] * pad[dj:dj + p.ny, di:di + p.nx]
    out = torch.where(G.reg, out / p.h ** 2, 0.0).reshape(-1)
    rows = (G.beta * u.reshape(-1)[G.cols]).sum(1)
    if g is not None:
        rows = rows + torch.where(G.seg >= 0, G.nb * g[G.seg.clamp(min=0)], 0.0)
    out[G.cell] = rows
    return out.view_as(u)


def _apply_T64(G, v):
    """(L^T v, N^T v) by plain torch in 64 bits."""
    p, w = G.p, _weights(G.p)
    pad = torch.nn.functional.pad(torch.where(G.reg, v, 0.0), (2, 2, 2, 2))
    out = torch.zeros_like(v)
    for dj in range(5):
        for di in range(5):
            if w[dj, di] != 0:
                out += w[dj, di] * pad[4 - dj:4 - dj + p.ny, 4 - di:4 - di + p.nx]
    out = (out / p.h ** 2).reshape(-1)
    vr = v.reshape(-1)[G.cell]
    out.index_add_(0, G.cols.reshape(-1), (G.beta * vr[:, None]).reshape(-1))
    og = torch.zeros(G.nseg, dtype=torch.float64, device="cuda")
    on = G.seg >= 0
    og[G.seg[on]] = (G.nb * vr)[on]
    return out.view_as(v) * G.live, og


def _fields(G, seed, nrhs, k0=0):
    """nrhs seeded (u*, g), stacked."""
    us, gs = zip(*[_averages(G, _waves(seed, k0 + k)) for k in range(nrhs)])
    return torch.stack(us), torch.stack(gs)


def _rhs(G, us, gs):
    return torch.stack([_apply64(G, u, g) for u, g in zip(us, gs)])


def prepare(case, seed):
    op, nrhs = case["op"], int(case.get("nrhs", 1))
    if op == "group":
        ss, fs, gs = [], [], []
        for k, m in enumerate(_members(case)):
            s = _solver(dict(m, op="solve"))
            G = _geometry(s)
            u, g = _fields(G, seed, 1, k)
            ss.append(s)
            fs.append(_rhs(G, u, g)[0])
            gs.append(g[0])
        return SimpleNamespace(op=op, group=ccm.Group(ss), f=fs, g=gs)
    s = _solver(case)
    G = _geometry(s)
    us, gs = _fields(G, seed, nrhs)
    if op == "apply":
        return SimpleNamespace(op=op, s=s, u=us, g=gs)
    if op == "apply_T":
        return SimpleNamespace(op=op, s=s, v=us)
    f = _rhs(G, us, gs)
    if op == "adjoint":
        # the fit's target: another field of the same kind with noise of standard deviation 1e-3
        t = _averages(G, _waves(seed, 1000))[0]
        gen = torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 31))
        t = t + 1e-3 * torch.randn(t.shape, generator=gen, dtype=torch.float64, device="cuda") * G.live
        return SimpleNamespace(op=op, s=s, f=f[0].requires_grad_(), g=gs[0].requires_grad_(), target=t)
    if op == "host":
        pin = lambda t: t.cpu().pin_memory()  # noqa: E731
        return SimpleNamespace(op=op, s=s, f=pin(f[0]), g=pin(gs[0]), u=torch.zeros_like(f[0], device="cpu").pin_memory())
    return SimpleNamespace(op=op, s=s, f=f if nrhs > 1 else f[0], g=gs if nrhs > 1 else gs[0])


def run(state):
    if state.op == "solve":
        return state.s.solve(state.f, state.g)[0]
    if state.op == "group":
        return state.group.solve(state.f, state.g)[0]
    if state.op == "host":
        return state.s.solve_host(state.f, state.g, state.u.zero_())[0]
    if state.op == "apply":
        return state.s.apply(state.u, state.g)
    if state.op == "apply_T":
        return state.s.apply_T(state.v)
    u = autograd.solve(state.s, state.f, state.g)
    loss = 0.5 * ((u - state.target) ** 2).sum()
    df, dg = torch.autograd.grad(loss, (state.f, state.g))
    return u.detach(), df, dg


def exact(case, seed):
    """The discrete solution is u* by construction; the operator's values come from plain torch in 64 bits.  Of
    this library only the set-up handle's numbers are used (cell map, fitted rows, quadrature nodes): they are the
    operator that a call is given."""
    op, nrhs = case["op"], int(case.get("nrhs", 1))
    if op == "group":
        return [_fields(_geometry(_solver(dict(m, op="solve"))), seed, 1, k)[0][0] for k, m in enumerate(_members(case))]
    G = _geometry(_solver(case))
    us, gs = _fields(G, seed, nrhs)
    if op == "apply":
        return torch.stack([_apply64(G, u, g) for u, g in zip(us, gs)])
    if op == "apply_T":
        ou, og = zip(*[_apply_T64(G, v) for v in us])
        return torch.stack(ou), torch.stack(og)
    if op == "adjoint":
        return us[0], None, None      # the gradients' exact values would take another solver
    u = us if nrhs > 1 else us[0]
    return u.cpu() if op == "host" else u


# ---------------------------------------------------------------- work

def _size(case):
    """(unknowns, irregular rows) of a case, from its area and boundary length."""
    n, d = case["n"], case["domain"]
    if d == "star":
        r0, am, k = case.get("r0", 0.3), case.get("amp", 0.08), case.get("k", 5)
        area, length = math.pi * (r0 * r0 + am * am / 2), 2 * math.pi * math.sqrt(r0 * r0 + am * am / 2 + (k * am) ** 2 / 2)
    elif d == "disk":
        area, length = 1 - math.pi * 0.04, 4 + 0.4 * math.pi
    elif d == "box":
        area, length = 1 / 2.25, 4 / 1.5
    else:
        area, length = 1 - math.pi * (0.006 + 0.0064 + 0.006), 4 + 1.6
    return area * n * n, 3.0 * length * n


def work(case):
    """Bytes: the right-hand sides (or vectors) read and the results written, and the operator of the irregular
    cells (15 coefficients and columns a row) read once.  Flops: one application is 2 x 25 (9 taps without the mixed
    term) a cell; a solve to its tolerance takes V-cycles of factor 0.28 with seven such passes over the levels."""
    if case["op"] == "group":
        ws = [work(dict(m, op="solve")) for m in _members(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    cells, rows = _size(case)
    nrhs = int(case.get("nrhs", 1))
    taps = 9 if case["domain"] in ("disk", "ellipses") and not case.get("b") else 25
    one = 2.0 * taps * cells
    if case["op"] in ("apply", "apply_T"):
        return {"bytes": nrhs * 16.0 * cells + 180.0 * rows, "flops": nrhs * one}
    cycles = math.ceil(math.log(case["rtol"]) / math.log(0.28))
    passes = 7 * 4 / 3 * cycles * (2 if case["op"] == "adjoint" else 1)
    return {"bytes": nrhs * (32.0 if case["op"] == "adjoint" else 16.0) * cells + 180.0 * rows, "flops": nrhs * passes * one}
