"""Measured workloads of the Newton-multigrid solver.

A case is one call that a user's program makes: Crank-Nicolson steps of one
domain whose state lives on the device (``Domain.step`` between
``set_state_device`` and ``get_state_device``), of a batch of domains
(``Batch.step``), or a stream of serving jobs (``Server.submit`` / ``wait`` on
host arrays).  Geometries, model constants, grid sizes and time steps are those
of the repository's workloads, tests and serving study; the seed draws each
geometry's parameters and the boundary value.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1902_07029_gb300 as sulf

# a, d, m_s, m_c, alpha, beta (the paper's constants), then s_ext, s0, c0
MODEL = (1.0e4, 0.1, 64.06, 100.09, 0.01, 0.1)
S0, C0 = 0.0, 10.0
DEV = torch.device("cuda" if torch.cuda.is_available() else "cpu")

# A CN step takes about this many Newton iterations and V(2,2) cycles
NEWTON, CYCLES = 4, 50


def listed():
    return [
        # the smallest domain in use (65^2 disk, the smoke test's): every
        # kernel is a few microseconds, launches and latency are the time
        _step("step_disk65_fp64", 2, 64, 8, "disk", "fp64", 2),
        # ordinary 2-D jobs of the serving and batch studies
        _step("step_star257_mixed", 2, 256, 8, "random_star", "mixed", 2),
        # the paper's Neumann condition, on a size that is no power of two
        _step("step_neumann_star321_fp64", 2, 320, 10, "random_star", "fp64", 2, bc=1),
        # the 2-D benchmark, five-lobed star at 1025^2, both precisions
        _step("step_star1025_fp64", 2, 1024, 8, "star", "fp64", 1),
        _step("step_star1025_mixed", 2, 1024, 8, "star", "mixed", 1),
        # the largest 2-D serving job
        _step("step_star2049_mixed", 2, 2048, 8, "random_star", "mixed", 1),
        # small, medium and headline 3-D boxes
        _step("step_box65_mixed", 3, 64, 4, "box", "mixed", 1),
        _step("step_box129_fp64", 3, 128, 4, "box", "fp64", 1),
        _step("step_box257_fp64", 3, 256, 4, "box", "fp64", 1),
        _step("step_box257_mixed", 3, 256, 4, "box", "mixed", 1),
        # the batching study: random stars of four sizes, lock-step, mixed
        dict(name="batch32_mixed", kind="batch", sizes="128,256,512,1024", instances=32, precision="mixed", steps=10,
             lockstep=True),
        # the serving study: jobs of both dimensions from host level sets to
        # host states, domain set-up included
        dict(name="serve8_mixed", kind="serve", sizes2="256,512,1024", sizes3="64", jobs=8, precision="mixed", steps=20,
             workers=4),
    ]


def _step(name, dim, N, coarsest, shape, precision, steps, bc=0, size=1.0):
    c = dict(kind="step", dim=dim, N=N, coarsest=coarsest, shape=shape, size=size, precision=precision, steps=steps,
             bc=bc)
    if name:
        c["name"] = name
    return c


def draw(rng):
    precision = rng.choice(["fp64", "mixed"])
    what = rng.random()
    if what < 0.15:
        sizes = sorted(rng.sample([96, 128, 160, 192, 256, 320, 384, 512, 640, 768, 1024], 3))
        return dict(kind="batch", sizes=",".join(str(n) for n in sizes), instances=rng.randint(6, 12),
                    precision=precision, steps=rng.randint(2, 4), lockstep=rng.random() < 0.7)
    if what < 0.25:
        sizes = rng.sample([128, 192, 256, 384, 512, 768, 1024], 3)
        return dict(kind="serve", sizes2=",".join(str(n) for n in sizes), sizes3=str(rng.choice([64, 80])),
                    jobs=rng.randint(4, 6), precision=precision, steps=rng.randint(5, 12), workers=rng.randint(2, 6))
    size = round(rng.uniform(0.75, 0.97), 3)
    if what < 0.65:
        N, coarsest = _size(rng, 64, 2048, range(8, 16))
        steps = rng.randint(1, 3) if N < 600 else 1
        bc = 1 if rng.random() < 0.2 else 0
        return _step("", 2, N, coarsest, rng.choice(["disk", "star", "random_star"]), precision, steps, bc, size)
    N, coarsest = _size(rng, 64, 256, (3, 4, 5))
    return _step("", 3, N, coarsest, "box", precision, 1, 0, size)


def _size(rng, lo, hi, coarsest):
    """N = coarsest * 2^k near a size spread over the logarithm of [lo, hi]."""
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(((c << k, c) for c in coarsest for k in range(10) if lo <= c << k <= hi),
               key=lambda t: (abs(math.log(t[0] / want)) // 0.05, rng.random()))


def _coarsest(N):
    """The smallest coarsest level of 8 to 15 intervals that N refines."""
    return next(c for c in range(8, 16) if N % c == 0 and (N // c) & (N // c - 1) == 0)


def _dt(dim, N):
    """dt = h; smaller on the coarse grids, where the boundary layer is
    thinner than h and some domains have no discrete solution at dt = h."""
    if dim == 2:
        f = 0.25 if N <= 96 else 0.5 if N < 128 else 1.0
    else:
        f = 0.25 if N <= 96 else 0.5 if N <= 160 else 1.0
    return f * 2.0 / N


# ---- inputs ----

def _levelset(dim, N, shape, seed, size=1.0):
    """phi on the (N+1)^dim nodes of [-1, 1]^dim (x fastest) of the shape
    scaled by `size`, and s_ext."""
    r = np.random.default_rng([seed, dim, N])
    x = (-1.0 + (2.0 / N) * torch.arange(N + 1, dtype=torch.float64, device=DEV)) / size
    s_ext = float(r.uniform(0.5, 1.0))
    if dim == 3:
        b, rho = r.uniform(0.55, 0.62), r.uniform(0.17, 0.21)
        o = r.uniform(-0.02, 0.02, 3)
        q = [((x - float(v)).abs() - float(b)).clamp(min=0.0) ** 2 for v in o]
        phi = (q[0][None, None, :] + q[1][None, :, None] + q[2][:, None, None]).sqrt() - float(rho)
        return phi, s_ext
    Y, X = torch.meshgrid(x, x, indexing="ij")
    if shape == "disk":
        ox, oy = r.uniform(-0.05, 0.05, 2)
        return ((X - float(ox)) ** 2 + (Y - float(oy)) ** 2).sqrt() - float(r.uniform(0.75, 0.82)), s_ext
    rad, th = (X * X + Y * Y).sqrt(), torch.atan2(Y, X)
    if shape == "star":
        return rad - float(r.uniform(0.57, 0.62)) - 0.2 * torch.sin(5 * th + float(r.uniform(0, 2 * math.pi))), s_ext
    phi = rad - 0.5
    for k in range(2, 7):
        phi = phi - float(r.uniform(0.0, 0.05)) * torch.sin(k * th + float(r.uniform(0, 2 * math.pi)))
    return phi, s_ext


def _domain(phi, dim, N, coarsest, s_ext, precision, bc=0):
    d = sulf.Domain(phi.cpu().numpy(), dim, (-1.0, 1.0), N, coarsest)
    d.set_model(MODEL + (s_ext, S0, C0))
    if bc:
        d.set_bc(bc)
    d.set_solver(precision=1 if precision == "mixed" else 0)
    return d


def _instances(case):
    sizes = [int(v) for v in case["sizes"].split(",")]
    return [sizes[i % len(sizes)] for i in range(case["instances"])]


def _jobs(case):
    two = [int(v) for v in case["sizes2"].split(",")]
    three = [int(v) for v in case["sizes3"].split(",")]
    jobs = []
    for i in range(case["jobs"]):
        N = three[i % len(three)] if i % 4 == 3 else two[i % len(two)]
        jobs.append((3, N, 5 if N % 5 == 0 else 4) if i % 4 == 3 else (2, N, _coarsest(N)))
    return jobs


def prepare(case, seed):
    if case["kind"] == "serve":
        jobs = []
        for i, (dim, N, coarsest) in enumerate(_jobs(case)):
            phi, s_ext = _levelset(dim, N, "random_star" if dim == 2 else "box", 1000 * seed + i)
            jobs.append((phi.cpu().numpy(), dim, N, coarsest, MODEL + (s_ext, S0, C0), _dt(dim, N)))
        return dict(case=case, jobs=jobs, server=sulf.Server(64 << 30, case["workers"]))
    if case["kind"] == "batch":
        doms, dts, n = [], [], 0
        for i, N in enumerate(_instances(case)):
            phi, s_ext = _levelset(2, N, "random_star", 1000 * seed + i)
            doms.append(_domain(phi, 2, N, _coarsest(N), s_ext, case["precision"]))
            dts.append(_dt(2, N))
            n += (N + 1) ** 2
        b = sulf.Batch(doms, nstreams=16, lockstep=case["lockstep"])
        return dict(case=case, doms=doms, batch=b, dts=dts, **_buffers(n))
    phi, s_ext = _levelset(case["dim"], case["N"], case["shape"], seed, case["size"])
    d = _domain(phi, case["dim"], case["N"], case["coarsest"], s_ext, case["precision"], case["bc"])
    return dict(case=case, dom=d, **_buffers(d.nn))


def _buffers(n):
    """Device buffers of a program that keeps its states: the initial one
    (values at inactive nodes are ignored) and the one read back."""
    s0 = torch.full((n,), S0, dtype=torch.float64, device=DEV)
    c0 = torch.full((n,), C0, dtype=torch.float64, device=DEV)
    st = dict(s0=s0, c0=c0, s=torch.empty_like(s0), c=torch.empty_like(c0))
    torch.cuda.synchronize()
    return st


# ---- one pass ----

def run(state):
    case = state["case"]
    if case["kind"] == "serve":
        srv = state["server"]
        ids = [srv.submit(phi, dim, N, model, dt, case["steps"], coarsest_N=coarsest,
                          precision=1 if case["precision"] == "mixed" else 0)
               for phi, dim, N, coarsest, model, dt in state["jobs"]]
        return [list(srv.wait(j)[:2]) for j in ids]
    s0, c0, s, c = state["s0"], state["c0"], state["s"], state["c"]
    if case["kind"] == "batch":
        at = 0
        for d in state["doms"]:
            d.set_state_device(s0.data_ptr() + 8 * at, c0.data_ptr() + 8 * at)
            at += d.nn
        state["batch"].step(state["dts"], case["steps"])
        at = 0
        for d in state["doms"]:
            d.get_state_device(s.data_ptr() + 8 * at, c.data_ptr() + 8 * at)
            at += d.nn
    else:
        d = state["dom"]
        d.set_state_device(s0.data_ptr(), c0.data_ptr())
        d.step(_dt(case["dim"], case["N"]), case["steps"])
        d.get_state_device(s.data_ptr(), c.data_ptr())
    return {"s": s, "c": c}


# ---- what a pass cannot do without ----

def _step_work(dim, N, precision, steps, share):
    """Per CN step and active node: the old-time part reads and writes 32 B;
    a Newton iteration's residual 48 B and update 32 B; a V(2,2) cycle, with
    the coefficients recomputed from (s, c), four relaxation sweeps at 64 B,
    residual and restriction 52 B, prolongation 36 B, times the hierarchy's
    factor (half of that in FP32).  share: active nodes per box node."""
    active = share * (N + 1) ** dim
    cycle = 344.0 * (4 / 3 if dim == 2 else 8 / 7) * (0.5 if precision == "mixed" else 1.0)
    sweep = 22 if dim == 2 else 30
    return (active * steps * (32 + NEWTON * 80 + CYCLES * cycle),
            active * steps * (NEWTON * 140 + CYCLES * 6 * sweep))


def work(case):
    if case["kind"] == "serve":
        parts = [_step_work(d, N, case["precision"], case["steps"], 0.2 if d == 2 else 0.45) for d, N, _ in _jobs(case)]
    elif case["kind"] == "batch":
        parts = [_step_work(2, N, case["precision"], case["steps"], 0.2) for N in _instances(case)]
    else:
        share = 0.45 if case["dim"] == 3 else {"disk": 0.5, "star": 0.3, "random_star": 0.2}[case["shape"]]
        parts = [_step_work(case["dim"], case["N"], case["precision"], case["steps"], share * case["size"] ** case["dim"])]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


# ---- the same steps in plain 64-bit torch ----

def exact(case, seed):
    """The discrete CN system solved to rounding: level-set geometry of the
    finest grid, Newton, and a GMRES solve of its equation for s alone (the c
    equations are pointwise and eliminated)."""
    if case["kind"] != "step":
        return None  # many domains one after the other: over 20 seconds
    phi, s_ext = _levelset(case["dim"], case["N"], case["shape"], seed, case["size"])
    g = _geometry(phi, case["dim"], case["N"], case["bc"])
    n = g["ni"] + g["ng"]
    s = torch.full((n,), S0, dtype=torch.float64, device=DEV)
    c = torch.full((n,), C0, dtype=torch.float64, device=DEV)
    for _ in range(case["steps"]):
        s, c = _cn_step(g, s, c, _dt(case["dim"], case["N"]), 2.0 / case["N"], s_ext)
    out = {}
    for name, v in (("s", s), ("c", c)):
        box = torch.zeros(phi.numel(), dtype=torch.float64, device=DEV)
        box[g["node"]] = v
        out[name] = box
    return out


def _basis(order, xi):
    """1-D Lagrange values and derivatives at local coordinate xi of the
    offsets 0, 1, 2 (coordinates 1, 0, -1), per-entry order 0, 1 or 2."""
    one, zero = torch.ones_like(xi), torch.zeros_like(xi)
    v = {0: (one, zero, zero), 1: (xi, 1 - xi, zero), 2: (xi * (1 + xi) / 2, (1 - xi) * (1 + xi), xi * (xi - 1) / 2)}
    d = {0: (zero, zero, zero), 1: (one, -one, zero), 2: (xi + 0.5, -2 * xi, xi - 0.5)}
    pick = lambda t: torch.stack([torch.where(order == 2, t[2][k], torch.where(order == 1, t[1][k], t[0][k]))  # noqa: E731
                                  for k in range(3)], -1)
    return pick(v), pick(d)


def _tensor(parts):
    """Tensor products over the axes (members k = k0 + 3 k1 + 9 k2)."""
    w = parts[0]
    for p in parts[1:]:
        w = (p[:, :, None] * w[:, None, :]).reshape(w.shape[0], -1)
    return w


def _geometry(phi, dim, N, bc):
    n, h = N + 1, 2.0 / N
    st = [n ** a for a in range(dim)]
    inside = phi < 0
    near = torch.zeros_like(inside)
    for ax in range(dim):
        a, b = inside.narrow(ax, 0, N), inside.narrow(ax, 1, N)
        near.narrow(ax, 1, N).logical_or_(a)
        near.narrow(ax, 0, N).logical_or_(b)
    f = phi.reshape(-1)
    inn = torch.nonzero(inside.reshape(-1))[:, 0]
    gh = torch.nonzero((near & ~inside).reshape(-1))[:, 0]
    pos = torch.full((f.numel(),), -1, dtype=torch.int64, device=DEV)
    pos[inn] = torch.arange(len(inn), device=DEV)
    pos[gh] = len(inn) + torch.arange(len(gh), device=DEV)
    active = pos >= 0
    ii = torch.stack([(gh // st[a]) % n for a in range(dim)], 1)
    grad = torch.stack([(f[gh + st[a]] - f[gh - st[a]]) / (2 * h) for a in range(dim)], 1)
    nv = grad / (grad * grad).sum(1, keepdim=True).sqrt()
    m = torch.where(nv >= 0, 1.0, -1.0).double()
    G = -1.0 + ii.double() * h
    off = [torch.tensor([(k // 3 ** a) % 3 for k in range(3 ** dim)], device=DEV) for a in range(dim)]
    member = gh[:, None] - sum(m[:, a:a + 1].long() * off[a][None, :] * st[a] for a in range(dim))

    def fits(order):
        low = ii - m.long() * order
        return ((low >= 0) & (low <= N)).all(1)

    def at(order, X):
        xi = 1 - m * (G - X) / h
        o = torch.full_like(ii, order)
        w = _tensor([_basis(o[:, a], xi[:, a])[0] for a in range(dim)])
        return (torch.where(w != 0, f[member.clamp(0, f.numel() - 1)], 0.0) * w).sum(1)

    B, border = G.clone(), torch.zeros(len(gh), dtype=torch.int64, device=DEV)
    for order in (2, 1):
        P = G - order * h * nv
        ok = fits(order) & (border == 0) & (at(order, P) < 0)
        lo, hi = torch.zeros_like(B[:, 0]), torch.ones_like(B[:, 0])
        for _ in range(47):
            mid = 0.5 * (lo + hi)
            neg = at(order, P + mid[:, None] * (G - P)) < 0
            lo, hi = torch.where(neg, mid, lo), torch.where(neg, hi, mid)
        B = torch.where(ok[:, None], P + (0.5 * (lo + hi))[:, None] * (G - P), B)
        border = torch.where(ok, order, border)
    th = 1 - m * (G - B) / h
    q = torch.where(fits(2), 2, torch.where(fits(1), 1, 0))
    bv, bd = zip(*[_basis(q, th[:, a]) for a in range(dim)])
    values = f[member.clamp(0, f.numel() - 1)]
    gt = torch.stack([m[:, a] / h * (_tensor([bd[b] if b == a else bv[b] for b in range(dim)]) * values).sum(1)
                      for a in range(dim)], 1)
    size = (gt * gt).sum(1, keepdim=True).sqrt()
    nt = torch.where((q > 0)[:, None] & (size > 0), gt / size, nv)
    # axes by increasing |n|, ties in axis order as a selection by swaps leaves them
    ax = torch.arange(dim, device=DEV).repeat(len(gh), 1)
    for i in range(dim):
        for j in range(i + 1, dim):
            swap = nv.abs().gather(1, ax[:, j:j + 1])[:, 0] < nv.abs().gather(1, ax[:, i:i + 1])[:, 0]
            ai, aj = ax[:, i].clone(), ax[:, j].clone()
            ax[:, i], ax[:, j] = torch.where(swap, aj, ai), torch.where(swap, ai, aj)
    row = torch.zeros(len(gh), 3 ** dim, dtype=torch.float64, device=DEV)
    row[:, 0] = 1.0 / h if bc else 1.0
    found = torch.zeros(len(gh), dtype=torch.bool, device=DEV)
    live = active[member.clamp(0, f.numel() - 1)]
    for nzero in range(dim):
        for top in (2, 1):
            o = torch.full_like(ii, top)
            for z in range(nzero):
                o.scatter_(1, ax[:, z:z + 1], 0)
            v, d = zip(*[_basis(o[:, a], th[:, a]) for a in range(dim)])
            if bc:
                w = sum((nt[:, a] * (m[:, a] / h))[:, None] * _tensor([d[b] if b == a else v[b] for b in range(dim)])
                        for a in range(dim))
            else:
                w = _tensor(v)
            use = ~found & (border >= top) & ((w == 0) | live).all(1)
            row = torch.where(use[:, None], w, row)
            found |= use
    ne = [pos[inn + s * st[a]] for a in range(dim) for s in (1, -1)]
    return dict(ni=len(inn), ng=len(gh), node=torch.cat([inn, gh]), nbr=ne, row=row,
                mem=torch.where(row != 0, pos[member.clamp(0, f.numel() - 1)], 0))


def _cn_step(g, sn, cn, dt, h, s_ext):
    a, d, ms, mc, al, be = MODEL
    ni, nbr, row, mem = g["ni"], g["nbr"], g["row"], g["mem"]
    k = d / (2 * h * h)

    def Ls(s, c):
        ph = al * c + be
        flux = sum((ph[q] + ph[:ni]) * (s[q] - s[:ni]) for q in nbr)
        return -(a / mc) * ph[:ni] * s[:ni] * c[:ni] + k * flux

    def M(s, c):
        ph = al * c + be
        return ph[:ni] * s[:ni] / dt, c / dt + (a / ms) / 2 * ph * s * c

    L0, (M0, _) = Ls(sn, cn), M(sn, cn)
    C0n = cn / dt - (a / ms) / 2 * (al * cn + be) * sn * cn

    def F(s, c):
        Ms, Mc = M(s, c)
        return Ms - M0 - 0.5 * (Ls(s, c) + L0), (row * s[mem]).sum(1) - s_ext, Mc - C0n

    s, c = sn.clone(), cn.clone()
    last = math.inf
    for _ in range(12):
        Fi, Fg, Fc = F(s, c)
        ph = al * c + be
        cs = a / (2 * ms) * ph * c
        cc = 1 / dt + a / (2 * ms) * (al * s * c + ph * s)
        rho = cs / cc
        u, e = (k / 2) * ph, (k / 2) * al * s
        gq = [u[q] + u[:ni] for q in nbr]
        eq = [e[:ni] - e[q] for q in nbr]
        ss = ph[:ni] / dt + a / (2 * mc) * ph[:ni] * c[:ni] + sum(gq)
        sc = al * s[:ni] / dt + a / (2 * mc) * (al * s[:ni] * c[:ni] + ph[:ni] * s[:ni]) + sum(eq)
        diag = ss - sc * rho[:ni]
        off = [x + y * rho[q] for x, y, q in zip(gq, eq, nbr)]
        t = Fc / cc
        b = torch.cat([Fi - sc * t[:ni] - sum(y * t[q] for y, q in zip(eq, nbr)), Fg])
        del gq, eq
        scale = torch.cat([1 / diag, 1 / row.abs().amax(1)])

        def apply(v):
            w = diag * v[:ni]
            for x, q in zip(off, nbr):
                w -= x * v[q]
            return torch.cat([w, (row * v[mem]).sum(1)])

        ds = _gmres(apply, b, scale)
        dc = t - rho * ds
        s, c = s - ds, c - dc
        size = max(float(ds.abs().max() / s.abs().max()), float(dc.abs().max() / c.abs().max()))
        if size < 1e-14 or (size < 1e-12 and size >= 0.5 * last):
            break
        last = size
    return s, c


def _gmres(apply, b, scale, rtol=1e-9, restart=80, rounds=12):
    """Restarted GMRES, rows scaled by `scale`."""
    b = b * scale
    x = torch.zeros_like(b)
    goal = rtol * float(b.norm())
    V = torch.empty(restart + 1, b.numel(), dtype=b.dtype, device=b.device)
    for _ in range(rounds):
        r = b - scale * apply(x)
        beta = float(r.norm())
        if not beta > goal:
            break
        V[0] = r / beta
        H = np.zeros((restart + 1, restart))
        for j in range(restart):
            w = scale * apply(V[j])
            for _twice in range(2):
                p = V[:j + 1] @ w
                w -= p @ V[:j + 1]
                H[:j + 1, j] += p.cpu().numpy()
            H[j + 1, j] = float(w.norm())
            V[j + 1] = w / H[j + 1, j] if H[j + 1, j] > 0 else 0.0
            rhs = np.zeros(j + 2)
            rhs[0] = beta
            y, left, *_ = np.linalg.lstsq(H[:j + 2, :j + 1], rhs, rcond=None)
            if np.linalg.norm(H[:j + 2, :j + 1] @ y - rhs) <= goal or H[j + 1, j] == 0:
                break
        x += torch.from_numpy(y).to(b.device) @ V[:len(y)]
    return x
