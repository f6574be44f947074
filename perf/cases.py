"""The work a user has this solver do, as cases that can be measured.

One case is one call chain of the public binding (``paper_2110_13055_gb300.cdi``)
on a synthetic electrode image: the Stokes solve, the explicit transport, the
potential, the implicit transport, the batched studies, and the whole path
from a voxel image to its fields as the serving loop runs it.

    listed()            the cases
    draw(rng)           one more of the same ranges
    prepare(case, seed) what a program holds before the call
    run(state)          the call, and everything it computes
    work(case)          bytes and operations the method itself needs
    exact(case, seed)   the same values from plain torch in 64 bits

Flows and potentials stop at a fixed step count or a tolerance far below the
storage's own rounding, so that the amount of work is the case's alone.
"""
import math

import numpy as np
import torch

from paper_2110_13055_gb300 import cdi

PREC = {"f64": cdi.FP64, "f32": cdi.FP32, "pair": cdi.FP32_SPLIT, "cpair": cdi.FP32_CPAIR}
Z, D = (1, -1), (1.33e-9, 2.03e-9)          # Na+, Cl-
DX, TEMP, EPS_R = 1e-7, 298.15, 78.5
E_CHARGE, K_B, FARADAY, EPS0 = 1.6e-19, 1.38e-23, 96485.0, 8.854e-12
FORCE, TAU = 1e-6, 1.0


def _case(kind, prec, shape, **kw):
    """Sizes are (nx, ny, nz); nz = 1 is a 2D image (D2Q9, 5-point faces)."""
    nx, ny, nz = shape
    two = nz == 1
    c = dict(kind=kind, prec=prec, nx=nx, ny=ny, nz=nz, phi=0.5 if two else 0.45,
             rmin=4.0 if two else 6.0, rmax=16.0 if two else 12.0, mirror=True, walls=False,
             flow_steps=200, steps=0, V=0.8 if two else 1.2, U=1e-4 if two else 1e-6,
             c0=10.0 if two else 20.0, Ka=1e-6, lambda_D=0.0, mode="debye", members=1, dt_mult=1)
    c.update(kw)
    return c


def listed():
    return [
        # The smallest Stokes solve: the 128x64 image in FP64 storage that
        # parity runs and parameter fits use; thousands of short steps.
        dict(_case("flow", "f64", (128, 64, 1), phi=0.6, rmin=6.0, rmax=6.0, flow_steps=2000),
             name="flow-2d-128x64-f64"),
        # The 2D benchmark image: FP32-pair populations, resident in L2.
        dict(_case("flow", "pair", (1024, 512, 1), flow_steps=2000), name="flow-2d-1024x512-pair"),
        # The 3D benchmark image: populations far above L2.
        dict(_case("flow", "f32", (256, 256, 256), flow_steps=600), name="flow-3d-256-f32"),
        # A geometry study: several uneven images solved together.
        dict(_case("flow_batch", "pair", (448, 320, 1), phi=0.55, flow_steps=1000, members=6),
             name="flow-batch-2d-pair"),
        # Explicit transport on the smallest image, FP64.
        dict(_case("transport", "f64", (128, 64, 1), phi=0.6, rmin=6.0, rmax=6.0, steps=2000,
                   V=1.0), name="step-2d-128x64-f64"),
        # Explicit transport of the two benchmark images.
        dict(_case("transport", "pair", (1024, 512, 1), steps=2000), name="step-2d-1024x512-pair"),
        dict(_case("transport", "cpair", (256, 256, 256), steps=600), name="step-3d-256-cpair"),
        # A ragged image whose double layer the grid resolves (large face
        # Peclet numbers), between lateral walls.
        dict(_case("transport", "f32", (101, 87, 93), steps=600, lambda_D=1.5e-7, walls=True,
                   V=0.8, c0=10.0), name="step-3d-101-resolved"),
        # The velocity x potential study on one image (12 members).
        dict(_case("sweep", "pair", (640, 384, 1), phi=0.55, steps=600, members=12),
             name="sweep-2d-640x384-pair"),
        # A potential that needs many iterations: Laplace in 3D.
        dict(_case("potential", "cpair", (128, 128, 128), mode="laplace"),
             name="potential-3d-128-laplace"),
        # Implicit transport far beyond the explicit time step.
        dict(_case("implicit", "cpair", (80, 80, 80), steps=6, dt_mult=40, lambda_D=1.5e-7,
                   V=0.8, c0=10.0), name="implicit-3d-80-cpair"),
        # One request of the serving mix: image in, fields and amounts out.
        dict(_case("whole", "cpair", (96, 96, 96), phi=0.5, flow_steps=1000, steps=1000, V=0.8,
                   U=1e-5, c0=10.0), name="serve-3d-96-cpair"),
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["flow", "flow", "transport", "transport", "transport", "flow_batch", "sweep",
                       "potential", "implicit", "whole"])
    two = kind in ("flow_batch", "sweep") or rng.random() < 0.5
    kw = dict(mirror=rng.random() < 0.75, walls=rng.random() < 0.3,
              phi=round(rng.uniform(0.45, 0.7), 3), V=round(rng.uniform(0.2, 1.2), 3),
              lambda_D=rng.choice([0.0, 0.0, 1.5e-7]))
    if two:
        prec = rng.choice(["f64", "pair", "pair", "f32"])
        top = 200 if prec == "f64" else 1024 if kind in ("flow", "transport") else 512
        shape = (_size(rng, 32, top), _size(rng, 32, top // 2), 1)
        kw.update(rmin=2.0, rmax=round(rng.uniform(3.0, 12.0), 2), U=rng.choice([1e-5, 1e-4, 1e-3]))
    else:
        prec = rng.choice(["f32", "cpair", "cpair"])
        top = 200 if kind in ("flow", "transport") else 96
        shape = tuple(_size(rng, 20, top) for _ in range(3))
        kw.update(rmin=2.0, rmax=round(rng.uniform(3.0, 8.0), 2), U=rng.choice([1e-6, 1e-5, 1e-4]))
    if kind in ("flow", "flow_batch", "whole"):
        kw["flow_steps"] = 100 * rng.randint(2, 6)
    if kind in ("transport", "sweep", "whole"):
        kw["steps"] = rng.randint(100, 600)
    if kind in ("flow_batch", "sweep"):
        kw["members"] = rng.randint(2, 8)
    if kind == "implicit":
        kw.update(steps=rng.randint(2, 6), dt_mult=rng.choice([10, 40]))
    if kind == "potential":
        kw["mode"] = rng.choice(["debye", "laplace", "pb"])
        if kw["mode"] == "pb":
            kw["V"] = round(rng.uniform(0.05, 0.4), 3)
    return _case(kind, prec, shape, **kw)


# ---------------------------------------------------------------------------
# images: a Boolean model of grains (centres uniform, lateral axes periodic),
# stamped on the device
# ---------------------------------------------------------------------------
def _mask(c, seed, nx=None, ny=None):
    nx, ny, nz = nx or c["nx"], ny or c["ny"], c["nz"]
    two = nz == 1
    g = np.random.default_rng(seed)
    r0, r1 = c["rmin"], c["rmax"]
    k = 2 if two else 3
    mean = (r0 ** k if r1 == r0 else (r1 ** (k + 1) - r0 ** (k + 1)) / ((k + 1) * (r1 - r0)))
    mean *= math.pi if two else 4.0 * math.pi / 3.0
    n = max(1, int(round(-math.log(c["phi"]) * nx * ny * nz / mean)))
    dev = "cuda"
    xyz = torch.tensor(g.random((n, 3)) * [nx, ny, nz], device=dev)
    rad = torch.tensor(r0 + (r1 - r0) * g.random(n), device=dev)
    h = int(math.ceil(r1)) + 1
    w = torch.arange(-h, h + 1, device=dev)
    wz = torch.zeros(1, dtype=w.dtype, device=dev) if two else w
    solid = torch.zeros(nz * ny * nx, dtype=torch.uint8, device=dev)
    for s in range(0, n, 512):
        p, r = xyz[s:s + 512], rad[s:s + 512]
        b = torch.floor(p).long()
        x = b[:, 0, None] + w
        y = b[:, 1, None] + w
        z = b[:, 2, None] + wz
        d2 = (((x + 0.5 - p[:, 0, None]) ** 2)[:, None, None, :]
              + ((y + 0.5 - p[:, 1, None]) ** 2)[:, None, :, None])
        if not two:
            d2 = d2 + ((z + 0.5 - p[:, 2, None]) ** 2)[:, :, None, None]
        hit = (d2 <= (r * r)[:, None, None, None]) & ((x >= 0) & (x < nx))[:, None, None, :]
        flat = (((z % nz)[:, :, None, None] * ny + (y % ny)[:, None, :, None]) * nx
                + x.clamp(0, nx - 1)[:, None, None, :]).expand(hit.shape)
        solid[flat[hit]] = 1
    m = solid.reshape(nz, ny, nx)
    m[nz // 2, ny // 2, :] = 0     # one open row: the image always carries flow
    m = m.cpu().numpy()
    return np.ascontiguousarray(m[0] if two else m)


def _batch_sizes(c):
    """The images' sizes, uneven, by the case alone (the grains follow the seed)."""
    g = np.random.default_rng([c["nx"], c["ny"], c["members"]])
    return [(max(16, int(c["nx"] * f)), max(16, int(c["ny"] * h)))
            for f, h in zip(g.uniform(0.6, 1.4, c["members"]), g.uniform(0.6, 1.4, c["members"]))]


def _combos(c):
    vs, us = (0.25, 0.5, 0.75, 1.0), (0.1, 1.0, 10.0)
    return [(c["U"] * u, c["V"] * v) for v in vs for u in us][:c["members"]]


# ---------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------
def _domain(c, m):
    return cdi.Domain(m, dx=DX, precision=PREC[c["prec"]], mirror=c["mirror"],
                      lateral_walls=c["walls"])


def _flow(c, d):
    d.solve_flow(tau=TAU, force=FORCE, tol=0.0, check_every=100, max_steps=c["flow_steps"],
                 U_target=c["U"])


def _potential(c, d):
    d.set_potential(c["V"], T=TEMP, eps_r=EPS_R, c_bulk=c["c0"], lambda_D=c["lambda_D"],
                    mode=c["mode"], tol=1e-13)


def prepare(case, seed):
    c, k = case, case["kind"]
    if k == "flow_batch":
        ms = [_mask(c, seed + 100 * i, nx, ny) for i, (nx, ny) in enumerate(_batch_sizes(c))]
        return {"case": c, "doms": [_domain(c, m) for m in ms]}
    m = _mask(c, seed)
    s = {"case": c, "mask": m}
    if k == "whole":
        return s
    d = s["dom"] = _domain(c, m)
    if k in ("transport", "sweep", "implicit"):
        _flow(c, d)
    if k in ("transport", "implicit"):
        _potential(c, d)
    if k == "implicit":
        s["dt"] = c["dt_mult"] * d.init_transport(Z, D, c0=c["c0"], Ka=c["Ka"])
        d.set_implicit(1e-13, 4000)
    return s


def _advance(c, d, dt=0.0):
    """A transport run from the saturated state: fields and accounts."""
    used = d.init_transport(Z, D, c0=c["c0"], Ka=c["Ka"], dt=dt)
    d.step(c["steps"])
    M, G, I, O = d.mass_balance()
    return {"C": d.C(), "dt": used, "M": M, "Gamma": G, "In": I, "Out": O, "cout": d.outlet()}


def run(state):
    c = state["case"]
    k = c["kind"]
    if k == "flow_batch":
        cdi.flow_batch(state["doms"], tau=TAU, force=FORCE, tol=0.0, check_every=100,
                       max_steps=c["flow_steps"], U_target=c["U"])
        return {"u": [d.u() for d in state["doms"]]}
    if k == "whole":
        with _domain(c, state["mask"]) as d:
            _flow(c, d)
            _potential(c, d)
            out = _advance(c, d)
            out.update(u=d.u(), psi=d.psi())
        return out
    d = state["dom"]
    if k == "flow":
        _flow(c, d)
        return {"u": d.u()}
    if k == "potential":
        _potential(c, d)
        return {"psi": d.psi()}
    if k == "sweep":
        gam, cout, dt = d.sweep(_combos(c), z=Z, D=D, c0=c["c0"], Ka=c["Ka"], n_steps=c["steps"],
                                T=TEMP, eps_r=EPS_R, lambda_D=c["lambda_D"], mode=c["mode"],
                                tol=1e-13)
        return {"Gamma": gam, "cout": cout, "dt": dt}
    return _advance(c, d, state.get("dt", 0.0))


def work(case):
    """Per lattice step a pore site's populations are read and written once;
    per transport step a cell's concentrations, with its velocity, potential
    and a mask byte read; per solver iteration the vectors of the method."""
    c = case
    dim = 2 if c["nz"] == 1 else 3
    q = 9 if dim == 2 else 19
    wide = 8 if c["prec"] == "f64" else 4
    pop = 8 if c["prec"] in ("f64", "pair") else 4
    con = 8 if c["prec"] in ("f64", "pair", "cpair") else 4
    cells = c["nx"] * c["ny"] * c["nz"]
    pores = cells * c["phi"]
    sites = pores * (2 if c["mirror"] else 1)
    flow_b, flow_f = sites * q * pop * 2, sites * (q * 12)
    step_b = pores * (2 * 2 * con + dim * wide + wide + 1)
    step_f = pores * (2 * dim * 2 * 12)
    k, nf, ns = c["kind"], c["flow_steps"], c["steps"]
    if k == "flow":
        b, f = nf * flow_b + dim * cells * 8, nf * flow_f
    elif k == "flow_batch":
        b, f = c["members"] * (nf * flow_b + dim * cells * 8), c["members"] * nf * flow_f
    elif k == "transport":
        b, f = ns * step_b + 2 * cells * 8, ns * step_f
    elif k == "sweep":
        b, f = c["members"] * ns * step_b, c["members"] * ns * step_f
    elif k == "potential":
        it = 3 * max(c["nx"], c["ny"], c["nz"]) if c["mode"] == "laplace" and not c["lambda_D"] else 20
        b, f = pores * 8 * 9 * it + cells * 8, pores * (4 * dim + 12) * it
    elif k == "implicit":
        it = 15 * 2 * ns
        b, f = it * pores * 8 * (2 * (2 * dim + 1) + 12), it * pores * (8 * dim + 20)
    else:
        b = nf * flow_b + ns * step_b + cells * (8 * (dim + 3) + 1)
        f = nf * flow_f + ns * step_f
    return {"bytes": float(b), "flops": float(f)}


# ---------------------------------------------------------------------------
# the same in plain torch, 64 bits: pore cells as a list, neighbours as index
# tables
# ---------------------------------------------------------------------------
def _lattice(dim):
    if dim == 2:
        e = [(0, 0, 0)] + [(x, y, 0) for x in (-1, 0, 1) for y in (-1, 0, 1) if x or y]
        w = {0: 4 / 9, 1: 1 / 9, 2: 1 / 36}
    else:
        e = [(0, 0, 0)] + [(x, y, z) for x in (-1, 0, 1) for y in (-1, 0, 1) for z in (-1, 0, 1)
                           if 0 < abs(x) + abs(y) + abs(z) < 3]
        w = {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}
    return e, [w[sum(abs(v) for v in i)] for i in e], [e.index(tuple(-v for v in i)) for i in e]


def _ref_flow(c, m):
    """Velocity of every pore cell of the image, (dim, cells), in m/s."""
    S = torch.tensor(np.atleast_3d(m) if m.ndim == 3 else m[None], device="cuda") != 0
    dim, nx = m.ndim, m.shape[-1]
    F = torch.cat([S, S.flip(2)], 2) if c["mirror"] else S
    pore = torch.nonzero(~F.reshape(-1)).reshape(-1)
    n = pore.numel()
    rank = torch.full((F.numel(),), -1, dtype=torch.int64, device="cuda")
    rank[pore] = torch.arange(n, device="cuda")
    rank = rank.reshape(F.shape)
    e, w, opp = _lattice(dim)
    own = torch.arange(n, device="cuda")
    src = []
    for i, (ex, ey, ez) in enumerate(e):
        up = torch.roll(rank, (ez, ey, ex), (0, 1, 2)).clone()   # rank of the site x - e_i
        if c["walls"]:
            for ax, s in ((1, ey), (0, ez)):
                if s:
                    up.select(ax, 0 if s > 0 else -1).fill_(-1)
        up = up.reshape(-1)[pore]
        src.append(torch.where(up >= 0, i * n + up, opp[i] * n + own))
    g = torch.zeros((len(e), n), dtype=torch.float64, device="cuda")
    post = torch.empty_like(g)
    om, fsrc = 1.0 / TAU, (1.0 - 0.5 / TAU) * 3.0 * FORCE

    def momentum():
        j = [torch.zeros(n, dtype=torch.float64, device="cuda") for _ in range(3)]
        j[0] += 0.5 * FORCE
        for i, v in enumerate(e):
            for a in range(dim):
                if v[a]:
                    j[a].add_(g[i], alpha=v[a])
        return j

    for _ in range(c["flow_steps"]):
        rho, j = g.sum(0), momentum()
        for i, v in enumerate(e):
            t = rho.clone()
            for a in range(dim):
                if v[a]:
                    t.add_(j[a], alpha=3.0 * v[a])
            torch.mul(g[i], 1.0 - om, out=post[i])
            post[i].add_(t, alpha=om * w[i]).add_(w[i] * v[0] * fsrc)
        flat = post.reshape(-1)
        for i in range(len(e)):
            torch.index_select(flat, 0, src[i], out=g[i])
    j = momentum()
    u = torch.zeros((dim,) + tuple(F.shape), dtype=torch.float64, device="cuda")
    for a in range(dim):
        u[a].reshape(-1)[pore] = j[a]
    u = u[..., :nx].contiguous()
    mean = u[0].sum() / int((~S).sum())
    return u.reshape(dim, -1) * (c["U"] / float(mean))


class _Cells:
    """Pore cells of the image and what lies across their faces."""

    def __init__(self, c, m):
        S = torch.tensor(m if m.ndim == 3 else m[None], device="cuda") != 0
        self.dim, self.shape, self.N = m.ndim, m.shape, m.size
        self.cell = torch.nonzero(~S.reshape(-1)).reshape(-1)
        n = self.n = self.cell.numel()
        rank = torch.full((S.numel(),), -1, dtype=torch.int64, device="cuda")
        rank[self.cell] = torch.arange(n, device="cuda")
        rank = rank.reshape(S.shape)
        own = torch.arange(n, device="cuda")
        self.nb, self.kind = [], []      # kind: 0 pore, 1 solid, 2 inlet, 3 outlet, 4 wall
        for f in range(2 * self.dim):
            ax, s = 2 - f // 2, -1 if f & 1 else 1
            q = torch.roll(rank, -s, ax).clone()
            q[q < 0] = -2
            edge = q.select(ax, -1 if s > 0 else 0)
            if ax == 2:
                edge.fill_(-4 if s > 0 else -3)
            elif c["walls"]:
                edge.fill_(-5)
            q = q.reshape(-1)[self.cell]
            self.kind.append(torch.where(q >= 0, torch.zeros_like(q), -q - 1))
            self.nb.append(torch.where(q >= 0, q, own))
        x = self.cell % m.shape[-1]
        self.outlet = x == m.shape[-1] - 1

    def full(self, v):
        o = torch.zeros(self.N, dtype=torch.float64, device="cuda")
        o[self.cell] = v
        return o.reshape(self.shape).cpu().numpy()


def _solve(apply, b, x, tol=1e-15, most=20000):
    """Jacobi-preconditioned BiCGStab (apply carries the preconditioner)."""
    r = b - apply(x)
    r0, p = r.clone(), r.clone()
    bb, rho, best = float(b.norm()), r.dot(r), (math.inf, x)
    for it in range(most):
        v = apply(p)
        al = rho / r0.dot(v)
        s = r - al * v
        t = apply(s)
        tt = t.dot(t)
        om = t.dot(s) / torch.where(tt == 0, torch.ones_like(tt), tt)
        x = x + al * p + om * s
        r = s - om * t
        new = r0.dot(r)
        rel = float(r.norm()) / bb
        if rel < best[0]:
            best = (rel, x)
        if rel < tol or not math.isfinite(rel) or float(new) == 0.0:
            break
        p = r + (new / rho) * (al / om) * (p - om * v)
        rho = new
    return best[1]


def _ref_psi(c, G, V=None):
    V = c["V"] if V is None else V
    vt = K_B * TEMP / E_CHARGE
    lam = c["lambda_D"] or math.sqrt(EPS_R * EPS0 * K_B * TEMP / (2.0 * c["c0"] * E_CHARGE * FARADAY))
    k2 = 0.0 if c["mode"] == "laplace" else (DX / lam) ** 2
    base = torch.zeros(G.n, dtype=torch.float64, device="cuda")
    b = torch.zeros_like(base)
    for kd in G.kind:
        base += ((kd == 0) | (kd == 2)).double() + 2.0 * (kd == 1).double()
        b += -2.0 * V * (kd == 1).double()
    open_ = [(kd == 0).double() for kd in G.kind]

    def lin(diag, rhs, x0):
        def apply(y):                    # A (y / diag)
            y = y / diag
            return diag * y - sum(o * y[q] for o, q in zip(open_, G.nb))
        for _ in range(2):               # restarted once: to rounding
            x0 = _solve(apply, rhs, x0 * diag) / diag
        return x0
    x = torch.zeros_like(base)
    if c["mode"] != "pb":
        return lin(base + k2, b, x)
    for _ in range(100):
        sh, ch = torch.sinh(x / vt), torch.cosh(x / vt)
        y = lin(base + k2 * ch, b + k2 * (x * ch - vt * sh), x)
        done = float((y - x).norm()) < 1e-14 * float(y.norm())
        x = y
        if done:
            break
    return x


def _bern(x):
    safe = torch.where(x == 0, torch.ones_like(x), x)
    small = x.abs() < 1e-3
    return torch.where(small, 1 - x / 2 + x * x / 12 - x ** 4 / 720, safe / torch.expm1(safe))


class _Operator:
    """Face coefficients of one species: J sums, accounts and the rate."""

    def __init__(self, c, G, u, psi, k):
        vt = K_B * TEMP / E_CHARGE
        Dk, ke = D[k], c["Ka"] / (1.0 + c["Ka"] * DX / (2.0 * D[k]))
        self.diag = torch.zeros(G.n, dtype=torch.float64, device="cuda")   # of sum_f J
        self.off, self.G, self.c0 = [], G, c["c0"]
        self.gam = torch.zeros_like(self.diag)
        rate = torch.zeros_like(self.diag)
        for f, (kd, q) in enumerate(zip(G.kind, G.nb)):
            s = -1.0 if f & 1 else 1.0
            ua = u[f // 2]
            phn = torch.where(kd == 2, torch.zeros_like(psi), psi[q]) / vt
            P = 0.5 * s * (ua + ua[q]) * DX / Dk - Z[k] * (phn - psi / vt)
            open_ = (kd == 0) | (kd == 2) | (kd == 3)
            bm = torch.where(open_, Dk / DX * _bern(-P), torch.zeros_like(P))
            bp = torch.where(open_, Dk / DX * _bern(P), torch.zeros_like(P))
            solid = (kd == 1).double() * ke
            self.gam += solid
            rate += bm + solid
            if f == 0:
                self.aout = torch.where(kd == 3, bm - bp, torch.zeros_like(P))
            if f == 1:
                self.ain, self.bin = (torch.where(kd == 2, v, torch.zeros_like(P)) for v in (bm, bp))
            self.diag += bm + solid - torch.where(kd == 3, bp, torch.zeros_like(P))
            self.off.append(torch.where(kd == 0, bp, torch.zeros_like(P)))
        self.src = self.bin * c["c0"]
        self.rate = float(rate.max()) / DX

    def flux(self, C):                   # sum_f J
        J = self.diag * C - self.src
        for o, q in zip(self.off, self.G.nb):
            J -= o * C[q]
        return J

    def accounts(self, C):
        return (self.gam * C).sum(), (self.src - self.ain * C).sum(), (self.aout * C).sum()


def _ref_run(c, G, u, psi, implicit=False):
    ops = [_Operator(c, G, u, psi, k) for k in range(len(Z))]
    dt = 0.9 / max(o.rate for o in ops) * c["dt_mult"]
    area, vol = DX ** (G.dim - 1), DX ** G.dim
    Cs, acc = [], []
    for o in ops:
        C = torch.full((G.n,), c["c0"], dtype=torch.float64, device="cuda")
        tot = [torch.zeros((), dtype=torch.float64, device="cuda") for _ in range(3)]
        K = 1.0 + dt / DX * o.diag
        for _ in range(c["steps"]):
            if implicit:
                def apply(y):
                    y = y / K
                    return y + dt / DX * (o.flux(y) + o.src)
                C = _solve(apply, C + dt / DX * o.src, C * K) / K
                new = C
            else:
                new = C - dt / DX * o.flux(C)
            for t, v in zip(tot, o.accounts(C)):
                t += v * (dt * area)
            C = new
        Cs.append(C)
        acc.append([float(t) for t in tot])
    ux = u[0][G.outlet]
    cout = np.array([float((ux * C[G.outlet]).sum() / ux.sum()) for C in Cs])
    a = np.array(acc)
    return {"C": np.stack([G.full(C) for C in Cs]), "dt": dt, "M": np.array([float(C.sum()) * vol for C in Cs]),
            "Gamma": a[:, 0].copy(), "In": a[:, 1].copy(), "Out": a[:, 2].copy(), "cout": cout}


def exact(case, seed):
    c, k = case, case["kind"]
    if k == "flow_batch":
        out = []
        for i, (nx, ny) in enumerate(_batch_sizes(c)):
            m = _mask(c, seed + 100 * i, nx, ny)
            out.append(_ref_flow(c, m).reshape((m.ndim,) + m.shape).cpu().numpy())
        return {"u": out}
    m = _mask(c, seed)
    if k == "flow":
        return {"u": _ref_flow(c, m).reshape((m.ndim,) + m.shape).cpu().numpy()}
    G = _Cells(c, m)
    if k == "potential":
        return {"psi": G.full(_ref_psi(c, G))}
    ua = _ref_flow(c, m)
    u = ua[:, G.cell]
    if k == "sweep":
        rows = []
        for U, V in _combos(c):
            rows.append(_ref_run(c, G, u * (U / c["U"]), _ref_psi(c, G, V)))
        return {"Gamma": np.stack([r["Gamma"] for r in rows]),
                "cout": np.stack([r["cout"] for r in rows]),
                "dt": np.array([r["dt"] for r in rows])}
    psi = _ref_psi(c, G)
    out = _ref_run(c, G, u, psi, implicit=k == "implicit")
    if k == "whole":
        out.update(u=ua.reshape((m.ndim,) + m.shape).cpu().numpy(), psi=G.full(psi))
    return out
