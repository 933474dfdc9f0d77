"""Performance cases of the solver: what a reservoir simulator, an ensemble
study and the training of the learned Newton update have the library do,
through the Python binding.

Kinds of case:
  step      one Newton step's linear work: new Jacobian values into the
            matrix, the CPR refreshed, FGMRES(30) to 1e-8
  ensemble  the same for a batch of realisations of uneven grid size
  newton    one implicit time step (assembly, linear work, update) by the
            device Newton method
  spmv      y = alpha A x + beta y, the public matrix-vector product
  conv      one 3x3x3 convolution layer of the network (forward, data
            gradient or weight gradient)

The systems are fully implicit black-oil Jacobians of five-spot waterfloods
(log-normal permeability with spatial correlation, a water front, wells at
fixed bottom-hole pressure), assembled here in FP64 torch.  A step's
right-hand side is A x for a drawn Newton update x, so its solution is known.
"""
from __future__ import annotations

import math

import torch
import torch.nn.functional as F

import paper_1606_00556_gb300 as bo

DEV = "cuda"
PRECISION = {"fp64": bo.BO_PREC_FP64, "fp32": bo.BO_PREC_FP32, "bf16": bo.BO_PREC_BF16}
VALUE_BYTES = {"fp64": 8, "fp32": 4, "bf16": 2}
DX, DY, DZ, DT = 100.0, 100.0, 20.0, 1.0
TOL = 1e-8
FLUID = dict(pref=3000.0, bw0=1.0, cw=3e-6, muw=0.5, bo0=1.25, dbo=6e-5, rs0=0.6, drs=1.5e-4, muo=1.0, bg0=0.9,
             dbg=1.5e-4, mug=0.02, rhow_sc=62.4, rhoo_sc=50.0, rhog_sc=0.06, cr=4e-6, swc=0.1, sorw=0.1, sorg=0.1,
             sgc=0.0, nw=2.0, now=2.0, ng=2.0, nog=2.0, gravity=1.0)
DARCY, BBL = 0.001127, 5.615
BATCH_STREAMS = 8  # pool width of the batched solves


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest system in use: a teaching or test model, or one well's sector; default options
        dict(name="step_tiny_fp64", kind="step", nx=20, ny=20, nz=5, precision="fp64", sigma=0.5),
        # an ordinary sector model with uneven sides
        dict(name="step_mid_fp32", kind="step", nx=62, ny=45, nz=19, precision="fp32", sigma=1.0),
        # the full-field model: 1M cells in mixed precision, the library's main workload ...
        dict(name="step_1m_fp32", kind="step", nx=128, ny=128, nz=64, precision="fp32", sigma=1.5),
        # ... and the same with the default FP64 preconditioner
        dict(name="step_1m_fp64", kind="step", nx=128, ny=128, nz=64, precision="fp64", sigma=1.5),
        # the refined field model, preconditioner stored in BF16 for its memory
        dict(name="step_8m_bf16", kind="step", nx=256, ny=256, nz=128, precision="bf16", sigma=1.5),
        # a batch of geostatistical realisations, grids from 32x32x8 to 96x96x24
        dict(name="ensemble_24_fp32", kind="ensemble", count=24, precision="fp32", sigma=1.0),
        # a whole time step of a simulation run on the device
        dict(name="newton_131k_fp32", kind="newton", nx=64, ny=64, nz=32, precision="fp32", sigma=1.0),
        # products for a caller's own Krylov method or residual check
        dict(name="spmv_1m_fp64", kind="spmv", nx=128, ny=128, nz=64, precision="fp64", beta=0.0),
        dict(name="spmv_ragged_bf16", kind="spmv", nx=190, ny=77, nz=41, precision="bf16", beta=0.5),
        # the network's hidden layer at its training size
        dict(name="conv_forward", kind="conv", op="forward", nx=64, ny=64, nz=32, batch=4, cin=32, cout=32),
        dict(name="conv_backward_data", kind="conv", op="backward_data", nx=64, ny=64, nz=32, batch=4, cin=32,
             cout=32),
        dict(name="conv_backward_weights", kind="conv", op="backward_weights", nx=64, ny=64, nz=32, batch=4, cin=32,
             cout=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _even(n):
    return n + n % 2


def draw(rng):
    kind = rng.choice(["step", "step", "step", "ensemble", "newton", "spmv", "conv", "conv"])
    prec = rng.choice(["fp64", "fp32", "bf16"])
    sigma = round(rng.uniform(0.5, 1.2), 3)
    if kind == "ensemble":
        return dict(kind=kind, count=rng.randint(4, 32), precision=rng.choice(["fp64", "fp32"]), sigma=sigma)
    if kind == "newton":
        return dict(kind=kind, nx=_even(_log_int(rng, 16, 96)), ny=_log_int(rng, 16, 96), nz=_log_int(rng, 4, 32),
                    precision=rng.choice(["fp64", "fp32"]), sigma=min(sigma, 1.0))
    if kind == "conv":
        cin, cout = rng.choice([(16, 32), (32, 32), (32, 32), (32, 16)])
        return dict(kind=kind, op=rng.choice(["forward", "backward_data", "backward_weights"]),
                    nx=_log_int(rng, 12, 80), ny=_log_int(rng, 12, 80), nz=_log_int(rng, 4, 40),
                    batch=rng.randint(1, 8), cin=cin, cout=cout)
    if kind == "spmv":
        return dict(kind=kind, nx=_even(_log_int(rng, 20, 256)), ny=_log_int(rng, 20, 200),
                    nz=_log_int(rng, 5, 64), precision=prec, beta=rng.choice([0.0, 0.5, 1.0]))
    return dict(kind=kind, nx=_even(_log_int(rng, 20, 200)), ny=_log_int(rng, 20, 160), nz=_log_int(rng, 5, 80),
                precision=prec, sigma=sigma)


# ------------------------------------------------------------------ reservoirs
def _gen(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + salt)
    return g


def _noise(shape, corr, g):
    """White noise filtered by a Gaussian of std `corr` cells per axis, zero mean and unit variance."""
    w = torch.randn(shape, generator=g, device=DEV, dtype=torch.float64)
    e = 0.0
    for ax, (n, s) in enumerate(zip(shape, corr)):
        k = torch.fft.fftfreq(n, device=DEV, dtype=torch.float64)
        e = e + ((s * k) ** 2).view([-1 if a == ax else 1 for a in range(3)])
    f = torch.fft.ifftn(torch.fft.fftn(w) * torch.exp(-2.0 * math.pi ** 2 * e)).real
    f = f - f.mean()
    return f / f.std()


class Reservoir:
    """Rock, wells and state of a five-spot waterflood; fields of shape (nz, ny, nx)."""

    def __init__(self, nx, ny, nz, sigma, seed, salt=0):
        g = _gen(seed, salt)
        self.nx, self.ny, self.nz = nx, ny, nz
        self.shape = shape = (nz, ny, nx)
        corr = (max(1.0, nz / 16), max(1.0, ny / 8), max(1.0, nx / 8))
        self.kh = torch.exp(4.0 + sigma * _noise(shape, corr, g))
        self.kv = 0.1 * self.kh
        j = torch.arange(ny, device=DEV, dtype=torch.float64).view(ny, 1)
        i = torch.arange(nx, device=DEV, dtype=torch.float64).view(1, nx)
        # four injectors in the corners, a producer in the middle: (x, y, type, bottom-hole pressure)
        self.wells = [(0, 0, 0, 4000.0), (nx - 1, 0, 0, 4000.0), (0, ny - 1, 0, 4000.0), (nx - 1, ny - 1, 0, 4000.0),
                      (nx // 2, ny // 2, 1, 2000.0)]
        dist = [torch.sqrt((i - a) ** 2 + (j - c) ** 2) for a, c, _, _ in self.wells]
        near = torch.stack(dist[:4]).amin(0) + 3.0 * _noise(shape, (1.0, 3.0, 3.0), g)
        k = torch.arange(nz, device=DEV, dtype=torch.float64)
        self.depth = (8000.0 + (k + 0.5) * DZ).view(nz, 1, 1).expand(shape).contiguous()
        p = 3000.0 + 0.35 * (self.depth - 8000.0)
        sw = 0.1 + 0.375 * (1.0 - torch.tanh((near - 0.3 * min(nx, ny)) / 4.0))
        self.xn = torch.stack([p, sw, torch.full(shape, 0.05, device=DEV, dtype=torch.float64)])
        # a Newton update of a day's step: pressure cones at the wells over a smooth field, saturations at the front
        cone = sum((1.0 if t == 0 else -1.0) * torch.exp(-d / (0.1 * (nx + ny))) for d, (_, _, t, _) in zip(dist, self.wells))
        self.dx = torch.stack([100.0 * cone + 10.0 * _noise(shape, corr, g), 0.01 * _noise(shape, (1.0, 2.0, 2.0), g),
                               0.002 * _noise(shape, (1.0, 2.0, 2.0), g)])

    def perforations(self):
        """(cell (z, y, x), type, bottom-hole pressure, reference depth, well index), all layers of each well."""
        top = float(self.depth[0, 0, 0])
        ro = 0.28 * math.sqrt(DX * DX + DY * DY) / 2.0
        for a, c, t, bhp in self.wells:
            wi = DARCY * 2.0 * math.pi * self.kh[:, c, a] * DZ / math.log(ro / 0.25)
            yield a, c, t, bhp, top, wi


class Dual:
    """A cell quantity and its derivatives by the cell's (p, Sw, Sg): v (...), d (3, ...)."""

    def __init__(self, v, d):
        self.v, self.d = v, d

    def __add__(self, o):
        return Dual(self.v + o.v, self.d + o.d) if isinstance(o, Dual) else Dual(self.v + o, self.d)

    __radd__ = __add__

    def __mul__(self, o):
        return Dual(self.v * o.v, self.d * o.v + self.v * o.d) if isinstance(o, Dual) else Dual(self.v * o, self.d * o)

    __rmul__ = __mul__

    def __neg__(self):
        return self * -1.0

    def __sub__(self, o):
        return self + (-o)

    def __rsub__(self, o):
        return -self + o

    def inv(self):
        r = 1.0 / self.v
        return Dual(r, -self.d * r * r)

    def __truediv__(self, o):
        return self * o.inv() if isinstance(o, Dual) else self * (1.0 / o)

    def pos(self):
        keep = (self.v > 0).to(self.v.dtype)
        return Dual(self.v * keep, self.d * keep)

    def at(self, idx):
        return Dual(self.v[idx], self.d[(slice(None),) + idx])


def _cells(x):
    """Mobilities, gravity gradients, solution ratio and masses of every cell at state x (3, ...)."""
    f = FLUID
    eye = torch.zeros((3, 3) + tuple(x.shape[1:]), device=x.device, dtype=x.dtype)
    for u in range(3):
        eye[u, u] = 1.0
    p, sw, sg = (Dual(x[u], eye[u]) for u in range(3))
    so, dp = 1.0 - sw - sg, p - f["pref"]
    phi = 0.2 * (1.0 + f["cr"] * dp)
    bw, bg = f["bw0"] * (1.0 - f["cw"] * dp), f["bg0"] - f["dbg"] * dp
    boil, rs = f["bo0"] + f["dbo"] * dp, f["rs0"] + f["drs"] * dp
    dw, dg = 1.0 - f["swc"] - f["sorw"], 1.0 - f["swc"] - f["sorg"] - f["sgc"]
    sq = lambda s: s * s  # noqa: E731
    krw, krow = sq(((sw - f["swc"]) / dw).pos()), sq(((1.0 - sw - f["sorw"]) / dw).pos())
    krg, krog = sq(((sg - f["sgc"]) / dg).pos()), sq(((1.0 - sg - (f["swc"] + f["sorg"])) / dg).pos())
    kro = ((krow + krw) * (krog + krg) - krw - krg).pos()
    lw, lo, lg = krw / (f["muw"] * bw), kro / (f["muo"] * boil), krg / (f["mug"] * bg)
    total = (krw / f["muw"] + kro / f["muo"] + krg / f["mug"]) / bw
    gw = (f["rhow_sc"] / 144.0) * bw.inv()
    go = (rs * (1000.0 * f["rhog_sc"]) + f["rhoo_sc"] * BBL) / (BBL * boil) / 144.0
    gg = (1000.0 * f["rhog_sc"] / BBL / 144.0) * bg.inv()
    mass = (phi * so / boil, phi * sw / bw, phi * (sg / bg + rs * so / boil))
    return dict(lw=lw, lo=lo, lg=lg, rslo=rs * lo, total=total, gw=gw, go=go, gg=gg, mass=mass)


def assemble(r, x):
    """Residual (3, nz, ny, nx) at state x with previous level r.xn, and the Jacobian as blocks
    J (7, 3, 3, nz, ny, nx): neighbours -z, -y, -x, the cell, +x, +y, +z."""
    c, prev = _cells(x), _cells(r.xn)
    J = torch.zeros((7, 3, 3) + r.shape, device=x.device, dtype=x.dtype)
    s = DX * DY * DZ / (BBL * DT)
    R = torch.stack([s * (m.v - n.v) for m, n in zip(c["mass"], prev["mass"])])
    for q, m in enumerate(c["mass"]):
        J[3, q] += s * m.d
    for ax, area, h, k in ((2, DY * DZ, DX, r.kh), (1, DX * DZ, DY, r.kh), (0, DX * DY, DZ, r.kv)):
        if r.shape[ax] < 2:
            continue
        lo = tuple(slice(0, -1) if a == ax else slice(None) for a in range(3))
        hi = tuple(slice(1, None) if a == ax else slice(None) for a in range(3))
        T = DARCY * area * 2.0 / (h / k[lo] + h / k[hi])
        dz = r.depth[hi] - r.depth[lo]
        flux = []
        for grav, lams in (("go", ("lo", "rslo")), ("gw", ("lw",)), ("gg", ("lg",))):
            ga, gb = c[grav].at(lo), c[grav].at(hi)
            phi = x[0][hi] - x[0][lo] - 0.5 * (ga.v + gb.v) * dz
            pa, pb = -0.5 * dz * ga.d, -0.5 * dz * gb.d
            pa[0] -= 1.0
            pb[0] += 1.0
            up = (phi > 0).to(x.dtype)  # 1: the upper-index cell is upstream
            for name in lams:
                la, lb = c[name].at(lo), c[name].at(hi)
                lam = up * lb.v + (1.0 - up) * la.v
                flux.append((T * lam * phi, T * (lam * pa + (1.0 - up) * phi * la.d),
                             T * (lam * pb + up * phi * lb.d)))
        oil, gas_in_oil, water, gas = flux
        for q, parts in enumerate(((oil,), (water,), (gas_in_oil, gas))):
            v, da, db = (sum(t) for t in zip(*parts))
            R[(q,) + lo] -= v
            R[(q,) + hi] += v
            J[(3, q, slice(None)) + lo] -= da
            J[(3, q, slice(None)) + hi] += db
            J[(6 - ax, q, slice(None)) + lo] = -db
            J[(ax, q, slice(None)) + hi] = da
    for a, b, kind, bhp, top, wi in r.perforations():
        col = (slice(None), b, a)
        rise = top - r.depth[col]
        p = Dual(x[0][col], torch.zeros((3, r.nz), device=x.device, dtype=x.dtype))
        p.d[0] = 1.0
        head = lambda grav: bhp - p - c[grav].at(col) * rise  # noqa: E731
        if kind == 0:
            rates = {1: wi * (c["total"].at(col) * head("gw"))}
        else:
            o = head("go")
            rates = {0: wi * (c["lo"].at(col) * o), 1: wi * (c["lw"].at(col) * head("gw")),
                     2: wi * (c["rslo"].at(col) * o + c["lg"].at(col) * head("gg"))}
        for q, rate in rates.items():
            R[(q,) + col] -= rate.v
            J[(3, q, slice(None)) + col] -= rate.d
    return R, J


_SHIFT = {0: (0, -1), 1: (1, -1), 2: (2, -1), 4: (2, 1), 5: (1, 1), 6: (0, 1)}


def apply_blocks(J, x):
    """The product of the blocks J with x (3, nz, ny, nx)."""
    y = torch.einsum("rc...,c...->r...", J[3], x)
    for s, (ax, step) in _SHIFT.items():
        mine = tuple((slice(1, None) if step < 0 else slice(0, -1)) if a == ax else slice(None) for a in range(3))
        its = tuple((slice(0, -1) if step < 0 else slice(1, None)) if a == ax else slice(None) for a in range(3))
        all_ = (slice(None),)
        y[all_ + mine] += torch.einsum("rc...,c...->r...", J[(s,) + all_ * 2 + mine], x[all_ + its])
    return y


def flat(x):
    """A field per unknown (3, nz, ny, nx) as the library's interleaved vector."""
    return x.reshape(3, -1).t().contiguous().view(-1)


def _pattern(nx, ny, nz):
    """7-point BSR pattern: existing neighbours (N, 7), rowptr, col."""
    N = nx * ny * nz
    c = torch.arange(N, device=DEV)
    i, j, k = c % nx, (c // nx) % ny, c // (nx * ny)
    ok = torch.stack([k > 0, j > 0, i > 0, c >= 0, i < nx - 1, j < ny - 1, k < nz - 1], 1)
    off = torch.tensor([-nx * ny, -nx, -1, 0, 1, nx, nx * ny], device=DEV)
    col = (c.view(-1, 1) + off)[ok].to(torch.int32)
    rowptr = torch.zeros(N + 1, device=DEV, dtype=torch.int32)
    rowptr[1:] = ok.sum(1).cumsum(0)
    return ok, rowptr, col


def _values(J, ok):
    N = ok.shape[0]
    return J.reshape(63, N).t().reshape(N, 7, 9)[ok].view(-1)


def _count_blocks(nx, ny, nz):
    return nx * ny * nz + 2 * ((nx - 1) * ny * nz + nx * (ny - 1) * nz + nx * ny * (nz - 1))


def _ensemble(case, seed):
    """Grids of the batch: nx, ny 32..96 (nx even), nz 8..24, log-uniform, as the case's own count says;
    rock and states from the seed."""
    import random
    rng = random.Random(7 + case["count"])
    return [(_even(_log_int(rng, 32, 96)), _log_int(rng, 32, 96), _log_int(rng, 8, 24),
             case["sigma"] * rng.uniform(0.5, 1.0), seed, 17 + q) for q in range(case["count"])]


class _System:
    """A matrix with its preconditioner, the next Jacobian's values and right-hand side."""

    def __init__(self, ctx, args, precision):
        r = Reservoir(*args)
        _, J = assemble(r, r.xn)
        self.b = flat(apply_blocks(J, r.dx))
        ok, rowptr, col = _pattern(r.nx, r.ny, r.nz)
        self.val = _values(J, ok)
        self.x = torch.zeros_like(self.b)
        self.A = bo.Matrix.from_bsr(ctx, bo.grid(r.nx, r.ny, r.nz, DX, DY, DZ), rowptr, col, self.val)
        self.A._keep = None
        self.P = bo.Preconditioner(self.A, precision=PRECISION[precision])


# ------------------------------------------------------------------ prepare and run
def prepare(case, seed):
    ctx = bo.Context(0)
    kind = case["kind"]
    if kind == "conv":
        return dict(case, ctx=ctx, **_conv_inputs(case, seed))
    if kind == "ensemble":
        systems = [_System(ctx, a, case["precision"]) for a in _ensemble(case, seed)]
        for s in systems:
            s.P.set_launch_mode(bo.BO_LAUNCH_GRAPH)
        bo.bo_set_batch_streams(BATCH_STREAMS)
        return dict(kind=kind, systems=systems)
    dims = (case["nx"], case["ny"], case["nz"])
    if kind == "spmv":
        r = Reservoir(*dims, 1.0, seed)
        _, J = assemble(r, r.xn)
        ok, rowptr, col = _pattern(*dims)
        A = bo.Matrix.from_bsr(ctx, bo.grid(*dims, DX, DY, DZ), rowptr, col, _values(J, ok))
        A._keep = None
        return dict(kind=kind, A=A, x=flat(r.dx), y0=flat(r.xn), y=flat(r.xn), beta=case["beta"],
                    precision=PRECISION[case["precision"]])
    if kind == "step":
        return dict(kind=kind, system=_System(ctx, dims + (case["sigma"], seed), case["precision"]))
    r = Reservoir(*dims, case["sigma"], seed)
    host = lambda t: t.reshape(-1).cpu().numpy()  # noqa: E731
    cell, ptype, pbhp, pref, pwi = [], [], [], [], []
    for a, b, t, bhp, top, wi in r.perforations():
        for k, w in enumerate(wi.tolist()):
            cell.append(a + r.nx * (b + r.ny * k))
            ptype.append(t)
            pbhp.append(bhp)
            pref.append(top)
            pwi.append(w)
    g = bo.grid(*dims, DX, DY, DZ)
    M = bo.Model(ctx, g, bo.fluid(**FLUID), host(r.kh), host(r.kh), host(r.kv),
                 host(torch.full_like(r.kh, 0.2)), host(r.depth), cell, ptype, pbhp, pref, pwi)
    _, J = assemble(r, r.xn)
    ok, rowptr, col = _pattern(*dims)
    A = bo.Matrix.from_bsr(ctx, g, rowptr, col, _values(J, ok))
    A._keep = None
    P = bo.Preconditioner(A, precision=PRECISION[case["precision"]])
    xn = flat(r.xn)
    return dict(kind=kind, M=M, P=P, xn=xn, x=xn.clone())


def run(state):
    kind = state["kind"]
    if kind == "step":
        s = state["system"]
        s.A.update_values(s.val)
        s.P.update()
        s.P.solve(s.b, s.x, tol=TOL)
        return s.x
    if kind == "ensemble":
        ss = state["systems"]
        bo.bo_update_batched([s.P for s in ss], [s.val for s in ss])
        bo.bo_solve_batched([s.P for s in ss], [s.b for s in ss], [s.x for s in ss], tol=TOL)
        return [s.x for s in ss]
    if kind == "newton":
        state["x"].copy_(state["xn"])
        state["M"].newton(state["P"], state["x"], state["xn"], DT)
        return state["x"]
    if kind == "spmv":
        if state["beta"]:
            state["y"].copy_(state["y0"])
        return state["A"].spmv(state["x"], state["y"], 1.0, state["beta"], state["precision"])
    return _conv_run(state)


# ------------------------------------------------------------------ convolution layers
def _conv_inputs(case, seed):
    g = _gen(seed)
    V, B, ci, co = case["nx"] * case["ny"] * case["nz"], case["batch"], case["cin"], case["cout"]
    n = lambda *s: torch.randn(s, generator=g, device=DEV)  # noqa: E731
    z = lambda *s, dtype=torch.float32: torch.empty(s, device=DEV, dtype=dtype)  # noqa: E731
    bf = torch.bfloat16
    w = (n(27, co, ci) * math.sqrt(2.0 / (27 * ci))).to(bf)
    if case["op"] == "forward":
        s = dict(x=torch.relu(n(B, V, ci)).to(bf), w=w, bias=0.1 * n(co), res=None, yf=None, y=z(B, V, co, dtype=bf))
        if (ci, co) == (32, 32):
            s["res"] = torch.relu(n(B, V, co)).to(bf)
        elif co == 16:
            s["yf"] = z(B, V, 4)
        return s
    dy = 1e-3 * n(B, V, co)
    if case["op"] == "backward_data":
        return dict(dy=dy.to(bf), w=w, dx=z(B, V, ci))
    return dict(x=torch.relu(n(B, V, ci)).to(bf), dy=dy, dw=z(27, co, ci), db=z(co))


def _conv_run(s):
    dims = (s["nx"], s["ny"], s["nz"])
    if s["op"] == "forward":
        bo.bo_conv3d_forward(s["ctx"], dims, s["x"], s["w"], s["bias"], s["res"], s["cout"] == 32, s["y"], s["yf"])
        return [s["y"], s["yf"]] if s["yf"] is not None else s["y"]
    if s["op"] == "backward_data":
        bo.bo_conv3d_backward_data(s["ctx"], dims, s["dy"], s["w"], s["dx"])
        return s["dx"]
    bo.bo_conv3d_backward_weights(s["ctx"], dims, s["x"], s["dy"], s["dw"], s["db"])
    return [s["dw"], s["db"]]


def _taps(x, dims, sign):
    """The 27 shifted views of x [B, V, C] (zero outside the grid): tap t reads voxel v + sign * offset(t)."""
    nx, ny, nz = dims
    B, _, C = x.shape
    p = F.pad(x.double().view(B, nz, ny, nx, C), (0, 0, 1, 1, 1, 1, 1, 1))
    for t in range(27):
        d = [sign * (t // 9 - 1), sign * (t // 3 % 3 - 1), sign * (t % 3 - 1)]
        yield p[:, 1 + d[0]:1 + d[0] + nz, 1 + d[1]:1 + d[1] + ny, 1 + d[2]:1 + d[2] + nx].reshape(-1, C)


def _conv_exact(case, seed):
    s = _conv_inputs(case, seed)
    dims = (case["nx"], case["ny"], case["nz"])
    B, V = case["batch"], dims[0] * dims[1] * dims[2]
    if case["op"] == "forward":
        y = sum(x @ w.double().t() for x, w in zip(_taps(s["x"], dims, 1), s["w"])) + s["bias"].double()
        if s["res"] is not None:
            y = y + s["res"].double().view(-1, case["cout"])
        y = (torch.relu(y) if case["cout"] == 32 else y).view(B, V, -1)
        return [y, y[..., :4].contiguous()] if s["yf"] is not None else y
    if case["op"] == "backward_data":
        return sum(d @ w.double() for d, w in zip(_taps(s["dy"], dims, -1), s["w"])).view(B, V, -1)
    dy = s["dy"].to(torch.bfloat16).double().view(-1, case["cout"])  # the products take dy in bf16
    return [torch.stack([dy.t() @ x for x in _taps(s["x"], dims, 1)]), s["dy"].double().sum((0, 1))]


# ------------------------------------------------------------------ work and exact results
def work(case):
    """Inputs read once and outputs written once; the operations of the product or convolution, and for a
    solve those of one product with the Jacobian (its number of iterations is the method's)."""
    if case["kind"] == "conv":
        v = case["batch"] * case["nx"] * case["ny"] * case["nz"]
        ci, co = case["cin"], case["cout"]
        per = {"forward": 2 * ci + 2 * co * (2 if (ci, co) == (32, 32) else 1) + (16 if co == 16 else 0),
               "backward_data": 2 * co + 4 * ci, "backward_weights": 2 * ci + 4 * co}[case["op"]]
        wb = 27 * ci * co * (4 if case["op"] == "backward_weights" else 2)
        return {"bytes": v * per + wb, "flops": 2 * 27 * ci * co * v}
    if case["kind"] == "ensemble":
        grids = [a[:3] for a in _ensemble(case, 0)]
    else:
        grids = [(case["nx"], case["ny"], case["nz"])]
    nnzb = sum(_count_blocks(*g) for g in grids)
    n = 3 * sum(a * b * c for a, b, c in grids)
    if case["kind"] == "spmv":
        return {"bytes": 9 * VALUE_BYTES[case["precision"]] * nnzb + 8 * n * (3 if case["beta"] else 2),
                "flops": 18 * nnzb}
    if case["kind"] == "newton":
        return {"bytes": 8 * (2 * n + 5 * n // 3), "flops": 18 * nnzb}
    return {"bytes": 72 * nnzb + 16 * n, "flops": 18 * nnzb}


def exact(case, seed):
    if case["kind"] == "conv":
        return _conv_exact(case, seed)
    if case["kind"] == "newton":
        return None  # needs a Newton method of its own
    if case["kind"] == "ensemble":
        return [flat(Reservoir(*a).dx) for a in _ensemble(case, seed)]
    dims = (case["nx"], case["ny"], case["nz"])
    r = Reservoir(*dims, case.get("sigma", 1.0), seed)
    if case["kind"] == "step":
        return flat(r.dx)
    _, J = assemble(r, r.xn)
    y = flat(apply_blocks(J, r.dx))
    return y + case["beta"] * flat(r.xn) if case["beta"] else y
