"""What is timed: the work users have this library do, through its public entry points.

A case is a dict of plain values.  Kinds:
  grid   a state comes in, `steps` time steps are taken, the new state goes out
         (Grid.set_state / run / get_state; loop=True: the caller's own loop of
         cfl_dt and step instead of run);
  tubes  the same for a batch of independent 1D tubes (Batch);
  grad   the allocation-free gradient of the star-pressure network.

`prepare` makes the inputs on the GPU from the seed and the handle that a
program keeps (it has taken one step, so its launch shape is tuned); `run` is
one pass; `exact` is the same computation in plain 64-bit torch.
"""
import math

import numpy as np
import torch

from paper_2503_04428_gb300 import hydro as H

DEV = "cuda:0"
F64 = torch.float64
HLL, HLLC, EXACT = 0, 1, 2
MINMOD, VANLEER, VANALBADA = 1, 2, 3
PERIODIC, TRANSMISSIVE, REFLECTIVE = 0, 1, 2


def listed():
    g = dict(kind="grid")
    t = dict(kind="tubes", lo=256, hi=8192, perturb=0.0, mlp=False, cfl=0.8)
    return [
        # the smallest calls: a small 2D run in FP64 whose caller asks for dt and steps
        dict(g, name="kh2d_64x128_f64_loop", setup="kh", nx=64, ny=128, precision=64, riemann=HLLC,
             limiter=MINMOD, steps=10, loop=True, totals=False),
        # a shock tube run to its end: many short steps of few cells, FP64
        dict(g, name="sod_1000_f64", setup="sod", nx=1000, precision=64, riemann=HLLC, limiter=MINMOD,
             steps=550, loop=False, totals=False),
        # 2D Rayleigh-Taylor with gravity and a passive scalar, FP32 bulk
        dict(g, name="rt2d_512x1536_f32", setup="rt", nx=512, ny=1536, precision=32, riemann=HLLC,
             limiter=MINMOD, steps=20, loop=False, totals=False),
        # a periodic 3D flow on an odd, ragged grid, exact solver and another limiter
        dict(g, name="smooth_101x67x53_f32", setup="smooth", nx=101, ny=67, nz=53, precision=32,
             riemann=EXACT, limiter=VANLEER, steps=10, loop=False, totals=False),
        # 3D blast wave in the FP32 bulk form with its conserved totals kept
        dict(g, name="sedov3d_256_f32", setup="sedov", nx=256, ny=256, nz=256, precision=32, riemann=HLL,
             limiter=MINMOD, steps=10, loop=False, totals=True),
        # the same blast in FP64
        dict(g, name="sedov3d_128_f64", setup="sedov", nx=128, ny=128, nz=128, precision=64, riemann=HLL,
             limiter=MINMOD, steps=3, loop=False, totals=False),
        # spherical wedge of a supernova-like envelope: 3 scalars, monopole gravity
        dict(g, name="wedge_1024x128x128_f32", setup="wedge", nx=1024, ny=128, nz=128, precision=32,
             riemann=HLLC, limiter=MINMOD, steps=5, loop=False, totals=False, rad=False),
        # the same with gas and radiation in equilibrium (a temperature solve per state)
        dict(g, name="wedge_rad_512x96x96_f32", setup="wedge", nx=512, ny=96, nz=96, precision=32,
             riemann=HLLC, limiter=MINMOD, steps=5, loop=False, totals=False, rad=True),
        # thousands of ragged shock tubes, exact solver with the learned guess, FP32
        dict(t, name="tubes_4096_f32_mlp", ntubes=4096, precision=32, steps=100, mlp=True),
        # tubes whose every cell is disturbed: each face runs the Newton iteration
        dict(t, name="tubes_1024_f32_dense", ntubes=1024, precision=32, steps=10, perturb=0.01),
        # the plain FP64 form of the batch
        dict(t, name="tubes_512_f64", ntubes=512, precision=64, steps=20),
        # one gradient of the guess network on a caller's training batch
        dict(kind="grad", name="mlp_grad_16384", n=16384),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sod", "kh", "rt", "smooth", "sedov", "wedge", "tubes", "tubes", "grad"])
    limiter = rng.choice([MINMOD, MINMOD, VANLEER, VANALBADA])
    g = dict(kind="grid", setup=kind, precision=rng.choice([32, 64]), riemann=rng.choice([HLL, HLLC, HLLC, EXACT]),
             limiter=limiter, loop=rng.random() < 0.25, totals=rng.random() < 0.25)
    if kind == "sod":
        return dict(g, nx=_log_int(rng, 100, 20000), steps=rng.randint(20, 200))
    if kind in ("kh", "rt"):
        return dict(g, nx=_log_int(rng, 32, 700), ny=_log_int(rng, 48, 1100), steps=rng.randint(5, 20))
    if kind in ("smooth", "sedov"):
        if kind == "sedov":  # (a blast into a cold medium: the approximate solvers)
            g["riemann"] = rng.choice([HLL, HLLC])
        hi = 80 if g["precision"] == 64 else 256
        n = [_log_int(rng, 20, hi) for _ in range(3)]
        steps = 3 if g["precision"] == 64 else rng.randint(3, 8)
        return dict(g, nx=n[0], ny=n[1], nz=n[2], steps=steps)
    if kind == "wedge":
        f32 = g["precision"] == 32
        rad = f32 and rng.random() < 0.4
        g["riemann"] = rng.choice([HLL, HLLC])
        return dict(g, nx=_log_int(rng, 64, 1024 if f32 else 256), ny=_log_int(rng, 24, 128 if f32 else 64),
                    nz=_log_int(rng, 24, 96 if f32 else 48), steps=3, rad=rad)
    if kind == "tubes":
        f32 = rng.random() < 0.7
        dense = rng.random() < 0.4
        lo = _log_int(rng, 32, 512)
        return dict(kind="tubes", ntubes=_log_int(rng, 16, 4096 if f32 and not dense else 512), lo=lo,
                    hi=lo + _log_int(rng, 16, 7000), precision=32 if f32 else 64,
                    steps=rng.randint(3, 50 if f32 and not dense else 10), perturb=0.01 if dense else 0.0,
                    mlp=f32 and rng.random() < 0.5, cfl=rng.choice([0.4, 0.8]))
    return dict(kind="grad", n=_log_int(rng, 64, 16384))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _rand(gen, *shape):
    return 2.0 * torch.rand(*shape, generator=gen, device=DEV, dtype=F64) - 1.0


def _cons(gamma, rho, vel, p, scalars=()):
    e = p / (gamma - 1.0) + 0.5 * rho * sum(v * v for v in vel)
    return torch.stack([rho] + [rho * v for v in vel] + [e] + [rho * f for f in scalars])


def _setup(c, seed):
    """Faces, boundaries, constants and the initial conserved state (FP64) of a grid case."""
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    lin = lambda a, b, n: torch.linspace(a, b, n + 1, dtype=F64)  # noqa: E731
    mid = lambda f: (0.5 * (f[1:] + f[:-1])).to(DEV)  # noqa: E731
    s, nx = c["setup"], c["nx"]
    d = dict(coords=0, gamma=1.4, ns=0, cfl=0.4, grav=None, rad=None)
    if s == "sod":  # (1,0,1) | (0.125,0,0.1), each within 10 %
        f = [lin(0, 1, nx)]
        j = 1.0 + 0.1 * _rand(gen, 4)
        left = mid(f[0]) < 0.5
        rho = torch.where(left, j[0], 0.125 * j[1])
        p = torch.where(left, j[2], 0.1 * j[3])
        d.update(faces=f, bc=[(TRANSMISSIVE,) * 2], cfl=0.8, U=_cons(1.4, rho, [0 * rho], p))
    elif s == "kh":  # shear layers with a seeded perturbation and a scalar
        f = [lin(0, 1, nx), lin(0, 2, c["ny"])]
        z, x = torch.meshgrid(mid(f[1]), mid(f[0]), indexing="ij")
        prof = torch.tanh((z - 0.5) / 0.05) - torch.tanh((z - 1.5) / 0.05)
        uz = 0.01 * torch.sin(2 * math.pi * x) * (torch.exp(-(z - 0.5) ** 2 / 0.04) + torch.exp(-(z - 1.5) ** 2 / 0.04))
        uz = uz + 0.001 * _rand(gen, *z.shape)
        d.update(faces=f, bc=[(PERIODIC,) * 2] * 2, gamma=5 / 3, ns=1,
                 U=_cons(5 / 3, 1 + 0.5 * prof, [prof, uz], torch.full_like(x, 10.0), [0.5 * prof]))
    elif s == "rt":  # heavy over light, random vertical velocities at the interface
        f = [lin(0, 0.5, nx), lin(0, 1.5, c["ny"])]
        y, x = torch.meshgrid(mid(f[1]), mid(f[0]), indexing="ij")
        heavy = y >= 0.75
        rho = torch.where(heavy, 2.0, 1.0).to(F64)
        vy = torch.where((y - 0.75).abs() < 6.0 / c["ny"], 0.01 * _rand(gen, *y.shape), 0.0)
        d.update(faces=f, bc=[(PERIODIC,) * 2, (REFLECTIVE,) * 2], ns=1, grav=(0.0, -0.1, 0.0),
                 U=_cons(1.4, rho, [0 * x, vy], 2.5 - 0.1 * rho * (y - 0.75), [heavy.to(F64)]))
    elif s == "smooth":  # a periodic wave field with noise, mildly non-uniform cells
        n = [nx, c["ny"], c["nz"]]
        f = []
        for m in n:
            q = torch.arange(m + 1, dtype=F64) / m
            f.append(q + 0.02 * torch.sin(2 * math.pi * q) / (2 * math.pi))
        k, j, i = torch.meshgrid(*[torch.arange(m, device=DEV, dtype=F64) / m for m in reversed(n)], indexing="ij")
        ph = 2 * math.pi * (k + 2 * j + 3 * i)
        rho = 1 + 0.2 * torch.sin(ph) + 0.1 * _rand(gen, *ph.shape)
        vel = [0.2 * torch.cos(ph + a) + 0.1 * _rand(gen, *ph.shape) for a in range(3)]
        p = 1 + 0.2 * torch.cos(2 * ph) + 0.1 * _rand(gen, *ph.shape)
        d.update(faces=f, bc=[(PERIODIC,) * 2] * 3, U=_cons(1.4, rho, vel, p))
    elif s == "sedov":  # a blast in the central cells of a medium with 1 % density noise
        n = [nx, c["ny"], c["nz"]]
        f = [lin(-1, 1, m) for m in n]
        rho = 1 + 0.01 * _rand(gen, n[2], n[1], n[0])
        zero = torch.zeros_like(rho)
        U = _cons(1.4, rho, [zero] * 3, torch.full_like(rho, 1e-5))
        vol = 8.0 / (n[0] * n[1] * n[2])
        b = [slice(m // 2 - 1, m // 2 + 1) for m in n]
        U[4, b[2], b[1], b[0]] += 1.0 / (8.0 * vol)
        d.update(faces=f, bc=[(TRANSMISSIVE,) * 2] * 3, U=U)
    else:  # wedge: rho ~ r^-2, H/He/O shells, an inner energy injection, 0.5 % density noise
        gamma, rho0 = 5 / 3, 1 / (4 * math.pi * 999.0)
        f = [10.0 ** (3.0 * torch.arange(nx + 1, dtype=F64) / nx),
             lin(math.pi / 2 - math.pi / 12, math.pi / 2 + math.pi / 12, c["ny"]), lin(0, math.pi / 6, c["nz"])]
        rc = mid(f[0])
        dm = 4 * math.pi * rho0 * (f[0][1:] - f[0][:-1]).to(DEV)
        Mi = 1.0 + torch.cumsum(dm, 0) - 0.5 * dm
        e_in = 1e-2 * float((Mi * dm / rc).sum()) / (4 / 3 * math.pi * float(f[0][8] ** 3 - f[0][0] ** 3))
        r = rc.expand(c["nz"], c["ny"], nx)
        rho = rho0 / r ** 2 * (1 + 0.005 * _rand(gen, *r.shape))
        zero = torch.zeros_like(rho)
        shells = [r >= 100, (r >= 10) & (r < 100), r < 10]
        U = _cons(gamma, rho, [zero] * 3, 1e-4 * rho / r, [q.to(F64) for q in shells])
        U[4, :, :, :8] += e_in
        d.update(faces=f, bc=[(REFLECTIVE, TRANSMISSIVE), (REFLECTIVE,) * 2, (REFLECTIVE,) * 2], coords=1, gamma=gamma,
                 ns=3, grav="mono", rad=(1.0, 2.5e8) if c["rad"] else None, U=U)
    d["dim"] = len(d["faces"])
    d["U"] = d["U"].reshape(d["U"].shape[0], *[c.get(k, 1) if i < d["dim"] else 1
                                               for i, k in ((2, "nz"), (1, "ny"), (0, "nx"))])
    return d


def _dtype(c):
    return F64 if c["precision"] == 64 else torch.float32


def _lengths(c):
    """Cells per tube: part of the plan, the same for every seed."""
    gen = torch.Generator().manual_seed(1000003 * c["ntubes"] + c["hi"])
    return torch.randint(c["lo"], c["hi"] + 1, (c["ntubes"],), generator=gen)


def _tube_states(gen, n):
    """Left and right (rho, u, p): ratios over 6 and 8 decades, a velocity jump in [-2, 2]."""
    rr, rp, du = 10.0 ** (3.0 * _rand(gen, n)), 10.0 ** (4.0 * _rand(gen, n)), 2.0 * _rand(gen, n)
    return (torch.stack([rr.sqrt(), -0.5 * du, rp.sqrt()]), torch.stack([rr.rsqrt(), 0.5 * du, rp.rsqrt()]))


def _tubes(c, seed):
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    n = _lengths(c).to(DEV)
    WL, WR = _tube_states(gen, c["ntubes"])
    first = torch.cumsum(n, 0) - n
    tube = torch.repeat_interleave(torch.arange(c["ntubes"], device=DEV), n)
    x = (torch.arange(tube.numel(), device=DEV) - first[tube] + 0.5) / n[tube]
    W = torch.where(x < 0.5, WL[:, tube], WR[:, tube])
    if c["perturb"]:
        W[0] *= 1 + c["perturb"] * _rand(gen, tube.numel())
        W[2] *= 1 + c["perturb"] * _rand(gen, tube.numel())
    return _cons(5 / 3, W[0], [W[1]], W[2])


def _trained(b, seed):
    """A network as a program has it: trained for a moment on faces of the tubes' distribution."""
    gen = torch.Generator(device=DEV).manual_seed(12345)
    WL, WR = _tube_states(gen, 8192)
    t = 0.5 + 0.5 * _rand(gen, 8192)
    WL, WR = WL.T.cpu().numpy(), (WL + t * (WR - WL)).T.cpu().numpy()
    ps, _, _ = H.hydro_exact_solve(WL, WR, 5 / 3)
    ok = ps > 0
    faces = torch.cat([torch.from_numpy(WL.copy()), torch.from_numpy(WR.copy())], 1).numpy()[ok]
    b.mlp_train(faces, np.log(ps[ok]), epochs=5, batch=512, lr=3e-3, seed=4)
    b.mlp_set(b.mlp_get(), True)


def _grad_inputs(c, seed):
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    WL, WR = _tube_states(gen, c["n"])
    rr, pr = (WL[0] * WR[0]).sqrt(), (WL[2] * WR[2]).sqrt()
    cr = (5 / 3 * pr / rr).sqrt()
    x = torch.stack([(WL[0] / rr).log(), (WR[0] / rr).log(), (WL[2] / pr).log(), (WR[2] / pr).log(),
                     WL[1] / cr, WR[1] / cr], 1)
    y = 0.5 * x[:, 4] - 0.5 * x[:, 5] + 0.3 * _rand(gen, c["n"])
    w = torch.zeros(H.HYDRO_MLP_NPARAM, device=DEV, dtype=F64)
    at = 0
    for rows, cols in ((64, 6), (64, 64), (1, 64)):
        w[at:at + rows * cols] = math.sqrt(6 / (rows + cols)) * _rand(gen, rows * cols)
        at += rows * cols
        w[at:at + rows] = 0.05 * _rand(gen, rows)
        at += rows
    return [t.to(torch.float32).contiguous() for t in (w, x, y)]


def prepare(case, seed):
    c = case
    if c["kind"] == "grad":
        w, x, y = _grad_inputs(c, seed)
        return dict(case=c, w=w, x=x, y=y, grad=torch.empty(H.HYDRO_MLP_NPARAM, device=DEV, dtype=F64),
                    loss=torch.empty(1, device=DEV, dtype=F64))
    if c["kind"] == "tubes":
        U = _tubes(c, seed).to(_dtype(c)).contiguous()
        h = H.Batch(_lengths(c).numpy(), 5 / 3, EXACT, MINMOD, c["precision"])
        if c["mlp"]:
            _trained(h, seed)
        torch.cuda.synchronize()
        h.set_state(U)
        h.run(1, c["cfl"])
        return dict(case=c, h=h, U=U, out=torch.empty_like(U))
    d = _setup(c, seed)
    U = d["U"].to(_dtype(c)).contiguous()
    n = [c.get(k, 1) for k in ("nx", "ny", "nz")]
    h = H.Grid(d["dim"], n, [f.numpy() for f in d["faces"]], d["bc"], d["coords"], d["gamma"], d["ns"], c["riemann"],
               c["limiter"], c["precision"])
    if d["rad"]:
        h.set_eos_radiation(*d["rad"])
    if d["grav"] == "mono":
        h.set_sources(gravity=H.HYDRO_GRAV_POINT_MONOPOLE, G=1.0, Mc=1.0)
    elif d["grav"]:
        h.set_sources(gravity=H.HYDRO_GRAV_UNIFORM, g0=d["grav"])
    h.set_step_totals(c["totals"])
    torch.cuda.synchronize()
    h.set_state(U)
    if c["loop"]:
        h.step(h.cfl_dt(d["cfl"]))
    else:
        h.run(1, d["cfl"])
    return dict(case=c, h=h, U=U, cfl=d["cfl"], out=torch.empty_like(U))


def run(state):
    c = state["case"]
    if c["kind"] == "grad":
        H.hydro_mlp_loss_grad_device(state["w"].data_ptr(), state["x"].data_ptr(), state["y"].data_ptr(), c["n"],
                                     state["grad"].data_ptr(), state["loss"].data_ptr(),
                                     torch.cuda.current_stream().cuda_stream)
        return state["grad"], state["loss"]
    h = state["h"]
    h.set_state(state["U"])
    if c["kind"] == "tubes":
        h.run(c["steps"], c["cfl"])
        return h.get_state(state["out"])
    if c["loop"]:
        for _ in range(c["steps"]):
            h.step(h.cfl_dt(state["cfl"]))
    else:
        h.run(c["steps"], state["cfl"])
    out = {"state": h.get_state(state["out"])}
    if c["totals"]:
        # (the totals carry the rounding of the state they sum)
        out["totals"] = h.step_totals().astype("f8" if c["precision"] == 64 else "f4")
    return out


def work(case):
    c = case
    if c["kind"] == "grad":  # forward, backward to the inputs of each layer, weight gradients
        per = 2 * 3 * (6 * 64 + 64 * 64 + 64) - 2 * 6 * 64
        return dict(bytes=c["n"] * 28 + H.HYDRO_MLP_NPARAM * 12 + 8, flops=c["n"] * per)
    if c["kind"] == "tubes":
        cells, nv, dim = int(_lengths(c).sum()), 3, 1
    else:
        dim = 1 + ("ny" in c) + ("nz" in c)
        cells = c["nx"] * c.get("ny", 1) * c.get("nz", 1)
        nv = 2 + dim + {"kh": 1, "rt": 1, "wedge": 3}.get(c["setup"], 0)
    # each step reads the state once and writes it once; per cell and axis: slopes
    # and two face states (8 per variable), two fluxes, the half step, two
    # conversions back, one face solve and the update (about 24 per variable)
    return dict(bytes=2 * nv * (c["precision"] // 8) * cells * c["steps"],
                flops=32 * nv * dim * cells * c["steps"])


# ---------------------------------------------------------------------------
# The same in 64 bits, in plain torch
# ---------------------------------------------------------------------------
class _Gas:
    def __init__(self, gamma, rad):
        self.g, self.rad = gamma, rad

    def _temp(self, c1, c4, y):  # c1 T + c4 T^4 = y, Newton from above
        t = torch.minimum(y / c1, (y / c4).sqrt().sqrt())
        for _ in range(60):
            n = t - (c1 * t + c4 * t ** 4 - y) / (c1 + 4 * c4 * t ** 3)
            done = bool(((n - t).abs() <= 1e-15 * n).all())
            t = n
            if done:
                break
        return t

    def p(self, rho, e):
        if not self.rad:
            return (self.g - 1) * e
        R, a = self.rad
        t = self._temp(rho * R / (self.g - 1), a, e)
        return rho * R * t + a / 3 * t ** 4

    def e_c(self, rho, p):
        """Internal energy and sound speed."""
        if not self.rad:
            return p / (self.g - 1), (self.g * p / rho).sqrt()
        R, a = self.rad
        t = self._temp(rho * R, a / 3, p)
        pg, pr = rho * R * t, a / 3 * t ** 4
        al, k = pr / pg, 1 / (self.g - 1)
        return pg * k + 3 * pr, ((self.g * k + 20 * al + 16 * al * al) / (k + 12 * al) * pg / rho).sqrt()


def _prim(gas, U, D):
    W = U / U[0]
    W[0] = U[0]
    W[1 + D] = gas.p(U[0], U[1 + D] - 0.5 * (U[1:1 + D] * W[1:1 + D]).sum(0))
    return W


def _flux(gas, W, D, d):
    """Conserved state, flux along d and sound speed."""
    e, cs = gas.e_c(W[0], W[1 + D])
    U = W * W[0]
    U[0] = W[0]
    U[1 + D] = e + 0.5 * (U[1:1 + D] * W[1:1 + D]).sum(0)
    F = U * W[1 + d]
    F[1 + d] += W[1 + D]
    F[1 + D] += W[1 + D] * W[1 + d]
    return U, F, cs


def _limit(kind, a, b):
    pr = a * b
    if kind == MINMOD:
        s = torch.where(a.abs() < b.abs(), a, b)
    elif kind == VANLEER:
        s = 2 * pr / (a + b)
    else:
        s = pr * (a + b) / (a * a + b * b)
    return torch.where(pr > 0, s, torch.zeros_like(s))


def _star(g, WL, WR, cL, cR, D, d):
    """Pressure and velocity between the waves (Newton on the pressure functions)."""
    (rL, uL, pL), (rR, uR, pR) = [(W[0], W[1 + d], W[1 + D]) for W in (WL, WR)]
    z = (g - 1) / (2 * g)
    p = ((cL + cR - 0.5 * (g - 1) * (uR - uL)) / (cL / pL ** z + cR / pR ** z)) ** (1 / z)

    def f(p, r, q, c):
        A, B = 2 / ((g + 1) * r), (g - 1) / (g + 1) * q
        s = (A / (p + B)).sqrt()
        x = (p / q) ** z
        shock = p > q
        return (torch.where(shock, (p - q) * s, 2 * c / (g - 1) * (x - 1)),
                torch.where(shock, s * (1 - 0.5 * (p - q) / (B + p)), x * q / (p * r * c)))

    for _ in range(60):
        fL, dL = f(p, rL, pL, cL)
        fR, dR = f(p, rR, pR, cR)
        n = p - (fL + fR + uR - uL) / (dL + dR)
        n = torch.where(n > 0, n, 1e-14 * (pL + pR))
        done = not bool(((n - p).abs() > 2e-15 * n).any())
        p = n
        if done:
            break
    return p, 0.5 * (uL + uR + f(p, rR, pR, cR)[0] - f(p, rL, pL, cL)[0])


def _sample(g, WL, WR, D, d):
    """The state on the face of the exact solution."""
    cL, cR = (g * WL[1 + D] / WL[0]).sqrt(), (g * WR[1 + D] / WR[0]).sqrt()
    ps, us = _star(g, WL, WR, cL, cR, D, d)
    left = us >= 0
    s = torch.where(left, 1.0, -1.0)
    W = torch.where(left, WL, WR)
    c = torch.where(left, cL, cR)
    r, u, p = W[0], s * W[1 + d], W[1 + D]  # a left wave, seen from its side
    q, us = ps / p, s * us
    b = (g - 1) / (g + 1)
    cs = c * q ** ((g - 1) / (2 * g))
    cf = 2 / (g + 1) * (c + 0.5 * (g - 1) * u)
    shock = ps > p
    head = torch.where(shock, u - c * ((g + 1) / (2 * g) * q + (g - 1) / (2 * g)).sqrt(), u - c)
    tail = torch.where(shock, head, us - cs)
    rs = torch.where(shock, r * (q + b) / (b * q + 1), r * q ** (1 / g))
    x = (cf / c).clamp(min=1e-300)
    out = W.clone()
    for k, (star, fan) in {0: (rs, r * x ** (2 / (g - 1))), 1 + d: (us, cf), 1 + D: (ps, p * x ** (2 * g / (g - 1)))}.items():
        own = u if k == 1 + d else W[k]
        v = torch.where(head >= 0, own, torch.where(tail <= 0, star, fan))
        out[k] = s * v if k == 1 + d else v
    return out


def _solve(gas, rs, WL, WR, D, d):
    if rs == EXACT:
        diff = (WL != WR).any(0)
        W = WL.clone()
        W[:, diff] = _sample(gas.g, WL[:, diff], WR[:, diff], D, d)
        return _flux(gas, W, D, d)[1]
    UL, FL, cL = _flux(gas, WL, D, d)
    UR, FR, cR = _flux(gas, WR, D, d)
    uL, uR, pL, pR = WL[1 + d], WR[1 + d], WL[1 + D], WR[1 + D]
    SL, SR = torch.minimum(uL - cL, uR - cR), torch.maximum(uL + cL, uR + cR)
    if rs == HLL:
        F = (SR * FL - SL * FR + SL * SR * (UR - UL)) / (SR - SL)
    else:
        aL, aR = WL[0] * (SL - uL), WR[0] * (SR - uR)
        Ss = (pR - pL + uL * aL - uR * aR) / (aL - aR)
        left = Ss >= 0
        S, a, W = torch.where(left, SL, SR), torch.where(left, aL, aR), torch.where(left, WL, WR)
        U, F = torch.where(left, UL, UR), torch.where(left, FL, FR)
        k = a / (S - Ss)
        Us = W * k
        Us[0] = k
        Us[1 + d] = k * Ss
        Us[1 + D] = k * (U[1 + D] / W[0] + (Ss - W[1 + d]) * (Ss + W[1 + D] / a))
        F = F + S * (Us - U)
    return torch.where(SL >= 0, FL, torch.where(SR <= 0, FR, F))


def _grid64(c, seed):
    d0 = _setup(c, seed)
    U = d0["U"].to(_dtype(c)).to(F64)
    D, gas, sph = d0["dim"], _Gas(d0["gamma"], d0["rad"]), d0["coords"] == 1
    ax = [3 - d for d in range(D)]  # tensor axis of grid axis d
    face, src, flip = [], [], []
    for d in range(D):
        f, (lo, hi) = d0["faces"][d].to(DEV), d0["bc"][d]
        n = f.numel() - 1
        i = torch.arange(-2, n + 2, device=DEV)
        low = {PERIODIC: i + n, TRANSMISSIVE: 0 * i, REFLECTIVE: -1 - i}[lo]
        top = {PERIODIC: i - n, TRANSMISSIVE: 0 * i + n - 1, REFLECTIVE: 2 * n - 1 - i}[hi]
        s = torch.where(i < 0, low, torch.where(i >= n, top, i))
        w = (f[1:] - f[:-1])[s]
        e = torch.cat([f[:1] - w[1] - w[0], f[:1] - w[1], f, f[-1:] + w[-2], f[-1:] + w[-2] + w[-1]])
        face.append(e)
        src.append(s)
        flip.append(((i < 0) & (lo == REFLECTIVE)) | ((i >= n) & (hi == REFLECTIVE)))

    def on(v, d):  # a vector along grid axis d, to be used with (nv, nz, ny, nx)
        shape = [1, 1, 1, 1]
        shape[ax[d]] = -1
        return v.reshape(shape)

    def cut(t, d, a, b):
        return t.narrow(ax[d], a, t.shape[ax[d]] - a - b)

    def inner(t, skip=-1):
        for d in range(D):
            if d != skip:
                t = cut(t, d, 1, 1)
        return t

    f = [v.to(DEV) for v in d0["faces"]]
    wid = [v[1:] - v[:-1] for v in f]
    # physical widths of interior cells
    h = [on(w, d) for d, w in enumerate(wid)]
    area = [torch.ones(1, device=DEV, dtype=F64)] * D   # of the faces along d, over its cells' common factors
    inv = [1 / x for x in h]                            # what multiplies (area flux) differences
    if sph:
        r, th = f[0], f[1]
        rc, sn = 0.5 * (r[1:] + r[:-1]), torch.sin(th)
        s_mid = 0.5 * (sn[1:] + sn[:-1])
        h[1], h[2] = h[1] * on(rc, 0), h[2] * on(rc, 0) * on(s_mid, 1)
        a = (r[1:] ** 3 - r[:-1] ** 3) / 3
        a2 = 0.5 * (r[1:] ** 2 - r[:-1] ** 2)
        b = torch.cos(th[:-1]) - torch.cos(th[1:])
        area = [on(r * r, 0), on(sn, 1), torch.ones(1, device=DEV, dtype=F64)]
        inv = [on(1 / a, 0), on(a2 / a, 0) * on(1 / b, 1), on(a2 / a, 0) * on(wid[1] / b, 1) * on(1 / wid[2], 2)]
        qr = on(wid[0] / ((r[1:] + r[:-1]) * a), 0)
        gr = on((r[1:] ** 2 - r[:-1] ** 2) / a, 0)
        gt = on(a2 / a, 0) * on((sn[1:] - sn[:-1]) / b, 1)
        qt = on(a2 / a, 0) * on((sn[1:] - sn[:-1]) / ((sn[1:] + sn[:-1]) * b), 1)
    hx = h  # widths of the cells -1..n: those of the cells they copy
    hext = []
    for d in range(D):
        t = hx[d]
        for k in range(D):
            if t.shape[ax[k]] > 1:
                t = t.index_select(ax[k], src[k][1:-1])
        hext.append(t)
    cen = [0.5 * (e[1:] + e[:-1]) for e in face]

    for _ in range(c["steps"]):
        W0 = _prim(gas, U, D)
        cs = gas.e_c(W0[0], W0[1 + D])[1]
        dt = d0["cfl"] / float(sum((W0[1 + d].abs() + cs) / h[d][0] for d in range(D)).max())
        Ue = U
        for d in range(D):
            Ue = Ue.index_select(ax[d], src[d])
            if flip[d].any():
                Ue[1 + d] *= torch.where(on(flip[d], d)[0], -1.0, 1.0)
        W = _prim(gas, Ue, D)
        Uc, Wc = inner(Ue), inner(W)
        lohi, dU = [], torch.zeros_like(Uc)
        for d in range(D):
            x = cen[d]
            wm, wp = inner(cut(W, d, 0, 2), d), inner(cut(W, d, 2, 0), d)
            sig = _limit(c["limiter"], (Wc - wm) / on(x[1:-1] - x[:-2], d), (wp - Wc) / on(x[2:] - x[1:-1], d))
            sig = sig * on(0.5 * (face[d][2:-1] - face[d][1:-2]), d)
            (Ul, Fl, _), (Uh, Fh, _) = _flux(gas, Wc - sig, D, d), _flux(gas, Wc + sig, D, d)
            dU += 0.5 * dt * (Fl - Fh) / hext[d]
            lohi.append((Ul, Uh))
        dudt = torch.zeros_like(U)
        keep = []
        for d in range(D):
            side = []
            for u in lohi[d]:
                u = u + dU
                e = u[1 + D] - 0.5 * (u[1:1 + D] ** 2).sum(0) / u[0]
                u = torch.where((u[0] > 0) & (e > 0), u, Uc)
                side.append(_prim(gas, inner(u, d), D))
            F = _solve(gas, c["riemann"], cut(side[1], d, 0, 1), cut(side[0], d, 1, 0), D, d)
            AF = F * area[d]
            dudt += (cut(AF, d, 0, 1) - cut(AF, d, 1, 0)) * inv[d]
            keep.append((F, AF))
        if sph:
            mean = lambda F, d: 0.5 * (cut(F, d, 0, 1) + cut(F, d, 1, 0))  # noqa: E731
            T2, T3 = mean(keep[1][0][2:3], 1)[0], mean(keep[2][0][3:4], 2)[0]
            dudt[1] += 0.5 * (T2 + T3) * gr[0]
            dudt[2] += -qr[0] * 2 * mean(keep[0][1][2:3], 0)[0] + T3 * gt[0]
            dudt[3] += -qr[0] * 2 * mean(keep[0][1][3:4], 0)[0] - qt[0] * 2 * mean(keep[1][1][3:4], 1)[0]
            dV = on(a, 0)[0] * on(b, 1)[0] * on(wid[2], 2)[0]
            m = (U[0] * dV).sum((0, 1)) * 4 * math.pi / (b.sum() * wid[2].sum())
            g = -(1.0 + torch.cumsum(m, 0) - 0.5 * m) / rc ** 2
            dudt[1] += U[0] * g
            dudt[1 + D] += U[1] * g
        elif d0["grav"]:
            for d in range(D):
                dudt[1 + d] += U[0] * d0["grav"][d]
                dudt[1 + D] += U[1 + d] * d0["grav"][d]
        U = U + dt * dudt
    out = {"state": U}
    if c["totals"]:
        vol = (on(a, 0) * on(b, 1) * on(wid[2], 2)) if sph else 1.0
        for d in range(0 if sph else D):
            vol = vol * on(wid[d], d)
        out["totals"] = (U * vol).sum((1, 2, 3))
    return out


def _tubes64(c, seed):
    gas = _Gas(5 / 3, None)
    U = _tubes(c, seed).to(_dtype(c)).to(F64)
    n = _lengths(c).to(DEV)
    end = torch.cumsum(n, 0)
    first, last = end - n, end - 1
    tube = torch.repeat_interleave(torch.arange(c["ntubes"], device=DEV), n)
    i = torch.arange(tube.numel(), device=DEV)
    im, ip = torch.maximum(i - 1, first[tube]), torch.minimum(i + 1, last[tube])
    inv = n[tube].to(F64)
    for _ in range(c["steps"]):
        W = _prim(gas, U, 1)
        s = torch.segment_reduce(W[1].abs() + gas.e_c(W[0], W[2])[1], "max", lengths=n)
        dtdx = (c["cfl"] / (s * n))[tube] * inv
        sig = 0.5 * _limit(MINMOD, W - W[:, im], W[:, ip] - W)
        (Ul, Fl, _), (Uh, Fh, _) = _flux(gas, W - sig, 1, 0), _flux(gas, W + sig, 1, 0)
        dU = 0.5 * dtdx * (Fl - Fh)
        side = []
        for u in (Ul + dU, Uh + dU):
            ok = (u[0] > 0) & (u[2] - 0.5 * u[1] ** 2 / u[0] > 0)
            side.append(_prim(gas, torch.where(ok, u, U), 1))
        L = side[1][:, im]
        L[:, first] = W[:, first]
        F = _solve(gas, EXACT, L, side[0], 1, 0)
        Fp = F[:, ip].clone()
        Fp[:, last] = _solve(gas, EXACT, side[1][:, last], W[:, last], 1, 0)
        U = U + dtdx * (F - Fp)
    return U


def exact(case, seed):
    c = case
    if c["kind"] == "tubes":
        return _tubes64(c, seed)
    if c["kind"] == "grid":
        return _grid64(c, seed)
    w, x, y = [t.to(F64) for t in _grad_inputs(c, seed)]
    w.requires_grad_(True)
    w1, b1, w2, b2, w3, b3 = torch.split(w, [384, 64, 4096, 64, 64, 1])
    act = torch.nn.functional.silu
    h = act(act(x @ w1.view(64, 6).T + b1) @ w2.view(64, 64).T + b2)
    loss = ((h @ w3 + b3 - y) ** 2).mean()
    loss.backward()
    return w.grad, loss.detach().reshape(1)
