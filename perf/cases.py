"""Performance cases of the solver: what a user has it do, through its public entry points.

``listed()`` names twelve workloads; ``draw(rng)`` gives more of the same ranges.  ``prepare``
builds what a user's program holds before the call (initial states and handles on the GPU,
or host states where the call streams through host memory), ``run`` is one pass, ``work``
what a pass cannot do without, and ``exact`` the same outputs from a plain torch FP64
restatement of the method in this file.

Every pass of a grid case is a whole call sequence: a new primitive state goes in
(``set_state``), a fixed number of CFL steps is taken (``run``), the conserved state comes out
(``get_state``).  Kinds of cases (``kind``):

  shock     1D shock tube run to a final time (the modified Sod test)
  one       a single step of a small 2D grid from a device buffer into another
            (``msh_step_noalloc``), as a host loop that owns its buffers takes it
  blast     2D anisotropic-stress blast
  disc      2D stellar disc in a fixed external potential, outflow
  box       3D turbulent box, also with other fluxes, boundaries, transverse terms, or
            self-gravity
  tubes     batched 1D Riemann problems in one persistent launch
  gradient  forward run of the disc and the gradient of a linear functional of the final
            state with respect to the initial state, through torch.autograd
  ensemble  independent 3D states streamed through host memory
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1210_5246_gb300 import autograd, msh

PER, OUT, REF = msh.PERIODIC, msh.OUTFLOW, msh.REFLECT
BCS = {"periodic": (PER, PER), "outflow": (OUT, OUT), "reflect": (REF, REF), "mixed": (REF, OUT)}
SCHEMES = {"hll": msh.MUSCL_HANCOCK, "kt": msh.KT, "roe": msh.MUSCL_HANCOCK_ROE, "hllc": msh.MUSCL_HANCOCK_HLLC}
PREC = {"f32": msh.FP32, "f64": msh.FP64}
DTYPE = {"f32": torch.float32, "f64": torch.float64}


def listed():
    return [
        # the paper's shock-tube test: a few hundred cells, one small launch after another
        dict(name="sod 256 f64", kind="shock", nx=256, prec="f64", bc="outflow", scheme="hll", t_end=0.2),
        # a host loop stepping its own small buffers, one call per step
        dict(name="one step 96x96 f32", kind="one", nx=96, ny=96, prec="f32", bc="periodic"),
        # the 2D benchmark workload, FP32; its states fit in L2
        dict(name="blast 1024x1024 f32", kind="blast", nx=1024, ny=1024, prec="f32", bc="periodic", scheme="hll",
             steps=48),
        # a 2D run in FP64 on a rectangular grid that no tile divides
        dict(name="blast 500x381 f64", kind="blast", nx=500, ny=381, prec="f64", bc="mixed", scheme="hll", steps=12),
        # the stellar disc's forward run: small 2D grid, gravity source, outflow
        dict(name="disc 512x512 f32", kind="disc", nx=512, prec="f32", steps=64),
        # the benchmark: the turbulent box
        dict(name="box 256^3 f32", kind="box", nx=256, ny=256, nz=256, prec="f32", bc="periodic", scheme="hll",
             ctu=False, grav=0.0, steps=10),
        # a small ragged box with walls and open sides and the contact-resolving flux
        dict(name="box 97x61x45 f32 hllc", kind="box", nx=97, ny=61, nz=45, prec="f32", bc="mixed", scheme="hllc",
             ctu=False, grav=0.0, steps=20),
        # the 3D box in FP64
        dict(name="box 64^3 f64", kind="box", nx=64, ny=64, nz=64, prec="f64", bc="periodic", scheme="hll", ctu=False,
             grav=0.0, steps=6),
        # the corner-transport-upwind form of the box
        dict(name="box 160^3 f32 ctu", kind="box", nx=160, ny=160, nz=160, prec="f32", bc="periodic", scheme="hll",
             ctu=True, grav=0.0, steps=8),
        # thousands of Riemann problems of uneven lengths
        dict(name="tubes 4096 f32", kind="tubes", count=4096, nmin=128, nmax=2048, prec="f32", t_end=0.1),
        # a gradient through a recorded run, in the precision that resolves it
        dict(name="disc gradient 128x128 f64", kind="gradient", nx=128, prec="f64", steps=20, ck=10),
        # a parameter study: states from host memory, one step each, results back
        dict(name="ensemble 6 x 128^3 f32", kind="ensemble", nx=128, ny=128, nz=128, count=6, prec="f32",
             bc="periodic", steps=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["shock", "one", "blast", "blast", "disc", "box", "box", "box", "tubes", "gradient", "ensemble"])
    prec = rng.choice(["f32", "f32", "f64"])
    if kind == "shock":
        return dict(kind=kind, nx=_log_int(rng, 64, 2048), prec=prec, bc=rng.choice(["outflow", "reflect"]),
                    scheme=rng.choice(["hll", "hllc", "kt"]), t_end=round(rng.uniform(0.05, 0.2), 4))
    if kind == "one":
        return dict(kind=kind, nx=_log_int(rng, 24, 512), ny=_log_int(rng, 24, 512), prec=prec,
                    bc=rng.choice(["periodic", "outflow", "reflect"]))
    if kind == "blast":
        hi = 1500 if prec == "f32" else 500
        return dict(kind=kind, nx=_log_int(rng, 64, hi), ny=_log_int(rng, 64, hi), prec=prec,
                    bc=rng.choice(["periodic", "outflow", "reflect", "mixed"]), scheme=rng.choice(["hll", "hllc", "kt"]),
                    steps=rng.randint(4, 48 if prec == "f32" else 12))
    if kind == "disc":
        return dict(kind=kind, nx=_log_int(rng, 96, 768 if prec == "f32" else 320), prec=prec,
                    steps=rng.randint(8, 64 if prec == "f32" else 16))
    if kind == "box":
        hi = 256 if prec == "f32" else 72
        sizes = [_log_int(rng, 24, hi) for _ in range(3)]
        form = rng.choice(["plain", "plain", "plain", "ctu", "gravity"])
        bc = rng.choice(["periodic", "periodic", "outflow", "mixed"]) if form == "plain" else "periodic"
        scheme = rng.choice(["hll", "hll", "hllc", "roe", "kt"]) if form == "plain" else "hll"
        return dict(kind=kind, nx=sizes[0], ny=sizes[1], nz=sizes[2], prec=prec, bc=bc, scheme=scheme,
                    ctu=form == "ctu", grav=round(rng.uniform(0.05, 0.3), 3) if form == "gravity" else 0.0,
                    steps=rng.randint(3, 8 if prec == "f32" else 5))
    if kind == "tubes":
        nmin = _log_int(rng, 32, 256 if prec == "f32" else 96)
        return dict(kind=kind, count=_log_int(rng, 64, 2048 if prec == "f32" else 256), nmin=nmin, nmax=4 * nmin,
                    prec=prec, t_end=round(rng.uniform(0.02, 0.1 if prec == "f32" else 0.04), 4))
    if kind == "gradient":
        return dict(kind=kind, nx=_log_int(rng, 48, 160), prec="f64", steps=rng.randint(4, 20), ck=rng.randint(2, 10))
    return dict(kind=kind, nx=_log_int(rng, 32, 128), ny=_log_int(rng, 32, 128), nz=_log_int(rng, 32, 128),
                count=rng.randint(2, 6), prec=prec if prec == "f32" else "f32", bc="periodic", steps=rng.randint(1, 3))


# ------------------------------------------------------------------------------- inputs
def _gen(seed, device="cuda"):
    g = torch.Generator(device=device)
    g.manual_seed(int(seed))
    return g


def _rand(g, shape):
    return torch.rand(shape, generator=g, device=g.device, dtype=torch.float64)


def _randn(g, shape):
    return torch.randn(shape, generator=g, device=g.device, dtype=torch.float64)


def _spd(g, shape, lo, hi, off):
    """P = L L^T per cell: diagonal of L uniform in [lo, hi], off-diagonal normal(0, off)."""
    a, b, c = (lo + (hi - lo) * _rand(g, shape) for _ in range(3))
    p, q, r = (off * _randn(g, shape) for _ in range(3))
    return [a * a, p * a, q * a, p * p + b * b, q * p + r * b, q * q + r * r + c * c]


def _random_field(g, nz, ny, nx):
    """Unit-variance periodic Gaussian field with 3D power ~ k^-4 (k in units of the box)."""
    kz = torch.fft.fftfreq(nz, 1.0 / nz, device=g.device, dtype=torch.float64)[:, None, None]
    ky = torch.fft.fftfreq(ny, 1.0 / ny, device=g.device, dtype=torch.float64)[None, :, None]
    kx = torch.fft.rfftfreq(nx, 1.0 / nx, device=g.device, dtype=torch.float64)[None, None, :]
    k2 = kx * kx + ky * ky + kz * kz
    amp = torch.where(k2 > 0, 1.0 / torch.clamp(k2, min=1.0), torch.zeros_like(k2))
    f = torch.fft.irfftn(torch.fft.rfftn(_randn(g, (nz, ny, nx))) * amp, s=(nz, ny, nx))
    return (f - f.mean()) / f.std()


def _box_state(seed, nz, ny, nx):
    """Lognormal density (sigma 0.5), k^-2-spectrum velocity with rms |u| = 1, random SPD P."""
    g = _gen(seed)
    rho = torch.exp(0.5 * _random_field(g, nz, ny, nx) - 0.125)
    u = [_random_field(g, nz, ny, nx) for _ in range(3)]
    rms = torch.sqrt(sum((x * x).mean() for x in u))
    return torch.stack([rho] + [x / rms for x in u] + _spd(g, (nz, ny, nx), 0.3, 1.0, 0.1))


def _blast_state(seed, ny, nx):
    """Background rho = 1 (1 % noise), P = 0.1; disc of radius 0.1 with P_xx 10, P_yy 1, P_xy 2."""
    g = _gen(seed)
    x = (torch.arange(nx, device="cuda", dtype=torch.float64) + 0.5) / nx
    y = (torch.arange(ny, device="cuda", dtype=torch.float64) + 0.5) / ny
    disc = ((x[None, :] - 0.5) ** 2 + (y[:, None] - 0.5) ** 2 < 0.01)[None]
    W = torch.zeros((10, 1, ny, nx), device="cuda", dtype=torch.float64)
    W[0] = 1.0 + 0.01 * (2.0 * _rand(g, (1, ny, nx)) - 1.0)
    W[4] = torch.where(disc, 10.0, 0.1)
    W[5] = torch.where(disc, 2.0, 0.0)
    W[7] = torch.where(disc, 1.0, 0.1)
    W[9] = 0.1
    return W


DISC_L = 20.0


def _disc_axes(n, ghost=0):
    dx = 2.0 * DISC_L / n
    return -DISC_L + (torch.arange(-ghost, n + ghost, device="cuda", dtype=torch.float64) + 0.5) * dx


def _disc_state(seed, n):
    """Exponential disc (scale length 3) with 1 % noise, rotating in the logarithmic potential,
    velocity dispersion from Toomre Q = 1.2 with a floor, isotropic in the plane."""
    g = _gen(seed)
    c = _disc_axes(n)
    X, Y = c[None, :], c[:, None]
    R = torch.sqrt(X * X + Y * Y)

    def profile(r):
        S = 0.1 * torch.exp(-r / 3.0)
        kap = torch.sqrt(2.0 * r * r + 4.0) / (r * r + 1.0)
        return S, torch.clamp(3.36 * 1.2 * S / kap, min=0.05)

    S, sig = profile(R)
    h = 1e-5
    f = lambda r: (lambda s, v: s * v * v)(*profile(r))
    lo = torch.clamp(R - h, min=0.0)
    jeans = R / S * (f(R + h) - f(lo)) / (R + h - lo)
    vphi = torch.sqrt(torch.clamp(R * R / (R * R + 1.0) + jeans, min=0.0))
    Rs = torch.clamp(R, min=1e-30)
    S = S * (1.0 + 0.01 * (2.0 * _rand(g, (n, n)) - 1.0))
    P = S * sig * sig
    Z = torch.zeros_like(S)
    return torch.stack([S, -vphi * Y / Rs, vphi * X / Rs, Z, P, Z, Z, P, Z, P]).reshape(10, 1, n, n).contiguous()


def _disc_potential(n):
    """Phi = ln(1 + R^2) / 2 at the cell centres with one ghost layer, [1][n+2][n+2]."""
    c = _disc_axes(n, 1)
    return (0.5 * torch.log(1.0 + c[None, :] ** 2 + c[:, None] ** 2)).reshape(1, n + 2, n + 2)


def _shock_state(seed, n):
    """The modified Sod states; the density on either side varies by a few per cent with the seed."""
    g = _gen(seed, "cpu")
    a, b = (0.05 * (2.0 * torch.rand(2, generator=g, dtype=torch.float64) - 1.0)).tolist()
    left = (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) / n < 0.5
    W = torch.zeros((10, 1, 1, n), device="cuda", dtype=torch.float64)
    W[0, 0, 0] = torch.where(left, 1.0 + a, 0.125 * (1.0 + b))
    for c in (4, 7, 9):
        W[c, 0, 0] = torch.where(left, 1.0, 0.1)
    return W


def _tube_states(seed, count, nmin, nmax):
    """Lengths spread evenly over the logarithm of [nmin, nmax], in random order; per side rho
    log-uniform [0.3, 3], u_x uniform [-0.3, 0.3], P = L L^T (diagonal uniform [0.5, 1],
    off-diagonal normal(0, 0.1)): ratios up to those of the shock-tube test.  Stronger jumps
    come near vacuum, where the solver's discrete choices (which cells fall back to first
    order) are decided by rounding and FP32 results are not comparable cell by cell."""
    rng = np.random.Generator(np.random.PCG64(seed))
    q = (np.arange(count) + 0.5) / count
    length = rng.permutation(np.rint(np.exp(math.log(nmin) + q * math.log(nmax / nmin))).astype(np.int32))

    def side(m):
        W = np.zeros((m, 10))
        W[:, 0] = np.exp(rng.uniform(math.log(0.3), math.log(3.0), m))
        W[:, 1] = rng.uniform(-0.3, 0.3, m)
        a, b, c = (rng.uniform(0.5, 1.0, m) for _ in range(3))
        p, q, r = (rng.normal(0.0, 0.1, m) for _ in range(3))
        W[:, 4], W[:, 5], W[:, 6] = a * a, p * a, q * a
        W[:, 7], W[:, 8], W[:, 9] = p * p + b * b, q * p + r * b, q * q + r * r + c * c
        return W

    return length, side(count), side(count)


def _cfl(case):
    return 0.8 if case["kind"] in ("shock", "tubes") and case.get("scheme") != "kt" else 0.4 if case.get("scheme") == "kt" else 0.5


def _geometry(case):
    """(n, lo, hi, bc pairs) of a grid case."""
    k = case["kind"]
    if k == "shock":
        return (case["nx"],), (0.0,), (1.0,), (BCS[case["bc"]],)
    if k in ("disc", "gradient"):
        return (case["nx"],) * 2, (-DISC_L,) * 2, (DISC_L,) * 2, (BCS["outflow"],) * 2
    n = (case["nx"], case["ny"]) + ((case["nz"],) if k in ("box", "ensemble") else ())
    return n, (0.0,) * len(n), (1.0,) * len(n), (BCS[case["bc"]],) * len(n)


def _initial(case, seed):
    """The primitive initial state of a grid case in the case's precision."""
    k = case["kind"]
    if k == "shock":
        W = _shock_state(seed, case["nx"])
    elif k in ("blast", "one"):
        W = _blast_state(seed, case["ny"], case["nx"])
    elif k in ("disc", "gradient"):
        W = _disc_state(seed, case["nx"])
    else:
        W = _box_state(seed, case["nz"], case["ny"], case["nx"])
    return W.to(DTYPE[case["prec"]]).contiguous()


def _ensemble_states(case, seed):
    return [_cons(_box_state(1000 * seed + k, case["nz"], case["ny"], case["nx"])).to(torch.float32)
            for k in range(case["count"])]


def _cotangent(case, seed):
    """dL/dU_N of the gradient case: a smooth weight on every conserved field."""
    g = _gen(seed + 77, "cpu")
    c = _disc_axes(case["nx"])
    a = torch.rand((10, 4), generator=g, dtype=torch.float64).tolist()
    return torch.stack([(torch.cos(0.3 * p * c[None, :] + q) * torch.cos(0.3 * r * c[:, None] + s))
                        for p, q, r, s in a]).reshape(10, 1, case["nx"], case["nx"]).contiguous()


def prepare(case, seed):
    k = case["kind"]
    if k == "tubes":
        length, WL, WR = _tube_states(seed, case["count"], case["nmin"], case["nmax"])
        return dict(case=case, batch=msh.Batch(length, WL, WR, case["t_end"], cfl=_cfl(case), precision=PREC[case["prec"]]))
    n, lo, hi, bc = _geometry(case)
    if k == "one":
        W = _cons(_initial(case, seed).double()).to(DTYPE[case["prec"]]).contiguous()
        return dict(case=case, n=n, lo=lo, hi=hi, bc=bc, U=W, out=torch.empty_like(W))
    grid = msh.Grid(n, lo, hi, bc, _cfl(case), PREC[case["prec"]])
    if k == "ensemble":
        ins = [U.cpu().pin_memory().numpy() for U in _ensemble_states(case, seed)]
        outs = [torch.empty(U.shape, dtype=torch.float32).pin_memory().numpy() for U in ins]
        return dict(case=case, grid=grid, ins=ins, outs=outs)
    if k in ("disc", "gradient"):
        grid.set_potential(_disc_potential(case["nx"]).cpu().numpy())
    W = _initial(case, seed)
    s = dict(case=case, grid=grid, W=W, out=torch.empty_like(W))
    if k == "gradient":
        s["G"] = _cotangent(case, seed)
        return s
    if case.get("scheme", "hll") != "hll":
        grid.set_scheme(SCHEMES[case["scheme"]])
    if case.get("ctu"):
        grid.set_ctu(True)
    if case.get("grav", 0.0) > 0.0:
        grid.set_self_gravity(case["grav"])
    return s


def run(state):
    case = state["case"]
    k = case["kind"]
    if k == "tubes":
        b = state["batch"]
        b.reset()
        b.run()
        return b.get_state()
    if k == "one":
        dt = msh.msh_step_noalloc(state["n"], state["lo"], state["hi"], state["bc"], PREC[case["prec"]], 0.5,
                                  state["U"], state["out"])
        return dict(U=state["out"], dt=dt)
    g = state["grid"]
    if k == "ensemble":
        g.run_ensemble(state["ins"], state["outs"], nsteps=case["steps"])
        return state["outs"]
    if k == "gradient":
        W = state["W"].detach().requires_grad_(True)
        U = autograd.run(W, g, case["steps"], case["ck"])
        grad, = torch.autograd.grad(U, W, state["G"])
        return dict(U=U.detach(), grad=grad)
    g.set_time(0.0)
    g.set_state(state["W"], msh.PRIMITIVE)
    if k == "shock":
        _, t = g.run(t_end=case["t_end"])
    else:
        _, t = g.run(max_steps=case["steps"])
    return dict(U=g.get_state(out=state["out"]), t=t)


def work(case):
    """Bytes: every step reads and writes the ten fields once (dt needs a global reduction, so
    steps cannot be merged); tubes stay on the chip, so theirs are read and written once per
    run.  Operations: about 600 per cell and direction (reconstruction 330, flux 190, update)
    and 100 for conversion, time step and totals; twice that for the central scheme's two
    stages, four times for a step and its reverse."""
    k = case["kind"]
    es = 4 if case["prec"] == "f32" else 8
    if k == "tubes":
        mean = (case["nmax"] - case["nmin"]) / math.log(case["nmax"] / case["nmin"])
        square = (case["nmax"] ** 2 - case["nmin"] ** 2) / (2.0 * math.log(case["nmax"] / case["nmin"]))
        # a tube of n cells takes about 3.4 n steps per unit time
        return dict(bytes=20.0 * es * case["count"] * mean, flops=700.0 * case["count"] * square * case["t_end"] * 3.4)
    n, _, _, _ = _geometry(case)
    cells, ndim = float(np.prod(n)), len(n)
    if k == "shock":
        steps = case["t_end"] * case["nx"] * 2.4 / _cfl(case)
    else:
        steps = case.get("steps", 1) * (case["count"] if k == "ensemble" else 1)
    b, f = 20.0 * es, 600.0 * ndim + 100.0
    if case.get("scheme") == "kt":
        b, f = 1.5 * b, 1.2 * f
    if case.get("ctu"):
        f *= 1.6
    if k in ("disc", "gradient"):
        b += 2.0 * es
    if case.get("grav", 0.0) > 0.0:
        b += 10.0 * es
    if k == "gradient":
        b, f = 3.5 * b, 4.0 * f
    return dict(bytes=b * cells * steps, flops=f * cells * steps)


# ---------------------------------------------------- the method in plain torch, 64 bits
# States are lists of ten tensors.  A direction's local frame moves its normal axis to the x
# slot: local slot k holds component FRAME[d][k].
FRAME = ((0, 1, 2, 3, 4, 5, 6, 7, 8, 9), (0, 2, 1, 3, 7, 5, 8, 4, 6, 9), (0, 3, 1, 2, 9, 6, 8, 4, 5, 7))
FLIP = ((1, 5, 6), (2, 5, 8), (3, 6, 8))


def _cons(W):
    r, u, v, w = W[0], W[1], W[2], W[3]
    U = [r, r * u, r * v, r * w, W[4] + r * u * u, W[5] + r * u * v, W[6] + r * u * w, W[7] + r * v * v,
         W[8] + r * v * w, W[9] + r * w * w]
    return torch.stack(U) if isinstance(W, torch.Tensor) else U


def _prim(U):
    r = U[0]
    u, v, w = U[1] / r, U[2] / r, U[3] / r
    return [r, u, v, w, U[4] - U[1] * u, U[5] - U[1] * v, U[6] - U[1] * w, U[7] - U[2] * v, U[8] - U[2] * w,
            U[9] - U[3] * w]


def _good(W):
    a, b, c, d, e, f = W[4:]
    return (W[0] > 0) & (a > 0) & (a * d - b * b > 0) & (a * (d * f - e * e) - b * (b * f - e * c) + c * (b * e - d * c) > 0)


def _project(w, d):
    """Characteristic amplitudes L d on the eigenvectors of the state w (local frame)."""
    r, xx, xy, xz, yy, yz, zz = w[0], w[4], w[5], w[6], w[7], w[8], w[9]
    cs = torch.sqrt(xx / r)
    cf = math.sqrt(3.0) * cs
    a, b, e = xy / xx, xz / xx, d[4] / (3.0 * xx)
    qv, rv = (d[2] - a * d[1]) / (2 * cs), (d[5] - a * d[4]) / (2 * xx)
    qw, rw = (d[3] - b * d[1]) / (2 * cs), (d[6] - b * d[4]) / (2 * xx)
    t = d[1] / (2 * cf)
    return [e / 2 - t, rv - qv, rw - qw, d[0] - r * e, d[7] - 2 * a * d[5] + (4 * a * xy - yy) * e,
            d[8] - b * d[5] - a * d[6] + (4 * a * xz - yz) * e, d[9] - 2 * b * d[6] + (4 * b * xz - zz) * e, rv + qv,
            rw + qw, e / 2 + t]


def _back(w, c):
    """R c, the primitive vector of the amplitudes c."""
    r, xx, xy, xz, yy, yz, zz = w[0], w[4], w[5], w[6], w[7], w[8], w[9]
    cs = torch.sqrt(xx / r)
    cf = math.sqrt(3.0) * cs
    a, b = xy / xx, xz / xx
    A, B, C, D, E, F = c[9] + c[0], (c[9] - c[0]) * cf, c[7] + c[1], (c[7] - c[1]) * cs, c[8] + c[2], (c[8] - c[2]) * cs
    return [r * A + c[3], B, a * B + D, b * B + F, 3 * xx * A, 3 * xy * A + xx * C, 3 * xz * A + xx * E,
            (yy + 2 * a * xy) * A + 2 * xy * C + c[4], (yz + 2 * a * xz) * A + xz * C + xy * E + c[5],
            (zz + 2 * b * xz) * A + 2 * xz * E + c[6]]


def _speeds(w):
    cs = torch.sqrt(w[4] / w[0])
    cf = math.sqrt(3.0) * cs
    z = torch.zeros_like(cs)
    return [-cf, -cs, -cs, z, z, z, z, cs, cs, cf]


def _mc(l, r):
    m = torch.minimum(torch.minimum(2 * l.abs(), 2 * r.abs()), 0.5 * (l + r).abs())
    return torch.where(l * r > 0, torch.sign(l) * m, torch.zeros_like(m))


def _check(w0, lo, hi):
    ok = (lo[0] > 0) & (hi[0] > 0) & (lo[4] > 0) & (hi[4] > 0)
    return [torch.where(ok, x, w) for x, w in zip(lo, w0)], [torch.where(ok, x, w) for x, w in zip(hi, w0)]


def _faces(wm, w0, wp, nu, scheme, X):
    """Face states (lower, upper) of the cells w0."""
    if scheme == "kt":
        s = [_mc(b - a, c - b) for a, b, c in zip(wm, w0, wp)]
        return _check(w0, [w - 0.5 * x for w, x in zip(w0, s)], [w + 0.5 * x for w, x in zip(w0, s)])
    cl, cr = _project(w0, [b - a for a, b in zip(wm, w0)]), _project(w0, [c - b for b, c in zip(w0, wp)])
    m = [_mc(l, r) for l, r in zip(cl, cr)]
    del cl, cr
    dw, g = _back(w0, m), _back(w0, [s * x for s, x in zip(_speeds(w0), m)])
    mid = [w - nu * (w0[1] * x + y) for w, x, y in zip(w0, dw, g)]
    if X is not None:
        mid = [a + x for a, x in zip(mid, X)]
    return _check(w0, [a - 0.5 * x for a, x in zip(mid, dw)], [a + 0.5 * x for a, x in zip(mid, dw)])


def _transverse(wm, w0, wp, nu):
    cl, cr = _project(w0, [b - a for a, b in zip(wm, w0)]), _project(w0, [c - b for b, c in zip(w0, wp)])
    return _back(w0, [-nu * (w0[1] + s) * torch.where(w0[1] + s > 0, l, r) for s, l, r in zip(_speeds(w0), cl, cr)])


def _pi(u, p):
    """The part of the normal flux that depends on (u_i, P_in) alone."""
    return [torch.zeros_like(u[0]), p[0], p[1], p[2], 2 * p[0] * u[0], p[1] * u[0] + p[0] * u[1], p[2] * u[0] + p[0] * u[2],
            2 * p[1] * u[1], p[1] * u[2] + p[2] * u[1], 2 * p[2] * u[2]]


def _flux(l, r, scheme):
    Ul, Ur, Pl, Pr = _cons(l), _cons(r), _pi(l[1:4], l[4:7]), _pi(r[1:4], r[4:7])
    Fl, Fr = [l[1] * u + p for u, p in zip(Ul, Pl)], [r[1] * u + p for u, p in zip(Ur, Pr)]
    cl, cr = torch.sqrt(3.0 * l[4] / l[0]), torch.sqrt(3.0 * r[4] / r[0])
    if scheme == "kt":
        a = torch.maximum(l[1].abs() + cl, r[1].abs() + cr)
        return [0.5 * (f + g) - 0.5 * a * (v - u) for f, g, u, v in zip(Fl, Fr, Ul, Ur)]
    SL, SR = torch.minimum(l[1] - cl, r[1] - cr), torch.maximum(l[1] + cl, r[1] + cr)
    inv = 1.0 / (SR - SL)
    F = [torch.where(SL >= 0, f, torch.where(SR <= 0, g, (SR * f - SL * g + SL * SR * (v - u)) * inv))
         for f, g, u, v in zip(Fl, Fr, Ul, Ur)]
    if scheme != "hllc":
        return F
    CL, CR = l[0] * (SL - l[1]), r[0] * (SR - r[1])
    us = [(CR * b - CL * a - (q - p)) / (CR - CL) for a, b, p, q in zip(l[1:4], r[1:4], l[4:7], r[4:7])]
    ps = [p + CL * (s - a) for p, s, a in zip(l[4:7], us, l[1:4])]
    SM, Ps = us[0], _pi(us, ps)
    inside = (SL < SM) & (SM < SR) & (SL < 0) & (SR > 0)
    out = []
    for f, u, v, p, q, s in zip(F, Ul, Ur, Pl, Pr, Ps):
        gl = (SM * (SL - l[1]) * u - SM * p + SL * s) / (SL - SM)
        gr = (SM * (SR - r[1]) * v - SM * q + SR * s) / (SR - SM)
        out.append(torch.where(inside, torch.where(SM >= 0, gl, gr), f))
    return out


class _Plain:
    """Uniform grids [nz, ny, nx]."""

    def __init__(self, n, dx, bc, cfl, scheme="hll", ctu=False, acc=None, grav=0.0, axes=None):
        self.n, self.dx, self.bc, self.cfl, self.scheme, self.ctu = n, dx, bc, cfl, scheme, ctu
        self.acc, self.grav, self.prev, self.dt_prev = acc, grav, None, None
        self.axis = [-(1 + d) for d in range(len(n))]  # direction d is the d-th last axis

    def ghost(self, W, d, flip=True):
        """W with two ghost cells on each side along direction d."""
        n, (lo, hi) = self.n[d], self.bc[d]
        idx, sgn = [], []
        for i in range(-2, n + 2):
            s, j = 1.0, i
            if i < 0:
                j = i + n if lo == PER else 0 if lo == OUT else -1 - i
                s = -1.0 if lo == REF else 1.0
            elif i >= n:
                j = i - n if hi == PER else n - 1 if hi == OUT else 2 * n - 1 - i
                s = -1.0 if hi == REF else 1.0
            idx.append(min(max(j, 0), n - 1))
            sgn.append(s)
        idx = torch.tensor(idx, device=W[0].device)
        G = [x.index_select(x.dim() + self.axis[d], idx) for x in W]
        if flip and -1.0 in sgn:
            s = torch.tensor(sgn, device=W[0].device, dtype=W[0].dtype).reshape([-1] + [1] * d)
            G = [x * s if k in FLIP[d] else x for k, x in enumerate(G)]
        return G

    def speed(self, W):
        s = [(W[1 + d].abs() + torch.sqrt(3.0 * W[(4, 7, 9)[d]] / W[0])) / self.dx[d] for d in range(len(self.n))]
        if self.ctu:
            return torch.stack(s).amax(0)
        return sum(s)

    def divergence(self, U, dt, tag=None):
        """sum_d (F_{i+1/2} - F_{i-1/2}) / dx_d; faces of tagged cells take first-order states."""
        W, nd, T, total = _prim(U), len(self.n), [], None
        if self.ctu and nd > 1:
            for d in range(nd):
                G = [self.ghost(W, d)[k] for k in FRAME[d]]
                a, n = G[0].dim() + self.axis[d], self.n[d]
                t = _transverse(*[[x.narrow(a, o, n) for x in G] for o in (1, 2, 3)], 0.5 * dt / self.dx[d])
                T.append([t[FRAME[d].index(k)] for k in range(10)])
        for d in range(nd):
            n = self.n[d]
            G = self.ghost(W, d)
            G = [G[k] for k in FRAME[d]]
            a = G[0].dim() + self.axis[d]
            cut = lambda v, o, m: [x.narrow(a, o, m) for x in v]
            X = None
            if T:
                X = self.ghost([sum(T[t][k] for t in range(nd) if t != d) for k in range(10)], d)
                X = cut([X[k] for k in FRAME[d]], 1, n + 2)
            w0 = cut(G, 1, n + 2)
            lo, hi = _faces(cut(G, 0, n + 2), w0, cut(G, 2, n + 2), 0.5 * dt / self.dx[d], self.scheme, X)
            del G, X
            if tag is not None:
                t = self.ghost([tag], d, flip=False)[0]
                tm, t0, tp = t.narrow(a, 0, n + 2), t.narrow(a, 1, n + 2), t.narrow(a, 2, n + 2)
                lo = [torch.where(t0 | tm, w, x) for w, x in zip(w0, lo)]
                hi = [torch.where(t0 | tp, w, x) for w, x in zip(w0, hi)]
            wl, wr = cut(hi, 0, n + 1), cut(lo, 1, n + 1)
            F = _flux(wl, wr, self.scheme)
            if tag is not None and self.scheme == "hllc":
                first = t.narrow(a, 1, n + 1) | t.narrow(a, 2, n + 1)
                F = [torch.where(first, f, g) for f, g in zip(_flux(wl, wr, "hll"), F)]
            del lo, hi, wl, wr, w0
            div = [(F[k].narrow(a, 1, n) - F[k].narrow(a, 0, n)) / self.dx[d] for k in range(10)]
            div = [div[FRAME[d].index(k)] for k in range(10)]
            del F
            total = div if total is None else [x + y for x, y in zip(total, div)]
        return total

    def gravity(self, U, dt):
        """m += dt rho a, E += dt (mbar a^T + a mbar^T) with the step's acceleration."""
        if self.acc is None and self.step_acc is None:
            return U
        a = self.step_acc if self.step_acc is not None else self.acc
        mn = [U[1 + i] + dt * U[0] * a[i] for i in range(3)]
        mb = [0.5 * (U[1 + i] + mn[i]) for i in range(3)]
        pairs = ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))
        return [U[0]] + mn + [U[4 + k] + dt * (mb[i] * a[j] + a[i] * mb[j]) for k, (i, j) in enumerate(pairs)]

    def self_gravity(self, rho, dt):
        """a^n of the periodic 3-point Poisson solve, interpolated forward in time."""
        nd = len(self.n)
        k2 = 0.0
        for d in range(nd):
            n = self.n[d]
            k = torch.arange(n // 2 + 1 if d == 0 else n, device=rho.device, dtype=torch.float64)
            k2 = k2 + ((2.0 * torch.sin(math.pi * k / n) / self.dx[d]) ** 2).reshape([-1] + [1] * d)
        hat = torch.fft.rfftn(rho)
        phi = torch.fft.irfftn(torch.where(k2 > 0, -4.0 * math.pi * self.grav / torch.where(k2 > 0, k2, 1.0), 0.0) * hat,
                               s=rho.shape)
        a = [-(torch.roll(phi, -1, self.axis[d]) - torch.roll(phi, 1, self.axis[d])) / (2.0 * self.dx[d])
             if d < nd else torch.zeros_like(phi) for d in range(3)]
        out = a if self.prev is None else [x + dt / (2.0 * self.dt_prev) * (x - y) for x, y in zip(a, self.prev)]
        self.prev, self.dt_prev = a, dt
        return out

    def step(self, U, dt):
        self.step_acc = self.self_gravity(U[0], dt) if self.grav > 0.0 else None
        if self.scheme == "kt":
            U1 = [u - dt * x for u, x in zip(U, self.divergence(U, dt))]
            V = [0.5 * (u + (v - dt * x)) for u, v, x in zip(U, U1, self.divergence(U1, dt))]
            return self.gravity(V, dt)
        tag = None
        for _ in range(5):  # the step, then up to four passes with first-order faces
            V = self.gravity([u - dt * x for u, x in zip(U, self.divergence(U, dt, tag))], dt)
            with torch.no_grad():
                bad = ~_good(_prim(V))
                if tag is not None:
                    bad = bad & ~tag
                if not bool(bad.any()):
                    break
                tag = bad if tag is None else tag | bad
        return V

    def dt(self, U):
        return float(self.cfl / self.speed(_prim(U)).max())


def _plain(case):
    n, lo, hi, bc = _geometry(case)
    dx = [(b - a) / m for a, b, m in zip(lo, hi, n)]
    acc = None
    if case["kind"] in ("disc", "gradient"):
        phi = _disc_potential(case["nx"])[0]
        acc = [-(phi[1:-1, 2:] - phi[1:-1, :-2]) / (2 * dx[0]), -(phi[2:, 1:-1] - phi[:-2, 1:-1]) / (2 * dx[1])]
        acc = [a[None] for a in acc] + [torch.zeros_like(acc[0])[None]]
        if case["prec"] == "f32":  # the acceleration is stored in the state's precision
            acc = [a.float().double() for a in acc]
    return _Plain(n, dx, bc, _cfl(case), case.get("scheme", "hll"), bool(case.get("ctu")), acc, case.get("grav", 0.0))


class _Rows(_Plain):
    """Independent 1D tubes as rows [tubes, nmax] of their own lengths, outflow at both ends of
    each.  Cells past a row's end hold copies and are neither read nor checked."""

    def __init__(self, length, nmax, cfl):
        super().__init__((nmax,), (None,), ((OUT, OUT),), cfl)
        self.dx = (1.0 / length.double()[:, None],)
        self.idx = torch.minimum(torch.arange(-2, nmax + 2, device=length.device).clamp(min=0)[None, :], length[:, None] - 1)
        self.live = torch.arange(nmax, device=length.device)[None, :] < length[:, None]

    def ghost(self, W, d, flip=True):
        return [x.gather(1, self.idx) for x in W]

    def step(self, U, dt):
        return [torch.where(self.live, v, u[:, :1]) for u, v in zip(U, super().step(U, dt))]


def _exact_tubes(case, seed):
    """The tubes in groups of similar length; every tube has its own time step."""
    length, WL, WR = _tube_states(seed, case["count"], case["nmin"], case["nmax"])
    out = np.zeros((10, int(length.sum())))
    off = np.concatenate([[0], np.cumsum(length)])
    dtype = np.float32 if case["prec"] == "f32" else np.float64
    order = np.argsort(length, kind="stable")
    for ks in np.array_split(order, max(1, -(-len(order) // 512))):
        n = torch.tensor(length[ks].astype(np.int64), device="cuda")
        nmax = int(n.max())
        a, b = (torch.tensor(X[ks].astype(dtype).astype(np.float64), device="cuda") for X in (WL, WR))
        left = (torch.arange(nmax, device="cuda", dtype=torch.float64)[None, :] + 0.5) / n[:, None] < 0.5
        U = _cons([torch.where(left, a[:, k:k + 1], b[:, k:k + 1]) for k in range(10)])
        g = _Rows(n, nmax, _cfl(case))
        t = torch.zeros((len(ks), 1), device="cuda", dtype=torch.float64)
        while bool((t < case["t_end"]).any()):
            smax = torch.where(g.live, g.speed(_prim(U)), 0.0).amax(1, keepdim=True)
            dt = torch.minimum(g.cfl / smax, case["t_end"] - t)
            U, t = g.step(U, dt), t + dt
        U = torch.stack(U).cpu().numpy()
        for i, k in enumerate(ks):
            out[:, off[k]:off[k + 1]] = U[:, i, :length[k]]
    return out


def exact(case, seed):
    k = case["kind"]
    if case.get("scheme") == "roe":
        return None
    if k == "tubes":
        return _exact_tubes(case, seed)
    g = _plain(case)
    if k == "ensemble":
        outs = []
        for U in _ensemble_states(case, seed):
            U = list(U.double().unbind(0))
            for _ in range(case["steps"]):
                U = g.step(U, g.dt(U))
            outs.append(torch.stack(U).cpu().numpy())
        return outs
    W = _initial(case, seed).double()
    if k == "one":
        U = list(_cons(W).to(DTYPE[case["prec"]]).double().unbind(0))
        dt = g.dt(U)
        return dict(U=torch.stack(g.step(U, dt)), dt=dt)
    if k == "gradient":
        Us, dts, U = [], [], _cons(W)
        with torch.no_grad():
            for _ in range(case["steps"]):
                Us.append(U)
                dts.append(g.dt(list(U.unbind(0))))
                U = torch.stack(g.step(list(U.unbind(0)), dts[-1]))
        lam = _cotangent(case, seed)
        for V, dt in zip(reversed(Us), reversed(dts)):
            V = V.detach().requires_grad_(True)
            lam, = torch.autograd.grad(torch.stack(g.step(list(V.unbind(0)), dt)), V, lam)
        W = W.detach().requires_grad_(True)
        grad, = torch.autograd.grad(_cons(W), W, lam)
        return dict(U=U, grad=grad)
    U, t = _cons(list(W.unbind(0))), 0.0
    if k == "shock":
        while t < case["t_end"]:
            dt = min(g.dt(U), case["t_end"] - t)
            last = dt == case["t_end"] - t
            U, t = g.step(U, dt), case["t_end"] if last else t + dt
    else:
        for _ in range(case["steps"]):
            dt = g.dt(U)
            U, t = g.step(U, dt), t + dt
    return dict(U=torch.stack(U), t=t)
