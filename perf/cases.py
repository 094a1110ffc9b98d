"""Performance cases: the calls a program makes of this library, over the range of sizes, types and options.

`listed()` gives the fixed cases, `draw(rng)` one more of the same ranges.  A case is a dict of plain values;
`prepare` makes its inputs on the GPU from a seed and the handle a program keeps, `run` is one pass through the
public calls, `work` the bytes and operations a pass cannot do without, and `exact` the result in 64 bits by plain
torch (cyclic reduction of every line system, no code of the library).

Inputs are the workloads of the repository: the ring of the paper's Section 3.1 (a circular field, a hot arc, no
flux through the walls) and seeded random fields (b along the contours of a random stream function, or of a random
divergence-free field in three dimensions, with Gaussian blobs of temperature on a periodic box).  Timesteps are
given in units of the explicit limit min(dx, dy)^2 / (2 chi).
"""
import math

import numpy as np
import torch

import paper_1008_0861_gb300 as A

CHI = 0.05
L2_BYTES = 126 << 20

_LIMITERS = {"vanleer": A.ANISO_LIM_VANLEER, "minmod": A.ANISO_LIM_MINMOD, "mc": A.ANISO_LIM_MC}
_ORDERS = {"xy": A.ANISO_ORDER_XY, "yx": A.ANISO_ORDER_YX, "alternate": A.ANISO_ORDER_ALTERNATE}
_SCHEMES = {"2step": A.ANISO_SCHEME_2STEP, "4step": A.ANISO_SCHEME_4STEP}


# ------------------------------------------------------------------ cases

def _case(**kw):
    """A case with every key: what it does not name has the library's default."""
    c = {"call": "step", "problem": "random", "nx": 0, "ny": 0, "nz": 0, "grids": 1, "prec": "fp32", "field_fp16": False,
         "compensated": False, "limiter": "vanleer", "order": "xy", "scheme": "2step", "kmax": 8, "cfl": 100.0, "steps": 1}
    c.update(kw)
    return c


def listed():
    return [
        # the paper's ring test as printed: 50 x 50 cells in double precision (the default), 250 steps in one call;
        # what a first-time user runs, and the smallest grid that is stepped for long
        _case(name="ring50_fp64", problem="ring", nx=50, ny=50, prec="fp64", cfl=10.0, steps=250),
        # the ring at the paper's resolution to t = 20 (52 steps at ncfl 1000), then the sum and the extrema of T,
        # as a program does that follows conservation and the lowest temperature
        _case(name="ring512_fp64_monitor", call="monitor", problem="ring", nx=512, ny=512, prec="fp64", cfl=500.0, steps=52),
        # an ordinary single-precision grid, stepped many times a call
        _case(name="random1024_fp32", nx=1024, ny=1024, steps=20),
        # one large grid (the second workload of the benchmark) in single and in double precision
        _case(name="random4096_fp32", nx=4096, ny=4096, steps=4),
        _case(name="random4096_fp64", nx=4096, ny=4096, prec="fp64", steps=2),
        # sides that are no multiple of a vector: grids whose size comes from a geometry
        _case(name="ragged1001x777_fp32", nx=1001, ny=777, steps=10),
        # the headline: 512 independent grids of uneven sizes, fields and timesteps advanced together
        _case(name="batch512_fp32", call="batch", nx=1024, ny=1024, grids=512, cfl=1000.0, steps=4),
        # sharp-gradient stress: copies of a large ring, each with its own timestep
        _case(name="ring8192_batch_fp32", call="batch", problem="stress", nx=8192, ny=8192, grids=8, cfl=30000.0, steps=2),
        # the largest grid: compensated state for long runs, half-precision coefficients
        _case(name="compensated16384", nx=16384, ny=16384, field_fp16=True, compensated=True, kmax=32, cfl=1000.0, steps=2),
        # the three-dimensional split
        _case(name="random3d_256_fp32", call="step3d", nx=256, ny=256, nz=256, kmax=3, cfl=10.0, steps=4),
        # conduction inside a flow code: the field moves, so every call sets it anew and takes one step, with the
        # diffusivity following T^(5/2) (Section 3.3)
        _case(name="coupled1024_fp32", call="coupled", nx=1024, ny=1024, cfl=10.0),
        # a small step from code that may not allocate device memory
        _case(name="noalloc96x64_fp32", call="noalloc", nx=96, ny=64),
    ]


def _side(rng, lo, hi, multiple=1):
    """A length spread evenly over the logarithm of [lo, hi], rounded down to a multiple."""
    n = int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))
    return max(lo, min(hi, n // multiple * multiple))


def _other_side(rng, n, lo, hi, multiple=1):
    """The other length of a grid at most twice as long or wide as it is wide or long."""
    return _side(rng, max(lo, n // 2 // multiple * multiple), min(hi, 2 * n), multiple)


def draw(rng):
    call = rng.choice(["step", "step", "step", "monitor", "batch", "compensated", "step3d", "coupled", "noalloc"])
    bc = rng.choice(["ring", "random"])
    prec = rng.choice(["fp32", "fp32", "fp64"])
    if call == "step":
        # any size of a single grid: sides of any number, of whole vectors, of whole tiles
        top = 4096 if prec == "fp32" else 2048
        m = rng.choice([1, 4, 32])
        nx = _side(rng, 32, top, m)
        ny = _other_side(rng, nx, 32, top, m)
        steps = max(2, min(100, int(2e7 / (nx * ny))) // 2 * 2)
        option = rng.choice(["", "", "limiter", "order", "scheme", "field"])
        return _case(problem=bc, nx=nx, ny=ny, prec=prec, steps=steps, cfl=round(10.0 ** rng.uniform(1, 2), 2),
                     limiter=rng.choice(["minmod", "mc"]) if option == "limiter" else "vanleer",
                     order=rng.choice(["yx", "alternate"]) if option == "order" else "xy",
                     scheme="4step" if option == "scheme" else "2step",
                     field_fp16=option == "field" and prec == "fp32")
    if call == "monitor":
        n = _side(rng, 50, 1024)
        return _case(call="monitor", problem="ring", nx=n, ny=n, prec=prec, cfl=round(10.0 ** rng.uniform(1, 2.7), 2),
                     steps=max(2, min(52, int(1e7 / (n * n)))))
    if call == "batch":
        top = 32 * rng.randint(4, 32)
        grids = max(2, min(256, int(2e8 / (top * top))))
        return _case(call="batch", nx=top, ny=top, grids=rng.randint(max(2, grids // 4), grids), prec=prec if top <= 512 else "fp32",
                     cfl=round(10.0 ** rng.uniform(1.3, 3), 2), steps=rng.randint(2, 6))
    if call == "compensated":
        # (powers of two are what large runs take; other sides are as welcome)
        n = rng.choice([1024, 2048, 4096, 8192, _side(rng, 64, 2048), _side(rng, 64, 2048)])
        return _case(problem=bc, nx=n, ny=n, field_fp16=rng.random() < 0.5, compensated=True,
                     cfl=round(10.0 ** rng.uniform(1, 3), 2), steps=rng.randint(2, 4))
    if call == "step3d":
        nx, ny, nz = (_side(rng, 32, 320, 4) for _ in range(3))
        return _case(call="step3d", nx=nx, ny=ny, nz=nz, kmax=3, cfl=round(rng.uniform(2, 10), 2), steps=rng.randint(2, 6),
                     field_fp16=rng.random() < 0.25, scheme=rng.choice(["2step", "2step", "2step", "4step"]))
    if call == "coupled":
        nx = _side(rng, 128, 2048, 4)
        return _case(call="coupled", nx=nx, ny=_other_side(rng, nx, 128, 2048, 4), cfl=round(rng.uniform(5, 10), 2))
    nx = _side(rng, 16, 1000)
    ny = _other_side(rng, nx, 16, 1000)
    while nx * ny > (1 << 20 if prec == "fp32" else 1 << 19):
        ny //= 2
    return _case(call="noalloc", problem=bc, nx=nx, ny=ny, prec=prec, cfl=round(10.0 ** rng.uniform(1, 2), 2), steps=rng.randint(1, 4))


# ----------------------------------------------------------------- inputs

def _grids(case):
    """(nx, ny, chi, dt / explicit limit) of every grid of the case."""
    if case["call"] != "batch":
        return [(case["nx"], case["ny"], CHI, case["cfl"])]
    if case["problem"] == "stress":
        # one timestep a copy, spread over the logarithm from 10 times the explicit limit
        g = case["grids"]
        return [(case["nx"], case["ny"], 0.01, 10.0 * (case["cfl"] / 10.0) ** (k / max(1, g - 1))) for k in range(g)]
    # uneven sizes in multiples of 32, diffusivities over two decades, timesteps from 10 times the limit
    rng = np.random.RandomState(case["grids"])
    out = []
    for _ in range(case["grids"]):
        u = rng.rand(4)
        out.append((32 * (2 + int(u[0] * (case["nx"] // 32 - 1))), 32 * (2 + int(u[1] * (case["ny"] // 32 - 1))),
                    10.0 ** (-3 + 2 * u[2]), 10.0 * (case["cfl"] / 10.0) ** u[3]))
    return out


def _spacing(case, nx, ny):
    side = 2.0 if case["problem"] in ("ring", "stress") else 1.0
    return side / nx, side / ny


def _dt(case, dx, dy, chi, cfl):
    return cfl * min(dx, dy) ** 2 / (2.0 * chi)


def _dtype(case):
    return torch.float64 if case["prec"] == "fp64" else torch.float32


def _centres(n, dtype):
    return (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5).div_(n).to(dtype)


def _periodic_blob(x, c, w):
    d = x[None, :] - c[:, None]
    d = d - torch.round(d)
    return torch.exp(-(d * d) / (2.0 * w * w)[:, None])


def _tensor(a, dtype):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dtype)


def _random2(rng, nx, ny, kmax, dtype):
    """b along the contours of a random stream function, T = 1 + 16 Gaussians."""
    k = np.arange(-kmax, kmax + 1)
    kx, ky = np.meshgrid(k, k, indexing="ij")
    k2 = kx * kx + ky * ky
    amp = np.where((k2 >= 1) & (k2 <= kmax * kmax), rng.randn(*k2.shape) / np.maximum(k2, 1), 0.0)
    w = amp * np.exp(2j * math.pi * rng.rand(*k2.shape))
    x, y = (np.arange(nx) + 0.5) / nx, (np.arange(ny) + 0.5) / ny
    ex, ey = np.exp(2j * math.pi * np.outer(k, x)), np.exp(2j * math.pi * np.outer(y, k))
    right = _tensor(np.concatenate([ex.imag, ex.real]), dtype)
    grad = []
    for c in (-kx * w, -ky * w):  # the gradient's components, up to 2 pi
        left = ey @ c.T
        grad.append(_tensor(np.concatenate([left.real, left.imag], axis=1), dtype) @ right)
    gx, gy = grad
    mag = torch.hypot(gx, gy)
    small = mag < 1e-9
    mag = torch.where(small, 1.0, mag)
    bx = torch.where(small, 1.0, -gy / mag)
    by = torch.where(small, 0.0, gx / mag)
    cx, cy, a, wd = (_tensor(v, dtype) for v in rng.rand(4, 16))
    wd = 0.01 + 0.04 * wd
    gx = _periodic_blob(_centres(nx, dtype), cx, wd) * (0.5 + 1.5 * a)[:, None]
    return bx, by, 1.0 + _periodic_blob(_centres(ny, dtype), cy, wd).T @ gx


def _ring2(rng, nx, ny, hot, cold, dtype):
    """The ring of Section 3.1, its hot arc at an angle of its own."""
    x, y = 2.0 * _centres(nx, torch.float64) - 1.0, 2.0 * _centres(ny, torch.float64) - 1.0
    r = torch.hypot(x[None, :], y[:, None])
    turn = 2.0 * math.pi * rng.rand()
    theta = torch.remainder(torch.atan2(y[:, None], x[None, :]) - turn, 2.0 * math.pi)
    arc = (r > 0.5) & (r < 0.7) & ((theta - math.pi).abs() < math.pi / 12.0)
    T = torch.where(arc, hot, cold).to(torch.float64)
    inside = (r <= 1.0) & (r > 0.0)
    rs = torch.where(inside, r, 1.0)
    bx = torch.where(inside, -y[:, None] / rs, 0.0)
    by = torch.where(inside, x[None, :] / rs, 0.0)
    return bx.to(dtype).contiguous(), by.to(dtype).contiguous(), T.to(dtype)


def _random3(rng, nx, ny, nz, kmax, dtype):
    """b = B / |B|, B = z + curl of a random vector potential, T = 1 + 16 Gaussians."""
    k = np.arange(-kmax, kmax + 1)
    kz, ky, kx = np.meshgrid(k, k, k, indexing="ij")
    k2 = kx * kx + ky * ky + kz * kz
    a = rng.randn(3, *k2.shape) * np.where((k2 >= 1) & (k2 <= kmax * kmax), 1.0 / np.maximum(k2, 1), 0.0)
    w = np.exp(2j * math.pi * rng.rand(*k2.shape))
    curl = np.stack([ky * a[2] - kz * a[1], kz * a[0] - kx * a[2], kx * a[1] - ky * a[0]])
    C = _tensor(-2.0 * math.pi * curl * w, torch.complex64)
    e = [_tensor(np.exp(2j * math.pi * np.outer((np.arange(n) + 0.5) / n, k)), torch.complex64) for n in (nx, ny, nz)]
    B = []
    for c in range(3):
        f = torch.einsum("zyx,ix->zyi", C[c], e[0])
        f = torch.einsum("zyi,jy->zji", f, e[1])
        B.append(torch.einsum("zji,kz->kji", f, e[2]).imag.to(dtype))
    B[2] = B[2] + 1.0
    mag = torch.sqrt(B[0] ** 2 + B[1] ** 2 + B[2] ** 2).clamp_min(1e-9)
    cx, cy, cz, a, wd = (_tensor(v, dtype) for v in rng.rand(5, 16))
    wd = 0.02 + 0.06 * wd
    gx = _periodic_blob(_centres(nx, dtype), cx, wd) * (0.5 + 1.5 * a)[:, None]
    T = 1.0 + torch.einsum("gz,gy,gx->zyx", _periodic_blob(_centres(nz, dtype), cz, wd),
                           _periodic_blob(_centres(ny, dtype), cy, wd), gx)
    return [(v / mag).contiguous() for v in B], T.contiguous()


def _inputs(case, seed):
    """The field and the temperature of every grid of the case, one at a time."""
    dtype = _dtype(case)
    for q, (nx, ny, _, _) in enumerate(_grids(case)):
        rng = np.random.RandomState((int(seed) * 1000 + q) % (1 << 32))
        if case["call"] == "step3d":
            yield _random3(rng, nx, ny, case["nz"], case["kmax"], dtype)
        elif case["problem"] == "random":
            yield _random2(rng, nx, ny, case["kmax"], dtype)
        elif case["problem"] == "ring":
            yield _ring2(rng, nx, ny, 12.0, 10.0, dtype)
        else:
            yield _ring2(rng, nx, ny, 10.0, 0.1, dtype)


# ---------------------------------------------------------------- running

class _State:
    """What a program keeps: its handles, its arrays and the arguments of its calls."""

    def __init__(self, case):
        self.case, self.handles, self.batch, self.handle3 = case, [], None, None

    def __del__(self):
        A.aniso_batch_destroy(self.batch)
        for h in self.handles:
            A.aniso_destroy(h)
        A.aniso3_destroy(self.handle3)


def _bc(case):
    return A.ANISO_BC_PERIODIC if case["problem"] == "random" else A.ANISO_BC_ZEROFLUX


def _handle(case, nx, ny, chi):
    dx, dy = _spacing(case, nx, ny)
    h = A.aniso_create(nx, ny, dx, dy, chi, 0.0, _bc(case))
    A.aniso_set_option(h, A.ANISO_OPT_PRECISION, A.ANISO_PREC_FP64 if case["prec"] == "fp64" else A.ANISO_PREC_FP32)
    A.aniso_set_option(h, A.ANISO_OPT_FIELD_FP16, int(case["field_fp16"]))
    A.aniso_set_option(h, A.ANISO_OPT_KAHAN, int(case["compensated"]))
    A.aniso_set_option(h, A.ANISO_OPT_LIMITER, _LIMITERS[case["limiter"]])
    A.aniso_set_option(h, A.ANISO_OPT_ORDER, _ORDERS[case["order"]])
    A.aniso_set_option(h, A.ANISO_OPT_SCHEME, _SCHEMES[case["scheme"]])
    return h


def prepare(case, seed):
    s = _State(case)
    grids = _grids(case)
    if case["call"] == "step3d":
        (b, s.T), = _inputs(case, seed)
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        s.handle3 = A.aniso3_create(nx, ny, nz, 1.0 / nx, 1.0 / ny, 1.0 / nz, CHI, 0.0, A.ANISO_BC_PERIODIC)
        A.aniso3_set_option(s.handle3, A.ANISO_OPT_PRECISION, A.ANISO_PREC_FP32)
        A.aniso3_set_option(s.handle3, A.ANISO_OPT_FIELD_FP16, int(case["field_fp16"]))
        A.aniso3_set_option(s.handle3, A.ANISO_OPT_SCHEME, _SCHEMES[case["scheme"]])
        A.aniso3_set_field(s.handle3, *b)
        s.dt = case["cfl"] / max(nx, ny, nz) ** 2 / (2.0 * CHI)
        torch.cuda.synchronize()  # the field's arrays may go
        return s
    s.dts = [_dt(case, *_spacing(case, nx, ny), chi, cfl) for nx, ny, chi, cfl in grids]
    if case["call"] == "batch":
        # all temperatures in one array, each grid's from a boundary of 256 bytes
        at = np.cumsum([0] + [-(-nx * ny // 64) * 64 for nx, ny, _, _ in grids])
        s.T = torch.zeros(int(at[-1]), dtype=_dtype(case), device="cuda")
        s.Ts = [s.T[int(o):int(o) + nx * ny].view(ny, nx) for o, (nx, ny, _, _) in zip(at, grids)]
        for (nx, ny, chi, _), view, (bx, by, T) in zip(grids, s.Ts, _inputs(case, seed)):
            view.copy_(T)
            s.handles.append(_handle(case, nx, ny, chi))
            A.aniso_set_field(s.handles[-1], bx, by)
        s.batch = A.aniso_batch_create(s.handles)
        s.steps = [case["steps"]] * len(grids)
        torch.cuda.synchronize()
        return s
    (s.bx, s.by, s.T), = _inputs(case, seed)
    if case["call"] != "noalloc":
        nx, ny, chi, _ = grids[0]
        s.handles.append(_handle(case, nx, ny, chi))
        A.aniso_set_field(s.handles[0], s.bx, s.by)
        if case["call"] == "coupled":
            A.aniso_set_nonlinear(s.handles[0], 2.5, 1.0)
        else:
            torch.cuda.synchronize()
            s.bx = s.by = None
    return s


def run(s):
    case = s.case
    call = case["call"]
    if call == "batch":
        A.aniso_step_batched(s.batch, s.Ts, s.dts, s.steps)
        return s.T
    if call == "step3d":
        A.aniso3_step(s.handle3, s.T, s.dt, case["steps"])
        return s.T
    if call == "noalloc":
        dx, dy = _spacing(case, case["nx"], case["ny"])
        A.aniso_step_noalloc(case["nx"], case["ny"], dx, dy, CHI, 0.0, _bc(case),
                             A.ANISO_PREC_FP64 if case["prec"] == "fp64" else A.ANISO_PREC_FP32,
                             s.bx, s.by, s.T, s.dts[0], case["steps"])
        return s.T
    h = s.handles[0]
    if call == "coupled":
        A.aniso_set_field(h, s.bx, s.by)
    A.aniso_step(h, s.T, s.dts[0], case["steps"])
    if call == "monitor":
        total, low, high, bad = A.aniso_total(h, s.T)
        return {"T": s.T, "sum": total, "min": low, "max": high, "nonfinite": bad}
    return s.T


# ------------------------------------------------------------------- work

def work(case):
    """Per update: T read and written, the axis's coefficients read.  A grid that fits the GPU's cache with its
    coefficients is read and written once a pass, a larger one once an update."""
    e = 8 if case["prec"] == "fp64" else 4
    c = 2 if case["field_fp16"] else e
    state = 2 * e if case["compensated"] else e
    axes = 3 if case["call"] == "step3d" else 2
    cells = sum(nx * ny for nx, ny, _, _ in _grids(case)) * (case["nz"] if axes == 3 else 1)
    updates = axes * case["steps"] * (2 if case["scheme"] == "4step" else 1)
    once = cells * (state + axes * axes * c)
    if once <= L2_BYTES:
        moved = once + cells * state
    else:
        moved = updates * cells * (2 * state + axes * c)
    if case["call"] in ("coupled", "noalloc"):  # from the field itself: its two components
        moved = cells * (2 * state + 2 * e)
    if case["call"] == "monitor":
        moved += cells * state
    # a line update: two differences and a limited mean a cell and face, the flux, one elimination and one recovery
    return {"bytes": moved, "flops": updates * cells * (60 if axes == 3 else 45)}


# ------------------------------------------------------------------ exact

def _limit(lim, a, b):
    same = a * b > 0
    if lim == "vanleer":
        return torch.where(same, 2 * a * b / torch.where(same, a + b, 1.0), 0.0)
    if lim == "minmod":
        m = torch.minimum(a.abs(), b.abs())
    else:
        m = torch.minimum(2 * torch.minimum(a.abs(), b.abs()), 0.5 * (a + b).abs())
    return torch.where(same, torch.sign(a) * m, 0.0)


def _solve(off, rhs):
    """Lines along the last axis: (1 + off_p + off_{p-1}) x_p - off_p x_{p+1} - off_{p-1} x_{p-1} = rhs_p, indices
    around the line (off is 0 at a wall), by cyclic reduction until the equations have come apart."""
    low, up = -off.roll(1, -1), -off
    mid = 1.0 - low - up
    h, n = 1, off.shape[-1]
    while True:
        k1, k2 = low / mid.roll(h, -1), up / mid.roll(-h, -1)
        rhs = rhs - k1 * rhs.roll(h, -1) - k2 * rhs.roll(-h, -1)
        mid, low, up = (mid - k1 * up.roll(h, -1) - k2 * low.roll(-h, -1), -k1 * low.roll(h, -1), -k2 * up.roll(-h, -1))
        h = 2 * h % n if 2 * h % n else n
        if float(((low.abs() + up.abs()) / mid).max()) < 1e-18 or h == n:
            # (h a multiple of n: every equation holds its own unknown alone)
            return rhs / (mid + low + up)


def _update(T, lam, normal, across, lim, alpha=0.0):
    """One directional update of T along its last axis, indices around every axis.  `across`: (axis, mu,
    coefficient) of each transverse term."""
    scale = 1.0
    if alpha:  # the harmonic mean of the two cells' diffusivities
        chi = T.clamp_min(0) ** alpha
        nchi = chi.roll(-1, -1)
        scale = torch.where((chi > 0) & (nchi > 0), 2 * chi * nchi / (chi + nchi), 0.0)
    flux = lam * normal * scale * (T.roll(-1, -1) - T)
    for axis, mu, coef in across:
        if mu:
            v = _limit(lim, T.roll(-1, axis) - T, T - T.roll(1, axis))
            flux += mu * coef * scale * _limit(lim, v, v.roll(-1, -1))
    return T + _solve(lam * normal * scale, flux - flux.roll(1, -1))


def _coefficients(case, along, cross):
    """Normal and transverse coefficients at the faces along the last axis (0 at a wall), rounded as the option asks."""
    f = [0.5 * (v + v.roll(-1, -1)) for v in [along] + cross]
    out = [f[0] * v for v in f]
    for v in out:
        if case["problem"] != "random":
            v[..., -1] = 0.0
    return [v.half().double() for v in out] if case["field_fp16"] else out


def _update_lines(case, T, along, cross, lam, mu, alpha):
    """A two-dimensional update along the last axis, some lines at a time, each time with the lines on both sides
    (mirrored at a wall), for which nothing is kept."""
    L, n = T.shape
    out = torch.empty_like(T)
    some = max(1, (1 << 25) // n)
    for i in range(0, L, some):
        j = min(L, i + some)
        rows = torch.arange(i - 1, j + 1, device=T.device)
        rows = rows % L if case["problem"] == "random" else rows.clamp(0, L - 1)
        normal, transverse = _coefficients(case, along[rows].double(), [cross[rows].double()])
        out[i:j] = _update(T[rows], lam, normal, [(0, mu, transverse)], case["limiter"], alpha)[1:-1]
    return out


def _exact2(case, T, bx, by, nx, ny, chi, cfl):
    dx, dy = _spacing(case, nx, ny)
    dt = _dt(case, dx, dy, chi, cfl)
    lam = {"x": chi * dt / dx ** 2, "y": chi * dt / dy ** 2}
    mu = chi * dt / (dx * dy)
    alpha = 2.5 if case["call"] == "coupled" else 0.0
    T = T.double()
    bxT, byT = bx.T.contiguous(), by.T.contiguous()
    for k in range(case["steps"]):
        first = {"xy": "x", "yx": "y", "alternate": "xy"[k % 2]}[case["order"]]
        for d in (first, "y" if first == "x" else "x"):
            halves = [(1.0, mu)] if case["scheme"] == "2step" else [(0.5, mu), (0.5, 0.0)]
            for part, m in halves:
                if d == "x":
                    T = _update_lines(case, T, bx, by, part * lam[d], m, alpha)
                else:
                    T = _update_lines(case, T.T.contiguous(), byT, bxT, part * lam[d], m, alpha).T.contiguous()
    return T


def _exact3(case, T, b):
    n = (case["nx"], case["ny"], case["nz"])
    dt = case["cfl"] / max(n) ** 2 / (2.0 * CHI)
    halves = [(1.0, 1.0)] if case["scheme"] == "2step" else [(0.5, 1.0), (0.5, 0.0)]
    T = T.double()
    for _ in range(case["steps"]):
        for d in range(3):  # axis d last: the others keep their order
            order = [a for a in (2, 1, 0) if a != d] + [d]
            perm = [2 - a for a in order]
            back = [perm.index(i) for i in range(3)]
            turned = [v.double().permute(perm) for v in b]
            cross = [a for a in (0, 1, 2) if a != d]
            coef = _coefficients(case, turned[d], [turned[a] for a in cross])
            T = T.permute(perm).contiguous()
            for part, transverse in halves:
                across = [(order.index(a), transverse * CHI * dt * n[d] * n[a], c) for a, c in zip(cross, coef[1:])]
                T = _update(T, part * CHI * dt * n[d] ** 2, coef[0], across, case["limiter"])
            T = T.permute(back).contiguous()
    return T


def exact(case, seed):
    grids = _grids(case)
    if case["call"] == "step3d":
        (b, T), = _inputs(case, seed)
        return _exact3(case, T, b)
    if case["call"] == "batch":
        parts = []
        for (nx, ny, chi, cfl), (bx, by, T) in zip(grids, _inputs(case, seed)):
            flat = _exact2(case, T, bx, by, nx, ny, chi, cfl).reshape(-1)
            parts.append(torch.nn.functional.pad(flat, (0, -flat.numel() % 64)))
        return torch.cat(parts)
    (bx, by, T), = _inputs(case, seed)
    out = _exact2(case, T, bx, by, *grids[0])
    if case["call"] == "monitor":
        return {"T": out, "sum": float(out.sum()), "min": float(out.min()), "max": float(out.max()), "nonfinite": None}
    return out
