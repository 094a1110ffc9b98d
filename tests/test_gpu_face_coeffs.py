"""The stored face coefficients, normal and transverse, in the natural and the
transposed layout: bit for bit the FP64 values rounded once to the storage type."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
LAUNCH = "_ZN5aniso18launch_face_coeffsEiiPKvS1_iiidPvS2_S2_S2_S2_S2_P11CUstream_st"
KIND = {0: np.float64, 1: np.float32, 2: np.float16}


def _field(kind, ny, nx, rng):
    if kind == "unit":
        a = 2 * np.pi * rng.rand(ny, nx)
        return np.cos(a), np.sin(a)
    if kind == "axis":  # along x, with zeros of both signs
        return np.ones((ny, nx)), np.where(rng.rand(ny, nx) < 0.5, 0.0, -0.0)
    if kind == "opposed":  # means that cancel
        a = rng.randn(ny, nx)
        s = 1 - 2 * (np.indices((ny, nx)).sum(0) % 2)
        return s * (1 + 1e-6 * a), s * a
    if kind == "short":  # 13-bit values: products halfway between two FP32 numbers
        return rng.randint(-8191, 8192, (2, ny, nx)) / 8192.0
    if kind == "graded":  # magnitudes over 60 binary orders and more
        e = rng.randint(-75, 3, (2, ny, nx))
        return np.ldexp(rng.randn(2, ny, nx), e)
    if kind == "tiny":
        return np.ldexp(rng.randn(2, ny, nx), -62)
    return np.ldexp(rng.randn(2, ny, nx), 40)  # large


def _want(bn, bt, ax, bc, kappa, dtype):
    omk = 1.0 - kappa
    with np.errstate(over="ignore", under="ignore"):
        fn, ft = (0.5 * (v + np.roll(v, -1, ax)) for v in (bn, bt))
        n, t = kappa + omk * (fn * fn), omk * (fn * ft)
        if bc == 0:
            edge = [slice(None)] * 2
            edge[ax] = -1
            n[tuple(edge)] = t[tuple(edge)] = 0.0
        return n.astype(dtype), t.astype(dtype)


@pytest.mark.parametrize("kind", ["unit", "axis", "opposed", "short", "graded", "tiny", "large"])
@pytest.mark.parametrize("prec,coef", [(1, 1), (1, 2), (0, 0)])
@pytest.mark.parametrize("nx,ny", [(3, 3), (33, 36), (64, 7), (31, 265), (200, 129)])
def test_coefficients_are_the_rounded_fp64_values(lib, kind, prec, coef, nx, ny):
    import torch
    launch = getattr(lib.load(), LAUNCH)
    launch.restype = ctypes.c_int
    vp = ctypes.c_void_p
    bits = {8: np.uint64, 4: np.uint32, 2: np.uint16}[np.dtype(KIND[coef]).itemsize]
    for bc in (0, 1):
        for kappa in (0.0, 0.3, 1e-7, 1.0):
            bx, by = (np.ascontiguousarray(v, dtype=KIND[prec])
                      for v in _field(kind, ny, nx, np.random.RandomState(nx + ny)))
            dev = [torch.from_numpy(v).cuda() for v in (bx, by)]
            out = [torch.zeros(nx * ny, dtype={0: torch.float64, 1: torch.float32, 2: torch.float16}[coef], device="cuda")
                   for _ in range(6)]
            rc = launch(prec, coef, vp(dev[0].data_ptr()), vp(dev[1].data_ptr()), nx, ny, bc, ctypes.c_double(kappa),
                        *(vp(o.data_ptr()) for o in out), vp(torch.cuda.current_stream().cuda_stream))
            assert rc == 0
            torch.cuda.synchronize()
            got = [o.cpu().numpy() for o in out]
            bx, by = bx.astype(np.float64), by.astype(np.float64)
            xx, xy = _want(bx, by, 1, bc, kappa, KIND[coef])
            yy, yx = _want(by, bx, 0, bc, kappa, KIND[coef])
            for g, w in zip(got, (xx, xy, yy, yx, yy.T, yx.T)):
                w = np.ascontiguousarray(w).reshape(-1)
                assert np.array_equal(g.view(bits), w.view(bits))
