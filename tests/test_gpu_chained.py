"""Launches that overlap the end of the one before them (programmatic
dependent launch) against plainly ordered ones: a profiled handle's launches
are kept apart by its timing events.  Same bits, from a graph and directly."""
import numpy as np
import pytest

import workloads as W
from gpu_util import GpuGrid

pytestmark = pytest.mark.gpu
FP64, FP32 = 0, 1


@pytest.mark.parametrize("nx,ny,prec,opts", [
    (64, 64, FP32, {}), (50, 50, FP64, {}), (1024, 96, FP32, {}), (1100, 64, FP64, {}), (2304, 64, FP32, {}),
    (96, 128, FP32, {"ANISO_OPT_SCHEME": 1}), (96, 128, FP64, {"ANISO_OPT_ORDER": 2}),
    (1024, 1024, FP32, {}), (51, 77, FP32, {})])
@pytest.mark.parametrize("graph", [True, False])
def test_chained_equals_plain(lib, nx, ny, prec, opts, graph):
    inst = W.random_instance(nx, ny, seed=nx + ny, dt_factor=50.0)
    a, b = (GpuGrid(lib, inst, prec, graph=graph) for _ in range(2))
    try:
        for g in (a, b):
            for k, v in opts.items():
                lib.aniso_set_option(g.h, getattr(lib, k), v)
        lib.aniso_set_option(b.h, lib.ANISO_OPT_PROFILE, 1)
        for steps in (7, 1, 30):
            assert np.array_equal(a.step(steps), b.step(steps))
    finally:
        a.close()
        b.close()


def test_calls_of_one_step_back_to_back(lib):
    """Many one-step calls without a wait between them, one stream, then a call
    on another array: each call's first launch follows the last one plainly."""
    inst = W.random_instance(128, 96, seed=4, dt_factor=50.0)
    a, b = (GpuGrid(lib, inst, FP32) for _ in range(2))
    try:
        for _ in range(40):
            lib.aniso_step(a.h, a.T, inst.dt, 1)
        assert np.array_equal(a.step(0), b.step(40))
    finally:
        a.close()
        b.close()


@pytest.mark.parametrize("nx,ny,prec", [(64, 48, FP32), (51, 33, FP32), (50, 50, FP64), (1024, 256, FP32)])
def test_fields_that_change_every_call(lib, nx, ny, prec):
    """Set a field, take one step, set another, and so on without a wait: each
    step sees its own field (the coefficients are rewritten between launches that
    overlap), as with a wait after every call."""
    import torch
    fields = [W.random_instance(nx, ny, seed=k, dt_factor=50.0) for k in range(3)]
    dt = torch.float64 if prec == FP64 else torch.float32
    b = [[torch.tensor(v, dtype=dt, device="cuda") for v in (f.bx, f.by)] for f in fields]
    got = []
    for wait in (False, True):
        g = GpuGrid(lib, fields[0], prec)
        t = g.T.clone()
        try:
            for k in range(30):
                bx, by = b[k % 3]
                lib.aniso_set_field(g.h, bx, by)
                if wait:
                    torch.cuda.synchronize()
                lib.aniso_step(g.h, g.T, fields[0].dt, 1)
                if wait:
                    torch.cuda.synchronize()
                f = fields[0]
                if nx * ny <= 1 << 17:
                    lib.aniso_step_noalloc(nx, ny, f.dx, f.dy, f.chi_par, 0.0, f.bc, prec, by, bx, t, f.dt, 1)
                    if wait:
                        torch.cuda.synchronize()
            lib.aniso_sync(g.h)
            got.append((g.T.cpu(), t.cpu()))
        finally:
            g.close()
    for x, y in zip(*got):
        assert torch.equal(x, y)
