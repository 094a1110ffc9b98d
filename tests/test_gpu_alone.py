"""FP32 grids stepped alone take other launch shapes than in a batch (eight-warp
blocks, more loads in flight): the same bits, on both sides of the rules' lines."""
import numpy as np
import pytest

import workloads as W
from gpu_util import GpuGrid

pytestmark = pytest.mark.gpu
FP32 = 1


# 768: the first 96 eight-warp blocks; 1216: the last single wave; 1280: four
# warps, still three rounds in flight; 2048 x 640: 16-chunk segments; 8 x 2000: one-lane teams
@pytest.mark.parametrize("nx,ny", [(64, 64), (768, 760), (768, 768), (1024, 1000), (1216, 1216), (1280, 1220), (2048, 640),
                                   (2000, 8)])
@pytest.mark.parametrize("fp16", [False, True])
def test_alone_equals_batch(lib, nx, ny, fp16):
    import torch
    inst = W.random_instance(nx, ny, seed=nx + ny, dt_factor=50.0)
    a, b, c = (GpuGrid(lib, inst, FP32, fp16=fp16) for _ in range(3))
    try:
        lib.aniso_set_option(c.h, lib.ANISO_OPT_BLOCK_WARPS, 4)
        bt = lib.aniso_batch_create([b.h])
        lib.aniso_step_batched(bt, [b.T], [inst.dt], [3])
        torch.cuda.synchronize()
        got = a.step(3)
        assert np.array_equal(got, b.T.double().cpu().numpy())
        assert np.array_equal(got, c.step(3))
        lib.aniso_batch_destroy(bt)
    finally:
        for g in (a, b, c):
            g.close()


@pytest.mark.parametrize("nx,ny", [(96, 64), (1024, 1024)])
def test_nonlinear_alone(lib, nx, ny):
    inst = W.random_instance(nx, ny, seed=5, dt_factor=10.0)
    a, c = (GpuGrid(lib, inst, FP32) for _ in range(2))
    try:
        lib.aniso_set_option(c.h, lib.ANISO_OPT_BLOCK_WARPS, 4)
        for g in (a, c):
            lib.aniso_set_nonlinear(g.h, 2.5, 1.0)
        assert np.array_equal(a.step(3), c.step(3))
    finally:
        a.close()
        c.close()


# every number of chunk rounds with a form of its own (4 .. 8), whole and uneven
# segments, teams of 32, 16, 8 and 4 lanes, and the lengths on both sides (3 and 9 rounds)
@pytest.mark.parametrize("n", [12, 48, 64, 92, 128, 132, 252, 256, 260, 400, 508, 512, 516, 640, 644, 768, 900, 1020, 1024, 1028])
def test_constant_rounds_equal_run_time_rounds(lib, n):
    """A grid alone, a batch of one shape and a batch whose other grid has another
    number of rounds (the run-time form), with and without tensor memory."""
    import torch
    inst = W.random_instance(n, 40, seed=n, dt_factor=50.0)
    other = W.random_instance(96 if n != 96 else 64, 16, seed=1, dt_factor=50.0)
    want = None
    for mixed in (False, True):
        for tmem in (0, 1):
            gs = [GpuGrid(lib, inst, FP32) for _ in range(2)] + ([GpuGrid(lib, other, FP32)] if mixed else [])
            s = GpuGrid(lib, inst, FP32)
            try:
                lib.aniso_set_option(gs[0].h, lib.ANISO_OPT_TMEM, tmem)
                b = lib.aniso_batch_create([g.h for g in gs])
                lib.aniso_step_batched(b, [g.T for g in gs], [g.inst.dt for g in gs], [2] * len(gs))
                torch.cuda.synchronize()
                want = s.step(2) if want is None else want
                for g in gs[:2]:
                    assert np.array_equal(g.T.double().cpu().numpy(), want)
                lib.aniso_batch_destroy(b)
            finally:
                for g in gs + [s]:
                    g.close()
