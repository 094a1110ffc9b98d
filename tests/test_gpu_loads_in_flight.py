"""FP32 grids alone on both sides of the line (38912 threads, 8 warps an SM) up
to which the warp-per-line kernel keeps three rounds of loads in flight: the
same bits as in a batch, which never does."""
import numpy as np
import pytest

import workloads as W
from gpu_util import GpuGrid

pytestmark = pytest.mark.gpu
FP32 = 1


# four-warp blocks of one line a warp: 1216 lines make 304 blocks of 128 threads, 1220 make 305;
# eight-warp blocks (the default where they run in one wave): 1216 lines make 152 of 256
@pytest.mark.parametrize("nx,ny,warps", [(1300, 1216, 4), (1300, 1220, 4), (1216, 1300, 4), (1220, 1300, 4),
                                         (1300, 1216, 0), (1300, 1220, 0)])
@pytest.mark.parametrize("limiter", [0, 1])
def test_three_rounds_in_flight_equal_one(lib, nx, ny, warps, limiter):
    import torch
    inst = W.random_instance(nx, ny, seed=nx + ny, dt_factor=50.0)
    a, b = (GpuGrid(lib, inst, FP32, limiter=limiter) for _ in range(2))
    try:
        lib.aniso_set_option(a.h, lib.ANISO_OPT_BLOCK_WARPS, warps)
        batch = lib.aniso_batch_create([b.h])
        lib.aniso_step_batched(batch, [b.T], [inst.dt], [3])
        torch.cuda.synchronize()
        assert np.array_equal(a.step(3), b.T.double().cpu().numpy())
        lib.aniso_batch_destroy(batch)
    finally:
        a.close()
        b.close()
