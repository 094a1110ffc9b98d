"""FP64 lines of 3074 to 4096 cells where there are few of them: minmod and MC
run on the general kernels, van Leer on the long-line kernel, whichever limiter
the handle had when its field was set."""
import numpy as np
import pytest

import workloads as W
from gpu_util import FP64_TOL_PER_STEP, GpuGrid, oracle_inputs, oracle_step, rel_linf

pytestmark = pytest.mark.gpu
FP64 = 0


@pytest.mark.parametrize("nx,ny", [(4096, 64), (64, 4096), (3074, 152), (4096, 33)])
@pytest.mark.parametrize("bc", [0, 1])
def test_limiters_in_turn_on_few_long_lines(lib, nx, ny, bc):
    inst = (W.random_instance(nx, ny, seed=nx + ny, dt_factor=20.0) if bc else
            W.ring_instance(nx, ny=ny, dt_factor=20.0))
    T0, co = oracle_inputs(lib, inst, FP64)
    g = GpuGrid(lib, inst, FP64, limiter=2)
    try:
        for limiter in (2, 0, 1, 3, 0):
            lib.aniso_set_option(g.h, lib.ANISO_OPT_LIMITER, limiter)
            g.T.copy_(g.T.new_tensor(T0))
            ref = oracle_step(inst, T0, co, 2, limiter=limiter)
            assert rel_linf(g.step(2), ref) < 2 * FP64_TOL_PER_STEP
    finally:
        g.close()


def test_few_long_lines_with_mc_run_the_general_kernels(lib):
    inst = W.random_instance(4096, 64, seed=9, dt_factor=20.0)
    a, b = GpuGrid(lib, inst, FP64, limiter=2), GpuGrid(lib, inst, FP64, limiter=2, fast=1)
    try:
        assert np.array_equal(a.step(3), b.step(3))
    finally:
        a.close()
        b.close()
