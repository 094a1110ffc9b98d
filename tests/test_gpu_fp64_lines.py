"""FP64 lines against the oracle: long ones on the kernel whose team spans four
warps (1024 < n <= 4096, first and last length, uneven segments), and small
grids stepped alone, whose lines take shorter segments."""
import numpy as np
import pytest

import workloads as W
from gpu_util import FP64_TOL_PER_STEP, GpuGrid, oracle_inputs, oracle_step, rel_linf

pytestmark = pytest.mark.gpu
FP64 = 0


def _inst(nx, ny, bc):
    if bc == 1:
        return W.random_instance(nx, ny, seed=nx + 7 * ny, dt_factor=100.0)
    return W.ring_instance(nx, ny=ny, dt_factor=100.0)


@pytest.mark.parametrize("nx,ny", [(1026, 32), (32, 1026), (1282, 1538), (4096, 34), (34, 4096), (2048, 2046)])
@pytest.mark.parametrize("bc", [0, 1])
def test_long_lines(lib, nx, ny, bc):
    inst = _inst(nx, ny, bc)
    T0, co = oracle_inputs(lib, inst, FP64)
    g = GpuGrid(lib, inst, FP64)
    try:
        assert rel_linf(g.step(2), oracle_step(inst, T0, co, 2)) < 2 * FP64_TOL_PER_STEP
    finally:
        g.close()


@pytest.mark.parametrize("limiter", [1, 2, 3])
def test_long_lines_limiters(lib, limiter):
    inst = _inst(1600, 64, 1)
    T0, co = oracle_inputs(lib, inst, FP64)
    g = GpuGrid(lib, inst, FP64, limiter=limiter)
    try:
        assert rel_linf(g.step(2), oracle_step(inst, T0, co, 2, limiter=limiter)) < 2 * FP64_TOL_PER_STEP
    finally:
        g.close()


def test_long_lines_in_a_batch_equal_single_grids(lib):
    import torch
    insts = [_inst(1100, 40, 1), _inst(40, 2050, 0), _inst(4096, 36, 1), _inst(96, 64, 1)]
    grids = [GpuGrid(lib, i, FP64) for i in insts]
    singles = [GpuGrid(lib, i, FP64) for i in insts[:3]]
    try:
        b = lib.aniso_batch_create([g.h for g in grids])
        lib.aniso_step_batched(b, [g.T for g in grids], [i.dt for i in insts], [2] * len(insts))
        torch.cuda.synchronize()
        for g, inst in zip(grids, insts):
            T0, co = oracle_inputs(lib, inst, FP64)
            assert rel_linf(g.T.cpu().numpy(), oracle_step(inst, T0, co, 2)) < 2 * FP64_TOL_PER_STEP
        assert np.array_equal(grids[2].T.cpu().numpy(), singles[2].step(2))
        lib.aniso_batch_destroy(b)
    finally:
        for g in grids + singles:
            g.close()


@pytest.mark.parametrize("nx,ny", [(4, 4), (8, 6), (10, 34), (50, 50), (62, 300), (300, 62)])
@pytest.mark.parametrize("bc", [0, 1])
def test_small_grids(lib, nx, ny, bc):
    inst = _inst(nx, ny, bc)
    T0, co = oracle_inputs(lib, inst, FP64)
    g = GpuGrid(lib, inst, FP64)
    try:
        assert rel_linf(g.step(5), oracle_step(inst, T0, co, 5)) < 5 * FP64_TOL_PER_STEP
    finally:
        g.close()


def test_tiny_and_zero_differences(lib):
    """Temperatures whose differences span 1e-300 to 1 (products that
    underflow are told from zero by the limiter's sign test), on flat ground."""
    inst = _inst(64, 48, 1)
    rng = np.random.RandomState(3)
    T0 = np.where(rng.rand(48, 64) < 0.5, 10.0 ** rng.uniform(-300, 0, (48, 64)), 0.0)
    _, co = oracle_inputs(lib, inst, FP64)
    g = GpuGrid(lib, inst, FP64, T0=T0)
    try:
        got = g.step(1)
        assert np.isfinite(got).all()
        assert rel_linf(got, oracle_step(inst, T0, co, 1)) < FP64_TOL_PER_STEP
    finally:
        g.close()
