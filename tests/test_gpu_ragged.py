"""Lines that are no multiple of the 16-byte vector, and arrays that are not
aligned to it, on the warp-per-line kernel's ragged form against the oracle."""
import numpy as np
import pytest

import workloads as W
from gpu_util import FP64_TOL_PER_STEP, GpuGrid, fp32_tol, oracle_inputs, oracle_step, rel_linf

pytestmark = pytest.mark.gpu
FP64, FP32 = 0, 1

# last chunks of 1, 2 and 3 cells; single-lane teams, segments of one cell,
# the first and the last length of a team, the longest line
SHAPES32 = [(3, 3), (4, 5), (5, 7), (6, 9), (13, 17), (33, 35), (65, 63), (129, 66), (130, 257), (511, 50), (50, 513),
            (1001, 77), (77, 1001), (2047, 21), (23, 2045), (2046, 9)]
SHAPES64 = [(3, 3), (5, 4), (7, 9), (17, 33), (51, 53), (65, 129), (1023, 30), (31, 1021)]


def _inst(nx, ny, bc, dt_factor=100.0):
    if bc == 1:
        return W.random_instance(nx, ny, seed=nx + 5 * ny, dt_factor=dt_factor)
    return W.ring_instance(nx, ny=ny, dt_factor=dt_factor)


@pytest.mark.parametrize("prec,shape", [(FP32, s) for s in SHAPES32] + [(FP64, s) for s in SHAPES64])
@pytest.mark.parametrize("bc", [0, 1])
def test_ragged_steps(lib, prec, shape, bc):
    inst = _inst(*shape, bc)
    T0, co = oracle_inputs(lib, inst, prec)
    g = GpuGrid(lib, inst, prec)
    try:
        got = g.step(3)
        ref = oracle_step(inst, T0, co, 3)
        tol = 3 * FP64_TOL_PER_STEP if prec == FP64 else fp32_tol(inst, T0, co, 3, ref)
        assert rel_linf(got, ref) < tol
    finally:
        g.close()


@pytest.mark.parametrize("limiter", [1, 2, 3])
@pytest.mark.parametrize("prec", [FP64, FP32])
def test_ragged_limiters_and_orders(lib, prec, limiter):
    inst = _inst(101, 67, 1)
    T0, co = oracle_inputs(lib, inst, prec)
    for order in (0, 1, 2):
        g = GpuGrid(lib, inst, prec, limiter=limiter, order=order)
        try:
            got = g.step(4)
            ref = oracle_step(inst, T0, co, 4, order=order, limiter=limiter)
            tol = 4 * FP64_TOL_PER_STEP if prec == FP64 else fp32_tol(inst, T0, co, 4, ref)
            assert rel_linf(got, ref) < tol
        finally:
            g.close()


@pytest.mark.parametrize("prec,fp16", [(FP64, False), (FP32, False), (FP32, True)])
@pytest.mark.parametrize("nx,ny", [(64, 48), (67, 48), (64, 50)])
def test_unaligned_temperature(lib, prec, fp16, nx, ny):
    """T one element past an aligned address, in whole and ragged shapes."""
    import torch
    inst = _inst(nx, ny, 1)
    T0, co = oracle_inputs(lib, inst, prec, fp16=fp16)
    g = GpuGrid(lib, inst, prec, fp16=fp16)
    try:
        room = torch.zeros(nx * ny + 2, dtype=g.T.dtype, device="cuda")
        T = room[1:1 + nx * ny].view(ny, nx)
        T.copy_(g.T)
        lib.aniso_step(g.h, T, inst.dt, 3)
        lib.aniso_sync(g.h)
        ref = oracle_step(inst, T0, co, 3)
        tol = 3 * FP64_TOL_PER_STEP if prec == FP64 else fp32_tol(inst, T0, co, 3, ref)
        assert rel_linf(T.double().cpu().numpy(), ref) < tol
        assert float(room[0]) == 0.0 and float(room[-1]) == 0.0
    finally:
        g.close()


@pytest.mark.parametrize("nx,ny", [(4096, 33), (35, 2304), (2303, 64)])
def test_ragged_across_long_lines(lib, nx, ny):
    """One side on a long-line kernel (or neither), the other ragged."""
    inst = _inst(nx, ny, 1)
    T0, co = oracle_inputs(lib, inst, FP32)
    g = GpuGrid(lib, inst, FP32)
    try:
        ref = oracle_step(inst, T0, co, 2)
        assert rel_linf(g.step(2), ref) < fp32_tol(inst, T0, co, 2, ref)
    finally:
        g.close()


def test_ragged_in_a_batch(lib):
    """Ragged and whole grids in one batch: each equals its grid alone, and the
    per-step diagnostics of ragged grids stay unrecorded (NaN)."""
    import torch
    insts = [_inst(101, 66, 1), _inst(64, 96, 1), _inst(300, 7, 0), _inst(97, 128, 0), _inst(2303, 16, 1)]
    grids = [GpuGrid(lib, i, FP32) for i in insts]
    singles = [GpuGrid(lib, i, FP32) for i in insts]
    lib.aniso_set_option(grids[0].h, lib.ANISO_OPT_DIAGNOSTICS, 1)
    try:
        b = lib.aniso_batch_create([g.h for g in grids])
        lib.aniso_step_batched(b, [g.T for g in grids], [i.dt for i in insts], [3] * len(insts))
        torch.cuda.synchronize()
        ring = lib.aniso_batch_diagnostics(b, len(insts))
        for k, (g, s) in enumerate(zip(grids, singles)):
            got = g.T.double().cpu().numpy()
            assert np.array_equal(got, s.step(3))
            if k == 1:
                assert ring[k, 2, 1] == got.min() and ring[k, 2, 2] == got.max()
            else:
                assert np.isnan(ring[k]).all()
        lib.aniso_batch_destroy(b)
    finally:
        for g in grids + singles:
            g.close()


def test_what_ragged_grids_cannot_do_is_refused(lib):
    inst = _inst(51, 53, 1)
    g = GpuGrid(lib, inst, FP32)
    try:
        lib.aniso_set_nonlinear(g.h, 2.5, 1.0)
        with pytest.raises(lib.AnisoError) as ei:
            lib.aniso_step(g.h, g.T, inst.dt, 1)
        assert ei.value.code == lib.ANISO_ERR_UNSUPPORTED
    finally:
        g.close()
