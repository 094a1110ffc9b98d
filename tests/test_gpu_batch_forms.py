"""Batches that mix the forms of the warp-per-line kernel: shared-memory,
tensor-memory and ragged classes of one sweep."""
import numpy as np
import pytest

import workloads as W
from gpu_util import FP64_TOL_PER_STEP, GpuGrid, fp32_tol, oracle_inputs, oracle_step, rel_linf

pytestmark = pytest.mark.gpu
FP64, FP32 = 0, 1


def test_diagnostics_of_a_sweep_with_classes_of_every_form(lib):
    """Columns of so many lengths that a y-update takes more launches than run
    side by side (FP32, 128-thread blocks: 768 and 1024 cells in tensor memory;
    256, 1500 and 2048 in shared memory; 101, 1501 and 2047 ragged): each
    launch has a region of partials to itself."""
    ny = [768, 1024, 256, 1500, 2048, 101, 1501, 2047]
    insts = [W.random_instance(64 + 32 * (k % 2), n, seed=40 + k, dt_factor=50.0, nsteps=2) for k, n in enumerate(ny)]
    grids = [GpuGrid(lib, i, FP32) for i in insts]
    singles = [GpuGrid(lib, i, FP32) for i in insts]
    lib.aniso_set_option(grids[0].h, lib.ANISO_OPT_DIAGNOSTICS, 1)
    b = lib.aniso_batch_create([g.h for g in grids])
    try:
        for call in range(2):
            lib.aniso_step_batched(b, [g.T for g in grids], [i.dt for i in insts], [2] * len(insts))
            ring = lib.aniso_batch_diagnostics(b, len(insts))
            for k, (g, s) in enumerate(zip(grids, singles)):
                got = g.T.double().cpu().numpy()
                assert np.array_equal(got, s.step(2))
                if ny[k] % 4 == 0:
                    assert ring[k, 1, 0] == pytest.approx(got.sum(), rel=1e-8)
                    assert ring[k, 1, 1] == got.min() and ring[k, 1, 2] == got.max()
                else:
                    assert np.isnan(ring[k]).all()
    finally:
        lib.aniso_batch_destroy(b)
        for g in grids + singles:
            g.close()


@pytest.mark.parametrize("prec,shape,offset", [(FP32, (2001, 1501), 0), (FP32, (2000, 64), 1), (FP32, (1001, 3000), 0),
                                               (FP64, (2000, 500), 0), (FP64, (1021, 40), 0)])
def test_a_first_grid_with_long_segments_takes_any_other(lib, prec, shape, offset):
    """The first grid's ANISO_OPT_SEGMENT gives the batch 16 chunks a lane,
    which leaves long lines more than the warp-per-line kernel holds: ragged
    grids, unaligned arrays and FP64 grids with a long side run all the same."""
    import torch
    first = W.random_instance(256, 128, seed=1, dt_factor=20.0)
    inst = W.random_instance(*shape, seed=2, dt_factor=20.0)
    a, g = GpuGrid(lib, first, prec), GpuGrid(lib, inst, prec)
    T0, co = oracle_inputs(lib, inst, prec)
    lib.aniso_set_option(a.h, lib.ANISO_OPT_SEGMENT, 16)
    b = lib.aniso_batch_create([a.h, g.h])
    try:
        room = torch.zeros(g.T.numel() + 1, dtype=g.T.dtype, device="cuda")
        T = room[offset:offset + g.T.numel()].view(g.T.shape)
        T.copy_(g.T)
        lib.aniso_step_batched(b, [a.T, T], [first.dt, inst.dt], [2, 2])
        torch.cuda.synchronize()
        ref = oracle_step(inst, T0, co, 2)
        tol = 2 * FP64_TOL_PER_STEP if prec == FP64 else fp32_tol(inst, T0, co, 2, ref)
        assert rel_linf(T.double().cpu().numpy(), ref) < tol
    finally:
        lib.aniso_batch_destroy(b)
        a.close()
        g.close()


@pytest.mark.parametrize("limiter", [0, 2])
def test_fp64_grids_of_one_segment_length_have_the_same_bits_alone_and_in_a_batch(lib, limiter):
    """A small FP64 grid alone takes shorter segments than in a batch; with the
    default of 4 chunks asked for on the handle it takes the batch's."""
    import torch
    shapes = [(50, 50), (24, 24), (33, 47), (64, 200), (128, 96), (101, 67), (300, 40), (512, 512), (1100, 64)]
    insts = [W.random_instance(*s, seed=k, dt_factor=20.0) for k, s in enumerate(shapes)]
    grids = [GpuGrid(lib, i, FP64, limiter=limiter) for i in insts]
    singles = [GpuGrid(lib, i, FP64, limiter=limiter) for i in insts]
    for s in singles:
        lib.aniso_set_option(s.h, lib.ANISO_OPT_SEGMENT, 4)
    b = lib.aniso_batch_create([g.h for g in grids])
    try:
        lib.aniso_step_batched(b, [g.T for g in grids], [i.dt for i in insts], [4] * len(insts))
        torch.cuda.synchronize()
        for g, s in zip(grids, singles):
            assert np.array_equal(g.T.cpu().numpy(), s.step(4))
    finally:
        lib.aniso_batch_destroy(b)
        for g in grids + singles:
            g.close()
