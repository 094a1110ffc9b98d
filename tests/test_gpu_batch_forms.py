"""Batches that mix the forms of the warp-per-line kernel: shared-memory,
tensor-memory and ragged classes of one sweep."""
import numpy as np
import pytest

import workloads as W
from gpu_util import GpuGrid

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
