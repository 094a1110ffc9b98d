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
