"""Ragged grids near the top of FP32's range: finite temperatures are not
reported, whatever their sums are."""
import numpy as np
import pytest

import workloads as W
from gpu_util import GpuGrid

pytestmark = pytest.mark.gpu
FP32 = 1


@pytest.mark.parametrize("nx,ny", [(51, 33), (66, 130), (1001, 40), (35, 2304), (4096, 33)])
def test_large_finite_temperatures(lib, nx, ny):
    inst = W.random_instance(nx, ny, seed=2, dt_factor=20.0)
    T0 = np.full((ny, nx), 2e38)  # (uniform: every flux is 0)
    g = GpuGrid(lib, inst, FP32, T0=T0)
    try:
        assert np.array_equal(g.step(2), T0.astype(np.float32).astype(np.float64))
        g.T[0, nx - 1] = float("inf")
        with pytest.raises(lib.AnisoError) as ei:
            g.step(1)
        assert ei.value.code == lib.ANISO_ERR_NONFINITE
    finally:
        g.close()
