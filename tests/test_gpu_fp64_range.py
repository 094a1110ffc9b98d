"""FP64 steps of fields whose differences, or their products, lie far from 1:
the limiter is that of the oracle there too."""
import numpy as np
import pytest

import workloads as W
from gpu_util import FP64_TOL_PER_STEP, GpuGrid, oracle_inputs, oracle_step, rel_linf

pytestmark = pytest.mark.gpu
FP64 = 0
# whole vectors, ragged, columns and rows on the long-line kernel, a small grid with short segments
SHAPES = [(64, 200), (51, 33), (1100, 40), (40, 1026), (24, 24)]


@pytest.mark.parametrize("nx,ny", SHAPES)
@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("scale", [1e-100, 1e-140, 1e-150, 1e-154, 1e-155, 1e-170, 1e120, 1e150])
def test_scaled_fields_follow_the_oracle(lib, nx, ny, bc, scale):
    """Relative to the field's own scale.  At 1e-155 the products of two
    differences have lost up to 14 bits to the denormal range, at 1e-170 all."""
    inst = (W.random_instance(nx, ny, seed=nx + ny, dt_factor=20.0) if bc else
            W.ring_instance(nx, ny=ny, dt_factor=20.0))
    T0, co = oracle_inputs(lib, inst, FP64)
    T0 = T0 * scale
    g = GpuGrid(lib, inst, FP64, T0=T0)
    try:
        got = g.step(2)
        assert rel_linf(got / scale, oracle_step(inst, T0, co, 2) / scale) < (
            2 * FP64_TOL_PER_STEP if scale > 1e-152 else 1e-9)
    finally:
        g.close()


@pytest.mark.parametrize("nx,ny", SHAPES)
def test_differences_whose_products_overflow_are_reported(lib, nx, ny):
    inst = W.random_instance(nx, ny, seed=nx + ny, dt_factor=20.0)
    T0, co = oracle_inputs(lib, inst, FP64)
    T0 = (T0 - T0.mean()) * 1e200
    assert not np.isfinite(oracle_step(inst, T0, co, 1)).all()
    g = GpuGrid(lib, inst, FP64, T0=T0)
    try:
        with pytest.raises(lib.AnisoError) as ei:
            g.step(1)
        assert ei.value.code == lib.ANISO_ERR_NONFINITE
    finally:
        g.close()
