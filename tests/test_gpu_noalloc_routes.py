"""aniso_step_noalloc over the kernels it chooses among: whole and ragged lines
on the warp-per-line kernel, short segments for few lines, and lines too long
for it on the general kernels.  Against the oracle, T guarded on both sides."""
import pytest

import workloads as W
from gpu_util import FP64_TOL_PER_STEP, fp32_tol, oracle_inputs, oracle_step, rel_linf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,prec", [
    (96, 64, 1), (16, 16, 1), (3, 5, 1), (37, 1000, 1), (1000, 37, 1), (609, 612, 1), (2048, 12, 1), (2052, 64, 1),
    (96, 64, 0), (5, 3, 0), (51, 53, 0), (1024, 10, 0), (1100, 64, 0)])
@pytest.mark.parametrize("bc", [0, 1])
def test_routes(lib, nx, ny, prec, bc):
    import torch
    inst = W.random_instance(nx, ny, seed=nx + ny, dt_factor=50.0) if bc == 1 else \
        W.ring_instance(nx, ny=ny, dt_factor=50.0)
    T0, co = oracle_inputs(lib, inst, prec)
    dt = torch.float64 if prec == 0 else torch.float32
    bx, by = (torch.tensor(v, dtype=dt, device="cuda") for v in (inst.bx, inst.by))
    room = torch.full((nx * ny + 8,), 7.0, dtype=dt, device="cuda")
    T = room[4:4 + nx * ny].view(ny, nx)
    T.copy_(torch.tensor(T0, dtype=dt))
    for _ in range(2):
        lib.aniso_step_noalloc(nx, ny, inst.dx, inst.dy, inst.chi_par, 0.0, bc, prec, bx, by, T, inst.dt, 2)
    ref = oracle_step(inst, T0, co, 4)
    tol = 4 * FP64_TOL_PER_STEP if prec == 0 else fp32_tol(inst, T0, co, 4, ref)
    assert rel_linf(T.double().cpu().numpy(), ref) < tol
    assert (room[:4] == 7.0).all() and (room[-4:] == 7.0).all()
