"""Which launches overlap the end of the one before them, and what that may
cost: a chained call is never much slower than the same call with its launches
kept apart (a profiled handle's timing events do that)."""
import time

import pytest

import workloads as W
from gpu_util import GpuGrid

pytestmark = pytest.mark.gpu
FP64, FP32 = 0, 1


def _best(f, calls=7):
    import torch
    times = []
    for _ in range(calls):
        torch.cuda.synchronize()
        t = time.perf_counter()
        f()
        torch.cuda.synchronize()
        times.append(time.perf_counter() - t)
    return min(times[2:])


# blocks that fill the chip less than once or twice, with room on an SM for
# several more of them (placed unevenly, these took 1.4 to 2.5 times as long)
@pytest.mark.parametrize("nx,ny,prec,order", [(352, 512, FP64, 0), (512, 352, FP64, 1), (777, 1001, FP32, 0),
                                              (1001, 777, FP32, 1), (777, 1001, FP64, 0), (1100, 200, FP64, 0)])
def test_chained_calls_keep_the_chip_evenly_filled(lib, nx, ny, prec, order):
    inst = W.random_instance(nx, ny, seed=7, dt_factor=20.0)
    a, b = (GpuGrid(lib, inst, prec, order=order) for _ in range(2))
    try:
        lib.aniso_set_option(b.h, lib.ANISO_OPT_PROFILE, 1)
        chained, apart = (_best(lambda g=g: lib.aniso_step(g.h, g.T, inst.dt, 20)) for g in (a, b))
        assert chained < 1.2 * apart
    finally:
        a.close()
        b.close()


@pytest.mark.parametrize("n", [(32, 32, 32), (20, 64, 36), (64, 64, 64), (96, 100, 104), (136, 192, 60)])
@pytest.mark.parametrize("prec,fp16", [(FP32, False), (FP32, True), (FP64, False)])
@pytest.mark.parametrize("scheme", [0, 1])
def test_3d_steps_of_one_call_equal_steps_waited_for(lib, n, prec, fp16, scheme):
    """Within a call the launches overlap and ask for other amounts of shared
    memory; one-step calls with a wait after each keep all but two apart."""
    import torch
    inst = W.random_instance3d(*n, seed=3)
    dt = torch.float64 if prec == FP64 else torch.float32
    got = []
    for calls, steps in ((1, 6), (6, 1)):
        h = lib.aniso3_create(*n, inst.dx, inst.dy, inst.dz, inst.chi_par, 0.0, inst.bc)
        try:
            lib.aniso3_set_option(h, lib.ANISO_OPT_PRECISION, prec)
            lib.aniso3_set_option(h, lib.ANISO_OPT_FIELD_FP16, int(fp16))
            lib.aniso3_set_option(h, lib.ANISO_OPT_SCHEME, scheme)
            lib.aniso3_set_field(h, *(torch.tensor(v, dtype=dt, device="cuda") for v in (inst.bx, inst.by, inst.bz)))
            T = torch.tensor(inst.T0, dtype=dt, device="cuda")
            for _ in range(calls):
                lib.aniso3_step(h, T, inst.dt, steps)
                torch.cuda.synchronize()
            lib.aniso3_sync(h)
            got.append(T)
        finally:
            lib.aniso3_destroy(h)
    assert torch.equal(*got)


@pytest.mark.parametrize("n,handles,most", [(512, 8, 4.0), (1024, 4, 3.0), (300, 16, 3.0), (1216, 4, 3.4)])
def test_handles_on_streams_of_their_own_share_the_gpu(lib, n, handles, most):
    """Several handles stepped at once, each on its own stream, against one of
    them alone: 1.7, 1.9, 1.4 and 2.8 times as long with every launch plain; 6.4,
    3.8 and 4.4 where chained blocks kept an SM to themselves, 4.1 (1216) with three
    rounds of loads in flight."""
    import torch
    insts = [W.random_instance(n, n, seed=k, dt_factor=20.0) for k in range(handles)]
    grids = [GpuGrid(lib, i, FP32) for i in insts]
    streams = [torch.cuda.Stream() for _ in insts]
    try:
        torch.cuda.synchronize()
        for g, s in zip(grids, streams):
            lib.aniso_set_option(g.h, lib.ANISO_OPT_STREAM, s.cuda_stream)

        def run(some):
            for _ in range(4):
                for g, i in some:
                    lib.aniso_step(g.h, g.T, i.dt, 20)

        pairs = list(zip(grids, insts))
        alone, all_at_once = (_best(lambda some=some: run(some), 9) for some in (pairs[:1], pairs))
        assert all_at_once < most * alone
    finally:
        torch.cuda.synchronize()
        for g in grids:
            g.close()
