"""Calls captured into a graph of the caller's, on the caller's stream: chained
launches become edges of that graph, and its replays give the same bits."""
import pytest

import workloads as W
from gpu_util import GpuGrid

pytestmark = pytest.mark.gpu
FP64, FP32 = 0, 1


@pytest.mark.parametrize("prec,nx,ny", [(FP32, 64, 48), (FP32, 51, 33), (FP32, 512, 500), (FP64, 50, 50), (FP64, 352, 256),
                                        (FP64, 1100, 40)])
def test_steps_captured_by_the_caller(lib, prec, nx, ny):
    import torch
    inst = W.random_instance(nx, ny, seed=4, dt_factor=20.0)
    a, b = (GpuGrid(lib, inst, prec, graph=False) for _ in range(2))
    t = a.T.clone()
    want = a.T.clone()
    stream = torch.cuda.Stream()
    small = nx * ny <= 1 << 18
    try:
        lib.aniso_set_option(a.h, lib.ANISO_OPT_STREAM, stream.cuda_stream)
        torch.cuda.synchronize()

        def noalloc(T, s):
            if small:
                lib.aniso_step_noalloc(nx, ny, inst.dx, inst.dy, inst.chi_par, 0.0, inst.bc, prec, a.bx, a.by, T, inst.dt,
                                       2, stream=s)

        noalloc(want.clone(), None)  # (its scratch memory, before the capture)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            lib.aniso_step(a.h, a.T, inst.dt, 3)
            noalloc(t, stream.cuda_stream)
        for _ in range(2):
            graph.replay()
        torch.cuda.synchronize()
        for _ in range(2):
            lib.aniso_step(b.h, b.T, inst.dt, 3)
            noalloc(want, None)
        torch.cuda.synchronize()
        assert torch.equal(a.T, b.T)
        assert torch.equal(t, want)
    finally:
        a.close()
        b.close()
