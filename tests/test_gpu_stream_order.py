"""A call's first launch follows everything the caller put on the stream, also
kernels that were launched to overlap their predecessor and do not wait for it."""
import ctypes

import pytest

import workloads as W
from gpu_build import build
from gpu_util import GpuGrid

pytestmark = pytest.mark.gpu
FP64, FP32 = 0, 1

SOURCE = r"""
#include <cuda_runtime.h>
// Lets its successor start at once, then writes `value` to p[0 .. n) late (about 0.3 ms).
__global__ void late_write(float *p, const float *value, int n)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const long long t0 = clock64();
    for (int i = 0; i < 100000 && clock64() - t0 < 600000; ++i) __nanosleep(100);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) p[i] = value[i];
}
__global__ void no_wait(int *out) { if (threadIdx.x == 0) *out = 1; }
extern "C" int late_then_no_wait(float *p, const float *value, int n, int *out, void *stream)
{
    late_write<<<4, 256, 0, (cudaStream_t)stream>>>(p, value, n);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1);
    cfg.blockDim = dim3(32);
    cfg.stream = (cudaStream_t)stream;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return (int)cudaLaunchKernelEx(&cfg, no_wait, out);
}
"""


@pytest.mark.parametrize("nx,ny", [(64, 64), (51, 33), (512, 256)])
def test_first_launches_follow_the_callers_kernels(lib, nx, ny, tmp_path):
    import torch
    probe = build(SOURCE, tmp_path)
    a, b = (W.random_instance(nx, ny, seed=k, dt_factor=50.0) for k in (1, 2))
    stream = torch.cuda.current_stream().cuda_stream
    out = torch.zeros(1, dtype=torch.int32, device="cuda")

    def late(dst, src):
        rc = probe.late_then_no_wait(ctypes.c_void_p(dst.data_ptr()), ctypes.c_void_p(src.data_ptr()), dst.numel(),
                                     ctypes.c_void_p(out.data_ptr()), ctypes.c_void_p(stream))
        assert rc == 0

    g, ref = GpuGrid(lib, a, FP32, graph=False), GpuGrid(lib, b, FP32, graph=False)
    try:
        for graph in (0, 1):
            lib.aniso_set_option(g.h, lib.ANISO_OPT_GRAPH, graph)
            # the field and T arrive late: b's over a's
            g.bx.copy_(torch.as_tensor(a.bx)), g.by.copy_(torch.as_tensor(a.by)), g.T.copy_(torch.as_tensor(a.T0))
            T0 = torch.tensor(b.T0, dtype=torch.float32, device="cuda")
            torch.cuda.synchronize()
            late(g.bx, ref.bx)
            late(g.by, ref.by)
            lib.aniso_set_field(g.h, g.bx, g.by)
            late(g.T, T0)
            lib.aniso_step(g.h, g.T, b.dt, 3)
            ref.T.copy_(T0)
            lib.aniso_step(ref.h, ref.T, b.dt, 3)
            torch.cuda.synchronize()
            assert torch.equal(g.T, ref.T)
            # the call without a handle
            t, want = T0.clone(), T0.clone()
            torch.cuda.synchronize()
            lib.aniso_step_noalloc(nx, ny, b.dx, b.dy, b.chi_par, 0.0, b.bc, FP32, ref.bx, ref.by, want, b.dt, 2)
            torch.cuda.synchronize()
            g.by.copy_(torch.as_tensor(a.by))
            torch.cuda.synchronize()
            late(g.by, ref.by)
            lib.aniso_step_noalloc(nx, ny, b.dx, b.dy, b.chi_par, 0.0, b.bc, FP32, g.bx, g.by, t, b.dt, 2)
            torch.cuda.synchronize()
            assert torch.equal(t, want)
    finally:
        g.close()
        ref.close()


@pytest.mark.parametrize("prec,nx,ny", [(FP32, 64, 64), (FP32, 51, 33), (FP32, 512, 500), (FP32, 1000, 1000), (FP64, 50, 50),
                                        (FP64, 512, 512)])
def test_noalloc_with_another_field_every_call(lib, prec, nx, ny):
    """The coefficients are rewritten between launches that overlap: each call
    sees its own field, as with a wait after every call."""
    import torch
    insts = [W.random_instance(nx, ny, seed=k, dt_factor=50.0) for k in range(3)]
    dt = torch.float64 if prec == FP64 else torch.float32
    fields = [[torch.tensor(v, dtype=dt, device="cuda") for v in (i.bx, i.by)] for i in insts]
    got = []
    for wait in (False, True):
        t = torch.tensor(insts[0].T0, dtype=dt, device="cuda")
        for k in range(24):
            i = insts[0]
            lib.aniso_step_noalloc(nx, ny, i.dx, i.dy, i.chi_par, 0.0, i.bc, prec, *fields[k % 3], t, i.dt, 1 + k % 2)
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        got.append(t)
    assert torch.equal(*got)
