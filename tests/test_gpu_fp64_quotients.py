"""The FP64 reciprocal and quotient of the line kernels against CUDA's own
1 / x and a / b: within one unit in the last place everywhere in their range,
and, with the remainder step, the rounded values but for those next to the
middle of two numbers."""
import ctypes

import numpy as np
import pytest

from gpu_build import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "line4_kernel.cuh"
using namespace aniso;
__global__ void all(const double *a, const double *b, double *out, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double y = drcp_approx(b[i]);
    out[i] = y;
    out[n + i] = drcp(b[i]);
    out[2 * n + i] = dquot(a[i], b[i], y);
    out[3 * n + i] = 1.0 / b[i];
    out[4 * n + i] = a[i] / b[i];
}
extern "C" int run(const double *a, const double *b, double *out, int n, void *stream)
{
    all<<<(n + 255) / 256, 256, 0, (cudaStream_t)stream>>>(a, b, out, n);
    return (int)cudaGetLastError();
}
"""


def _operands(n, rng):
    mant = 1.0 + rng.rand(2, n)
    mant[:, : n // 8] = 2.0 - np.ldexp(rng.randint(1, 4, (2, n // 8)), -52)  # all ones, and the next two
    mant[1, n // 8 : n // 4] = 1.0 + np.ldexp(rng.randint(0, 4, n // 8), -52)
    exp_b = rng.randint(-1021, 1021, n)  # 1 / b and b normal
    exp_q = np.clip(rng.randint(-900, 900, n), -960 - exp_b, 1020 - exp_b)
    exp_q = np.clip(exp_q, -960, 1020)  # quotient and remainder normal
    b = np.ldexp(mant[1], exp_b)
    a = np.ldexp(mant[0], np.clip(exp_b + exp_q, -960, 1022))
    sign = 1 - 2 * rng.randint(0, 2, (2, n))
    return a * sign[0], b * sign[1]


def _ulps(got, want):
    return np.abs(got.view(np.int64) - want.view(np.int64))


def test_reciprocals_and_quotients(lib, tmp_path):
    import torch
    probe = build(SOURCE, tmp_path)
    n = 1 << 22
    vp = ctypes.c_void_p
    for seed in range(3):
        a, b = _operands(n, np.random.RandomState(seed))
        q = np.abs(a / b)
        a = np.where((q > 2.0 ** -960) & (q < 2.0 ** 1020), a, b)  # (the others: a quotient of 1)
        da, db = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
        out = torch.zeros(5, n, dtype=torch.float64, device="cuda")
        rc = probe.run(vp(da.data_ptr()), vp(db.data_ptr()), vp(out.data_ptr()), n,
                       vp(torch.cuda.current_stream().cuda_stream))
        assert rc == 0
        y, r, d, inv, quo = out.cpu().numpy()
        assert np.array_equal(inv, 1.0 / b) and np.array_equal(quo, a / b)
        assert _ulps(y, inv).max() <= 1
        for got, want in ((r, inv), (d, quo)):
            off = _ulps(got, want)
            assert off.max() <= 1
            # (operands at random lie that close to a middle once in 2^50; the constructed ones are an eighth)
            assert not off[n // 4 :].any()
