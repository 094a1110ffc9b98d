// Instantiations and launch configuration of the cluster line kernel
// (line7_kernel.cuh): FP32 state, plain (gamma in shared or tensor memory) or
// compensated (shared memory), FP32 or FP16 face coefficients.
#include "line7_kernel.cuh"

namespace aniso {

// n = CS * np with CS = 1, 2, 4 or 8 blocks a cluster.  The plain state in its
// tensor-memory form (tmem): np = 1024 and eight lines a block up to 8192
// cells.  Otherwise, and for 16384: np = 2048 (1024 when n is not a multiple of
// it) and four lines.
static int pieces7(int n, bool tmem, int *np)
{
    *np = tmem && n <= 8192 ? 1024 : n % 2048 == 0 ? 2048 : 1024;
    if (n % *np != 0) return 0;
    const int c = n / *np;
    return c == 1 || c == 2 || c == 4 || c == 8 ? c : 0;
}
bool line7_config(int prec, int coef_fp16, int n, int *cs, int *nthreads, size_t *smem, bool tmem)
{
    if (prec != PREC_FP32 || n <= 0) return false;
    (void)coef_fp16;
    int np;
    const int c = pieces7(n, tmem, &np);
    if (!c) return false;
    const int lines = tmem && np == 1024 ? 8 : 4;
    *cs = c;
    *nthreads = L7_THREADS;
    *smem = (size_t)lines * (tmem ? 2 : 3) * (size_t)(np / 4) * 16 + (lines == 8 ? 64 : 0);
    return true;
}

template <typename Kern>
static cudaError_t run7(Kern kern, const Line2Args &a, int lines, int cs, size_t smem, cudaStream_t s)
{
    const int groups = (a.one.nlines + lines - 1) / lines;
    // (never chained: launches of 100 us and more gain nothing, 4096^2 lost 0.4 %)
    return launch_line_kernel(kern, a, groups * cs, L7_THREADS, smem, s, cs);
}

// Segments of 8 chunks (pieces of 2048 cells) or 4 (1024), each its own kernel
// with every loop unrolled.  us a pass with the run-time segment length / with
// this: 4096^2 FP32, 4 steps 845 / 750 (FP16 coefficients 745 / 666); 8192^2,
// 2 steps 1585 / 1447; compensated with FP16 coefficients 2279 / 2188; 1024^2
// compensated, 4 steps 107 / 101.
template <bool K, bool TM, bool TO, int U, int WPL>
static cudaError_t launch7u(int coef_fp16, const Line2Args &a, int cs, size_t smem, cudaStream_t s)
{
    const bool vl = a.limiter == LIM_VANLEER;
    constexpr int L = L7_THREADS / (32 * WPL);
    if (coef_fp16)
        return vl ? run7(line7_kernel<__half, true, K, TM, TO, U, WPL>, a, L, cs, smem, s)
                  : run7(line7_kernel<__half, false, K, TM, TO, U, WPL>, a, L, cs, smem, s);
    return vl ? run7(line7_kernel<float, true, K, TM, TO, U, WPL>, a, L, cs, smem, s)
              : run7(line7_kernel<float, false, K, TM, TO, U, WPL>, a, L, cs, smem, s);
}
template <bool K, bool TM, bool TO>
static cudaError_t launch7k(int coef_fp16, const Line2Args &a, int cs, size_t smem, cudaStream_t s)
{
    if constexpr (TM)
        return a.one.n / cs == 2048 ? launch7u<K, TM, TO, 8, 2>(coef_fp16, a, cs, smem, s)
                                    : launch7u<K, TM, TO, 8, 1>(coef_fp16, a, cs, smem, s);
    else
        return a.one.n / cs == 2048 ? launch7u<K, TM, TO, 8, 2>(coef_fp16, a, cs, smem, s)
                                    : launch7u<K, TM, TO, 4, 2>(coef_fp16, a, cs, smem, s);
}

cudaError_t launch_line7(int coef_fp16, const Line2Args &a, int cs, size_t smem, cudaStream_t s)
{
    if (a.jobs || (a.one.n != 2048 * cs && a.one.n != 1024 * cs)) return cudaErrorInvalidValue;
    const bool k = a.one.TinLo != nullptr;
    if (k && (!a.one.ToutLo)) return cudaErrorInvalidValue;
    // with args.tmem: the plain state keeps gamma and T_old in tensor memory
    // (two shared arrays, three blocks an SM); the compensated state keeps
    // T_old's hi and lo there (three shared arrays, two blocks an SM)
    if (k)
        return a.tmem ? launch7k<true, false, true>(coef_fp16, a, cs, smem, s)
                      : launch7k<true, false, false>(coef_fp16, a, cs, smem, s);
    return a.tmem ? launch7k<false, true, true>(coef_fp16, a, cs, smem, s)
                  : launch7k<false, false, false>(coef_fp16, a, cs, smem, s);
}

}  // namespace aniso
