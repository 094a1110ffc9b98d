// Instantiations of the warp-per-line kernel for lines of any length and arrays
// of any alignment (RAG).
#include "line4_kernel.cuh"

namespace aniso {

template <typename R, typename C, bool VL, int RING>
static cudaError_t run4r(const Line2Args &a, int nblocks, int nthreads, size_t smem, cudaStream_t s)
{
    auto kern = line4_kernel<R, C, VL, false, false, false, false, RING, true>;
    return launch_line_kernel(kern, a, nblocks, nthreads, smem, s);
}

cudaError_t launch_line4_ragged(int prec, int coef_fp16, const Line2Args &a, int nblocks, int nthreads, size_t smem,
                                cudaStream_t s)
{
    const bool vl = a.limiter == LIM_VANLEER;
    if (prec == PREC_FP64)
        return vl ? run4r<double, double, true, 1>(a, nblocks, nthreads, smem, s)
                  : run4r<double, double, false, 1>(a, nblocks, nthreads, smem, s);
    if (coef_fp16)
        return vl ? run4r<float, __half, true, 1>(a, nblocks, nthreads, smem, s)
                  : run4r<float, __half, false, 1>(a, nblocks, nthreads, smem, s);
    // (as launch_line4: two rounds of loads in flight where a grid alone leaves the SMs few warps)
    if (vl && !a.jobs && (long)nblocks * nthreads <= 152L * 32 * 8)
        return run4r<float, float, true, 2>(a, nblocks, nthreads, smem, s);
    return vl ? run4r<float, float, true, 1>(a, nblocks, nthreads, smem, s)
              : run4r<float, float, false, 1>(a, nblocks, nthreads, smem, s);
}

}  // namespace aniso
