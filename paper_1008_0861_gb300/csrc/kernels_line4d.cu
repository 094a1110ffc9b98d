// Instantiations of the warp-per-line kernel's 3-D form with the chunk rounds as
// a constant (VC), FP32 van Leer, 4 or 5 rounds (256^3, 4 steps: 1214 -> 1135 us;
// with 6 and more the unrolled form spills and loses 3-6 %).
#include "line4_rounds.cuh"

namespace aniso {

template <int VC> struct Cube {
    static cudaError_t run(int coef_fp16, const Line2Args &a, int nblocks, int nthreads, size_t smem, cudaStream_t s)
    {
        return coef_fp16 ? launch_line_kernel(line4_kernel<float, __half, true, true, false, false, false, 1, false, VC>, a,
                                      nblocks, nthreads, smem, s)
                         : launch_line_kernel(line4_kernel<float, float, true, true, false, false, false, 1, false, VC>, a,
                                      nblocks, nthreads, smem, s);
    }
};

cudaError_t launch_line4_rounds_3d(int coef_fp16, const Line2Args &a, int nblocks, int nthreads, size_t smem,
                                   cudaStream_t s)
{
    return a.rounds == 4   ? Cube<4>::run(coef_fp16, a, nblocks, nthreads, smem, s)
           : a.rounds == 5 ? Cube<5>::run(coef_fp16, a, nblocks, nthreads, smem, s)
                           : cudaErrorInvalidValue;
}

}  // namespace aniso
