// Instantiations of the warp-per-line kernel's tensor-memory form with the
// chunk rounds as a constant (VC), FP32 van Leer, 4 to 7 rounds (8 spilled: such
// lines keep the run-time form).
#include "line4_rounds.cuh"

namespace aniso {

template <int VC> struct Tensor {
    static cudaError_t run(int coef_fp16, const Line2Args &a, int nblocks, int nthreads, size_t smem, cudaStream_t s)
    {
        return coef_fp16 ? launch_line_kernel(line4_kernel<float, __half, true, false, false, false, true, 1, false, VC>, a,
                                      nblocks, nthreads, smem, s)
                         : launch_line_kernel(line4_kernel<float, float, true, false, false, false, true, 1, false, VC>, a,
                                      nblocks, nthreads, smem, s);
    }
};

cudaError_t launch_line4_rounds_tm(int coef_fp16, const Line2Args &a, int nblocks, int nthreads, size_t smem,
                                   cudaStream_t s)
{
    return by_rounds<Tensor, 7>(coef_fp16, a, nblocks, nthreads, smem, s);
}

}  // namespace aniso
