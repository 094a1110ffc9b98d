// Instantiations of the warp-per-line kernel with the chunk rounds as a
// constant (VC), FP32 van Leer in the shared-memory form: batched launches,
// grids alone with three rounds of loads in flight, and the
// temperature-dependent form.  us an update with the rounds from the job / as a
// constant: 128^2 4.21 / 3.28, 512^2 4.56 / 3.54, 768^2 7.48 / 6.45, 1024^2
// 9.02 / 8.34; field + T^2.5 step at 1024^2 39.3 / 37.8.
#include "line4_rounds.cuh"

namespace aniso {

template <int VC> struct Plain {
    static cudaError_t run(int coef_fp16, const Line2Args &a, int nblocks, int nthreads, size_t smem, cudaStream_t s)
    {
        return coef_fp16 ? launch_line_kernel(line4_kernel<float, __half, true, false, false, false, false, 1, false, VC>, a,
                                      nblocks, nthreads, smem, s)
                         : launch_line_kernel(line4_kernel<float, float, true, false, false, false, false, 1, false, VC>, a,
                                      nblocks, nthreads, smem, s);
    }
};
template <int VC> struct Alone {
    static cudaError_t run(int coef_fp16, const Line2Args &a, int nblocks, int nthreads, size_t smem, cudaStream_t s)
    {
        if (a.one.chi_alpha != 0.0)
            return launch_line_kernel(line4_kernel<float, float, true, false, true, false, false, 3, false, VC>, a, nblocks,
                              nthreads, smem, s);
        return coef_fp16 ? launch_line_kernel(line4_kernel<float, __half, true, false, false, false, false, 3, false, VC>, a,
                                      nblocks, nthreads, smem, s)
                         : launch_line_kernel(line4_kernel<float, float, true, false, false, false, false, 3, false, VC>, a,
                                      nblocks, nthreads, smem, s);
    }
};

cudaError_t launch_line4_rounds(int coef_fp16, bool alone, const Line2Args &a, int nblocks, int nthreads, size_t smem,
                                cudaStream_t s)
{
    return alone ? by_rounds<Alone>(coef_fp16, a, nblocks, nthreads, smem, s)
                 : by_rounds<Plain>(coef_fp16, a, nblocks, nthreads, smem, s);
}

}  // namespace aniso
