// line4_rounds.cuh -- host dispatch of the warp-per-line kernel's forms whose
// chunk rounds are a template constant (Line2Args::rounds, 4 to 8: the default
// segments of lines up to 1024 cells).
#pragma once
#include "line4_kernel.cuh"

namespace aniso {

template <template <int> class F, int LAST = 8>
static cudaError_t by_rounds(int coef_fp16, const Line2Args &a, int nblocks, int nthreads, size_t smem, cudaStream_t s)
{
    switch (a.rounds) {
    case 4: return F<4>::run(coef_fp16, a, nblocks, nthreads, smem, s);
    case 5: return F<5>::run(coef_fp16, a, nblocks, nthreads, smem, s);
    case 6: return F<6>::run(coef_fp16, a, nblocks, nthreads, smem, s);
    case 7: return F<7>::run(coef_fp16, a, nblocks, nthreads, smem, s);
    case 8:
        if constexpr (LAST == 8) return F<8>::run(coef_fp16, a, nblocks, nthreads, smem, s);
        else return cudaErrorInvalidValue;
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace aniso
