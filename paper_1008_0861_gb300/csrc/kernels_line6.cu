// Instantiations and launch configuration of the long-line kernel
// (line6_kernel.cuh): FP32 state with FP32 or FP16 face coefficients, and FP64.
#include "line6_kernel.cuh"

namespace aniso {

// FP32: lines of 2048 < n <= 4096 cells (multiples of the 16-byte vector): a
// team of P = 128 lanes (4 to 8 chunks of 4 cells a lane), `lines` (2 or 4)
// lines per block: 16-byte pieces in the transposed store with four, 8-byte
// ones with two (and then two blocks per SM).  FP64: lines line4 is too short
// for (1024 < n <= 4096), P = 128 lanes (4 to 16 chunks of 2 cells), two
// lines per block, 16-byte pieces.  The shared memory holds the three per-line
// arrays of line4 plus the team exchange area.
bool line6_config(int prec, int coef_fp16, int n, int *team, int *lines_per_block, int *nthreads, size_t *smem,
                  int lines)
{
    const int P = 128;
    const bool d = prec == PREC_FP64;
    const int N = d ? 2 : 4, L = d ? 2 : lines;
    if (n % N != 0 || n <= (d ? MAX_LINE4_FP64 : MAX_LINE2_TRANSPOSED) || n > 4096) return false;
    if (coef_fp16 && (d || n % 8 != 0)) return false;
    if (lines != 2 && lines != 4) return false;
    const int m = n / N;
    const size_t sm = (size_t)L * (3 * (size_t)m * 16 + 4 * (size_t)P * (d ? sizeof(double) : sizeof(float)));
    if (sm > SMEM_LIMIT - 2048) return false;
    *team = P;
    *lines_per_block = L;
    *nthreads = P * L;
    *smem = sm;
    return true;
}

cudaError_t launch_line6(int prec, int coef_fp16, const Line2Args &a, int nblocks, int nthreads, size_t smem, cudaStream_t s)
{
    const bool vl = a.limiter == LIM_VANLEER;
    if (prec == PREC_FP64)
        return vl ? launch_line_kernel(line6_kernel<double, double, true>, a, nblocks, nthreads, smem, s)
                  : launch_line_kernel(line6_kernel<double, double, false>, a, nblocks, nthreads, smem, s);
    if (coef_fp16)
        return vl ? launch_line_kernel(line6_kernel<float, __half, true>, a, nblocks, nthreads, smem, s)
                  : launch_line_kernel(line6_kernel<float, __half, false>, a, nblocks, nthreads, smem, s);
    return vl ? launch_line_kernel(line6_kernel<float, float, true>, a, nblocks, nthreads, smem, s)
              : launch_line_kernel(line6_kernel<float, float, false>, a, nblocks, nthreads, smem, s);
}

}  // namespace aniso
