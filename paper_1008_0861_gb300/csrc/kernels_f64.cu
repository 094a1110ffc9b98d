// FP64 instantiations of the sweep kernels.
#include "line2_kernel.cuh"

namespace aniso {

cudaError_t launch_line_f64(const LineArgs &a, int nblocks, int nthreads, size_t smem, cudaStream_t s)
{
    cudaError_t err = allow_smem(line_sweep_kernel<double, double, false>, smem);
    if (err != cudaSuccess) return err;
    line_sweep_kernel<double, double, false><<<nblocks, nthreads, smem, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_col_f64(const ColArgs &a, int nblocks, int nthreads, size_t smem, cudaStream_t s)
{
    cudaError_t err = allow_smem(col_sweep_kernel<double, double, false>, smem);
    if (err != cudaSuccess) return err;
    col_sweep_kernel<double, double, false><<<nblocks, nthreads, smem, s>>>(a);
    return cudaGetLastError();
}


cudaError_t launch_line2_f64(const Line2Args &a, int nblocks, int nthreads, size_t smem, cudaStream_t s)
{
    cudaError_t err = allow_smem(line2_kernel<double, double, false>, smem);
    if (err != cudaSuccess) return err;
    line2_kernel<double, double, false><<<nblocks, nthreads, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace aniso
