// Multi-step backward-Euler kernel of the heat operator with a 64-bit integer
// state (device code in pit_fixed.cuh).
#include "pit_fixed.cuh"

namespace pit {

cudaError_t fixed_init(int bytes)
{
    const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    const cudaError_t e = cudaFuncSetAttribute((const void *)fixed_kernel<false>, attr, bytes);
    return e != cudaSuccess ? e : cudaFuncSetAttribute((const void *)fixed_kernel<true>, attr, bytes);
}

cudaError_t fixed_launch(const StepArgs &a, dim3 grid, dim3 block, size_t smem, cudaStream_t s, bool xg)
{
    if (xg) fixed_kernel<true><<<grid, block, smem, s>>>(a);
    else fixed_kernel<false><<<grid, block, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace pit
