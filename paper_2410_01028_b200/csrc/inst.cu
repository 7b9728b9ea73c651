// Instantiations of the pass kernel; compiled once per ASD_M in 1..9 and 16 (the row count of a prefill pass).
#include "pass.cuh"

#ifndef ASD_M
#error "compile with -DASD_M=<rows>"
#endif

namespace asd {

#define ASD_CAT2(a, b) a##b
#define ASD_CAT(a, b) ASD_CAT2(a, b)

// The one-row pass exists in two variants: activations handed over through tagged words (p.use_ll) or through
// plain buffers behind the grid barrier. Each of them for heads of 256, 128, 64 and smaller ones.
template <bool LL>
static const void* pass_of(int head_dim) {
    if (head_dim == 128) return reinterpret_cast<const void*>(&pass_kernel<ASD_M, LL, 128>);
    if (head_dim == 256) return reinterpret_cast<const void*>(&pass_kernel<ASD_M, LL, 256>);
    if (head_dim == 64) return reinterpret_cast<const void*>(&pass_kernel<ASD_M, LL, 64>);
    return reinterpret_cast<const void*>(&pass_kernel<ASD_M, LL, 0>);
}

cudaError_t ASD_CAT(launch_pass_m, ASD_M)(const PassParams& p, int grid, size_t smem, cudaStream_t s) {
    void* args[] = {const_cast<PassParams*>(&p)};
    const void* fn = pass_of<false>(p.head_dim);
#if ASD_M == 1
    if (p.use_ll) fn = pass_of<true>(p.head_dim);
#else
    if (p.use_ll) return cudaErrorInvalidValue;
#endif
    return cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(kPassThreads), args, smem, s);
}

// opt every instantiation in to large dynamic shared memory
cudaError_t ASD_CAT(configure_m, ASD_M)(int max_smem) {
    for (int head_dim : {256, 128, 64, 0}) {
        cudaError_t e = cudaFuncSetAttribute(pass_of<false>(head_dim), cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
        if (e != cudaSuccess) return e;
#if ASD_M == 1
        if ((e = cudaFuncSetAttribute(pass_of<true>(head_dim), cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem)) != cudaSuccess) return e;
#endif
    }
    return cudaSuccess;
}

}  // namespace asd
