// Shared declarations of the CUDA library: kernel parameter blocks and small device helpers.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace asd {

constexpr int kMaxRows = 9;        // rows of the stand-alone fused GEMV: max draft length 8, plus the last accepted token

struct PassParams;

// launchers, one translation unit per row count (inst.cu compiled with -DASD_M=1..9)
#define ASD_DECLARE_LAUNCHERS(M)                                                                                 \
    cudaError_t launch_pass_m##M(const PassParams& p, int grid, size_t smem, cudaStream_t s);                    \
    cudaError_t configure_m##M(int max_smem);
ASD_DECLARE_LAUNCHERS(1)
ASD_DECLARE_LAUNCHERS(2)
ASD_DECLARE_LAUNCHERS(3)
ASD_DECLARE_LAUNCHERS(4)
ASD_DECLARE_LAUNCHERS(5)
ASD_DECLARE_LAUNCHERS(6)
ASD_DECLARE_LAUNCHERS(7)
ASD_DECLARE_LAUNCHERS(8)
ASD_DECLARE_LAUNCHERS(9)
cudaError_t launch_pass_m16(const PassParams& p, int grid, size_t smem, cudaStream_t s);
cudaError_t configure_m16(int max_smem);

// ---------------------------------------------------------------- launch helper
// Launches a kernel that begins with pdl_wait(): its launch and its CTAs' start overlap the end of the kernel before it.
template <class... P, class... A>
inline cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, int cluster, A&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid, cfg.blockDim = block, cfg.dynamicSmemBytes = smem, cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = (unsigned)cluster, at[1].val.clusterDim.y = 1, at[1].val.clusterDim.z = 1;
    cfg.attrs = at, cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<A&&>(args)...);
}

// ---------------------------------------------------------------- device helpers
__device__ __forceinline__ float bf_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf_hi(uint32_t u) { return __uint_as_float(u & 0xFFFF0000u); }

// Programmatic dependent launch: a kernel that was launched with the attribute may start while the one before it on the
// stream is still running (once all of that one's CTAs have asked for it or ended) and waits here for its end and its
// writes before it reads or writes anything itself. Without the attribute both do nothing.
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

}  // namespace asd
