// Prompt processing as dense products on the tensor cores (the first step of inference in Section 3.2: the
// whole prompt goes through M once, which fills the KV cache and yields every row's per-sublayer cosine
// similarity, the summands of C_l).
//
// With hundreds of rows the sublayer products are dense contractions, so they run as tcgen05 GEMMs: operand
// tiles staged in shared memory by TMA (128-byte swizzle), accumulators in tensor memory, one elected thread
// issuing tcgen05.mma, four epilogue warps reading the accumulators back with tcgen05.ld. Causal attention
// over the prompt is a flash-style tcgen05 kernel (prefill_attn.cu). Row-wise work (embedding, RMSNorm, residual add with
// the cosine sums) runs one CTA per row.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "gemm_plan.h"

namespace asd {

enum GemmEpilogue : int {
    kGemmF32 = 0,     // C[r, n] fp32
    kGemmQkv = 1,     // rotary embedding, bf16, queries to q, keys and values appended to the KV cache
    kGemmSwiglu = 2,  // columns alternate gate_i, up_i: t[r, i] = bf16(silu(gate_i) * up_i)
};

// What the epilogue of one GEMM does with the accumulators. Row r of the product is prompt row r of this chunk.
struct GemmEpi {
    int mode;
    int* err;  // device error words shared with the pass kernel (word 0 = code)
    int w_static;  // no kernel in flight writes W: its first tiles may be requested before the kernel in front has ended
    // kGemmF32
    float* c;
    int ldc;
    size_t c_part_stride;  // floats between the parts of a product whose reduction dimension is cut (the caller adds them in order)
    // kGemmQkv: columns are [q | k | v]; inside every q and k head the rotary partners (j, j + head_dim/2) are
    // neighbours (2j, 2j+1); v columns are in natural order. Row r sits at position pos0 + r.
    __nv_bfloat16 *q, *k_cache, *v_cache;
    const float *rope_cos, *rope_sin;
    int pos0, d_model, kv_dim, head_dim;
    // kGemmSwiglu
    __nv_bfloat16* t;
    int ldt;
};

cudaError_t configure_prefill(int max_smem);

// the plan of C[M, N] = A[M, K] * W[N, K]^T on this device; max_parts > 1 for kGemmF32 only (parts c_part_stride apart)
GemmPlan plan_gemm(int M, int N, int K, int max_parts);
// bf16 operands described by 2-D tensor maps (128-byte swizzle, A in boxes of 64 elements x 128 rows, W in boxes of 64 x
// w_box()), fp32 accumulation
cudaError_t launch_gemm_tn(const CUtensorMap& tm_a, const CUtensorMap& tm_w, int M, int N, int K, const GemmPlan& plan, const GemmEpi& ep, cudaStream_t s);

cudaError_t launch_clear_status(int* status /* 8 words */, cudaStream_t s);

// x[r, :] = embedding row of tokens[r] (fp32); xn[r, :] = bf16(RMSNorm(x[r]) * gain)
cudaError_t launch_embed_norm(const int* tokens, int n_rows, int d, int vocab, const __nv_bfloat16* embed, const __nv_bfloat16* gain,
                              float eps, float* x, __nv_bfloat16* xn, cudaStream_t s);

// y = x + c (in place in x; c is the sum of `parts` buffers, added in order), cos_out[r] = <x, y> / (|x| |y|) (Section 3.2), and, when gain is given,
// xn[r, :] = bf16(RMSNorm(y) * gain) for the next sublayer
cudaError_t launch_resid_norm(int n_rows, int d, float* x, const float* c, int parts, size_t part_stride, const __nv_bfloat16* gain, float eps, __nv_bfloat16* xn,
                              float* cos_out, cudaStream_t s);

// sumcos[b] += sum over rows of cos_rows[b * stride + r], rows in a fixed order, double precision; host: a copy in pinned memory
cudaError_t launch_sumcos(const float* cos_rows, int stride, int n_rows, int n_sub, double* sumcos, double* host, cudaStream_t s);

// causal attention of prompt rows [0, n_rows) at positions pos0 + r over keys 0 .. pos0 + r of the cache. Tensor maps (bf16,
// 128-byte swizzle): the queries [rows, d_model] in boxes of 64 columns x 128 rows, the caches [max_seq, kv_dim] in boxes of
// 64 columns x 64 keys. head_dim 64 or 128. totals: scratch of n_rows (rounded up to
// whole tiles of 128) x d_model floats, 32-byte aligned.
cudaError_t launch_flash_prefill(const CUtensorMap& tm_q, const CUtensorMap& tm_k, const CUtensorMap& tm_v, __nv_bfloat16* out, float* totals,
                                 int n_rows, int pos0, int d_model, int head_dim, int n_heads, int n_kv_heads, float scale, int* err, cudaStream_t s);
cudaError_t configure_prefill_attention();

}  // namespace asd
