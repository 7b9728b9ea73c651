// Kernels of the dense prompt path (see prefill.h).
#include "prefill.h"

#include <algorithm>

#include "common.cuh"
#include "ring.cuh"
#include "tcgen05.cuh"

namespace asd {

// ============================================================================================ GEMM epilogues
// One call per (row, 32 consecutive columns starting at col0) with the fp32 accumulators in v.
__device__ __forceinline__ void epi_f32(const GemmEpi& ep, int row, int col0, int N, const float (&v)[32], int part) {
    float* dst = ep.c + (size_t)part * ep.c_part_stride + (size_t)row * ep.ldc + col0;
    if (col0 + 32 <= N && (((ep.ldc | ep.c_part_stride) * 4) | ((uintptr_t)ep.c & 31)) % 32 == 0) {
        uint32_t w[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) w[i] = __float_as_uint(v[i]);
#pragma unroll
        for (int i = 0; i < 4; ++i) st_global_v8(dst + 8 * i, w + 8 * i);
    } else if (col0 + 32 <= N && (ep.ldc & 3) == 0) {
#pragma unroll
        for (int i = 0; i < 8; ++i) reinterpret_cast<float4*>(dst)[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    } else {
#pragma unroll
        for (int i = 0; i < 32; ++i)
            if (col0 + i < N) dst[i] = v[i];
    }
}

__device__ __forceinline__ void epi_swiglu(const GemmEpi& ep, int row, int col0, int N, const float (&v)[32]) {
    __nv_bfloat16* dst = ep.t + (size_t)row * ep.ldt + (col0 >> 1);
    float t[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const float g = v[2 * i], u = v[2 * i + 1];
        t[i] = g / (1.0f + expf(-g)) * u;
    }
    if (col0 + 32 <= N && (ep.ldt & 7) == 0) {
        uint32_t w[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) w[i] = pack_bf16(t[2 * i], t[2 * i + 1]);
        if ((ep.ldt & 15) == 0) {
            st_global_v8(dst, w);
        } else {
            reinterpret_cast<uint4*>(dst)[0] = make_uint4(w[0], w[1], w[2], w[3]);
            reinterpret_cast<uint4*>(dst)[1] = make_uint4(w[4], w[5], w[6], w[7]);
        }
    } else {
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (col0 + 2 * i + 1 < N) dst[i] = __float2bfloat16_rn(t[i]);
    }
}

// head_dim is 64 or 128 and the q, k and v column ranges start at multiples of head_dim, so the 32 columns
// belong to one head of one of q, k, v, and all rows and row parts are 32-byte aligned.
__device__ __forceinline__ void epi_qkv(const GemmEpi& ep, int row, int col0, int N, const float (&v)[32]) {
    if (col0 >= N) return;
    const int pos = ep.pos0 + row;
    const int hd = ep.head_dim, half = hd >> 1;
    if (col0 >= ep.d_model + ep.kv_dim) {  // values: natural order, no rotation
        __nv_bfloat16* dst = ep.v_cache + (size_t)pos * ep.kv_dim + (col0 - ep.d_model - ep.kv_dim);
        uint32_t w[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) w[i] = pack_bf16(v[2 * i], v[2 * i + 1]);
        st_global_v8(dst, w);
        st_global_v8(dst + 16, w + 8);
        return;
    }
    const bool is_q = col0 < ep.d_model;
    const int c = is_q ? col0 : col0 - ep.d_model;
    const int head = c / hd, j0 = (c - head * hd) >> 1;  // pairs j0 .. j0+15 of this head
    const float4* cs = reinterpret_cast<const float4*>(ep.rope_cos + (size_t)pos * half + j0);
    const float4* sn = reinterpret_cast<const float4*>(ep.rope_sin + (size_t)pos * half + j0);
    float lo[16], hi[16];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float4 c4 = cs[i], s4 = sn[i];
        const float cc[4] = {c4.x, c4.y, c4.z, c4.w}, ss[4] = {s4.x, s4.y, s4.z, s4.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float va = v[2 * (4 * i + u)], vb = v[2 * (4 * i + u) + 1];
            lo[4 * i + u] = va * cc[u] - vb * ss[u];
            hi[4 * i + u] = vb * cc[u] + va * ss[u];
        }
    }
    __nv_bfloat16* base = is_q ? ep.q + (size_t)row * ep.d_model : ep.k_cache + (size_t)pos * ep.kv_dim;
    __nv_bfloat16* dlo = base + (size_t)head * hd + j0;
    __nv_bfloat16* dhi = dlo + half;
    uint32_t w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = pack_bf16(lo[2 * i], lo[2 * i + 1]);
    st_global_v8(dlo, w);
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = pack_bf16(hi[2 * i], hi[2 * i + 1]);
    st_global_v8(dhi, w);
}

// ============================================================================================ the GEMM
// Persistent units (CG = 1: one SM; CG = 2: a cluster of two SMs) walk the 128 * CG x BN tiles of the product, row tiles
// fastest. Warp 0 is the TMA producer, warp 1 issues the MMAs and owns the tensor-memory allocation,
// warps 2-9 are the epilogue (warp w reads lanes 32 * (w % 4) .. + 31 of tensor memory, the quarter its position in the
// warp group gives it access to, and every second 32 columns: with four warps the epilogue of the last tile, which nothing covers, was longer:
// gate/up of 512 rows of the 7B width 68.4 -> 64.4 us in the prompt's chain, of 1023 rows 2048 wide 41.3 -> 37.0). Four warps where a tile has 32
// columns, and where rows of C are no multiple of 32 bytes: their stores bound the tile, and eight warps get in each other's way (pair tiles, 150 products
// with N odd: 1-3 % slower with eight than with four; N an odd multiple of 4: 1 %). The accumulator is double-buffered in tensor memory (2 x BN columns), so the epilogue
// of a tile runs while the MMAs of the next tile are already filling the other buffer. Barriers: full[s] (TMA bytes landed
// in stage s), empty[s] (the MMAs reading stage s have finished: tcgen05.commit), acc_full[b] (all MMAs of the tile in
// buffer b have finished), acc_empty[b] (the epilogue warps have read buffer b). Ragged edges: TMA fills out-of-range
// rows and reduction elements with zeros; the epilogue skips rows >= M and columns >= N. Every wait is bounded; after
// a failed wait the roles fall through to the common exit. Nothing outlives the kernel there: the MMA warp waits for its
// last MMA (drained), whatever the other roles do, and when a producer or the MMA warp has given up (abandoned, set in both
// CTAs of a pair) the copies that are still in flight land before shared and tensor memory are given back.
//
// What bounds it: on single SMs the operands' way from L2: a 128 x 256 tile wants 48 KB per 64 elements of the reduction and
// takes 0.35 us for them (139 bytes per ns and SM) where its MMAs take 0.27. Two SMs sharing a 256 x 256 tile (cta_group::2,
// CG = 2: each stages its 128 rows of A and half of the rows of W and keeps its 128 rows of the accumulator) want 32 KB each
// and take 0.315 us. Pairs that fill the chip for rounds are bound by the tensor core (93 % of active cycles at 2048 rows)
// and by the power limit, which takes the clock down (2048 x 22016 x 4096: 251 us alone on a cool chip, 294-302 us back to
// back; on single SMs 337 us); tiles of up to 64 columns by the issue of a k-block (0.14 us: wait, four MMAs, commit; 0.28 us when one lane of a divergent warp issued
// them). With CG = 2 the leader (rank 0) issues the MMAs; full[s] lives in the leader and counts both CTAs' bytes;
// empty[s] and acc_full[b] are signalled in both CTAs by multicast commits; acc_empty[b] lives in the leader and counts
// the epilogue warps of both.
//
// Units and tiles rarely divide evenly, so the host picks the kind of unit, the tile width and, for the products whose
// consumer adds them up (fp32 output), the number of parts the reduction dimension is cut into by the time they take
// over the rounds (gemm_plan.h). Cutting the tiles of a last round with an exchange of the parts through L2 inside the
// kernel (last arriver adds) was measured: 8-10 us per exchange, more than the part of a round it saves.
constexpr int kGemmThreads = 64 + 32 * 8;  // at most (see launch_gemm_tn)
static int g_gemm_ctas = 148;  // persistent CTAs per launch: the SM count of the device (set by configure_prefill)

// BN = 0: the width is a parameter of the launch (a multiple of 32).
template <int BN, int CG>
struct GemmCfg {
    static constexpr uint32_t kABytes = kGemmBM * kGemmBK * 2;
    static constexpr uint32_t kWRowBytes = kGemmBK * 2;
    static constexpr size_t kRing = BN ? 6 * (kABytes + BN / CG * kWRowBytes) : 196608;  // bytes of all stages (BN = 0: at most)
    static constexpr size_t kSmem = kRing + 1024 /* alignment */ + 256 /* barriers */;
    static constexpr int kMaxStages = BN ? 6 : 8;
    static constexpr int kAccStride = BN ? BN : 256;  // columns from one accumulator to the next
};

// The work of one launch: items (tile, part of the reduction dimension), tiles fastest, dealt round robin to the units.
struct GemmWork {
    int m_tiles, tiles, parts, bn, wide, narrow;  // (see GemmPlan; tiles: all of them)
};
struct GemmItem {
    int part, kb0, kb1;
    int m, n0, width;  // row of tiles, first column and columns
};
// item `local` of unit `unit`; false when there is none
__device__ __forceinline__ bool gemm_item(const GemmWork& w, int num_kb, int unit, int n_units, int local, GemmItem& it) {
    const int item = unit + local * n_units;
    if (item >= w.tiles * w.parts) return false;
    const int tile = item % w.tiles, col = tile / w.m_tiles;  // row tiles vary fastest: units that run together share their weight tile (read once from HBM, then from L2)
    it.part = item / w.tiles, it.m = tile - col * w.m_tiles;
    it.n0 = min(col, w.wide) * w.bn + max(col - w.wide, 0) * w.narrow, it.width = col < w.wide ? w.bn : w.narrow;
    it.kb0 = it.part * num_kb / w.parts, it.kb1 = (it.part + 1) * num_kb / w.parts;
    return true;
}

__device__ __forceinline__ void gemm_epilogue(const GemmEpi& ep, int row, int col0, int N, const float (&v)[32], int part) {
    if (ep.mode == kGemmF32) epi_f32(ep, row, col0, N, v, part);
    else if (ep.mode == kGemmSwiglu) epi_swiglu(ep, row, col0, N, v);
    else epi_qkv(ep, row, col0, N, v);
}

template <int BN, int CG>
__global__ void __launch_bounds__(kGemmThreads, 1)
gemm_tn_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_w, int M, int N, int K, const GemmWork work,
               const GemmEpi ep) {
    using Cfg = GemmCfg<BN, CG>;
    const int bn = BN ? BN : work.bn;
    const uint32_t stage_bytes = Cfg::kABytes + (uint32_t)(bn / CG) * Cfg::kWRowBytes;
    const int kStages = BN ? Cfg::kMaxStages : min(Cfg::kMaxStages, (int)(Cfg::kRing / stage_bytes));
    extern __shared__ unsigned char gemm_smem_raw[];
    unsigned char* base = gemm_smem_raw + ((1024u - (smem_u32(gemm_smem_raw) & 1023u)) & 1023u);
    uint64_t* full = reinterpret_cast<uint64_t*>(base + Cfg::kRing);
    uint64_t* empty = full + Cfg::kMaxStages;
    uint64_t* acc_full = empty + Cfg::kMaxStages;   // [2]
    uint64_t* acc_empty = acc_full + 2;     // [2]
    uint64_t* drained = acc_empty + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drained + 1);
    int* abandoned = reinterpret_cast<int*>(tmem_slot + 1);  // a producer or the MMA warp of this unit has given up
    int* requested = abandoned + 1;                          // [CG], in the leader: k-blocks that each CTA has requested

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = CG == 2 ? (int)cluster_rank() : 0, unit = blockIdx.x / CG, n_units = gridDim.x / CG;
    const int num_kb = (K + kGemmBK - 1) / kGemmBK;
    volatile int* err = ep.err;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], (blockDim.x / 32 - 2) * CG);
        }
        mbar_init(drained, 1);
        *abandoned = 0;
        mbar_fence_init();
    }
    if (warp == 1) {
        if (CG == 2) tmem_alloc_pair(tmem_slot, 512), tmem_relinquish_pair();
        else tmem_alloc(tmem_slot, 512), tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    if (CG == 2) cluster_sync_all();  // both CTAs' barriers exist before either signals the other's
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    pdl_launch_dependents();
    const uint32_t on = elect_one();
    auto give_up = [&]() {  // one lane; the other CTA's word as well
        *abandoned = 1;
        if (CG == 2) st_cluster(cluster_addr(abandoned, rank ^ 1), 1);
    };
    auto load_w = [&](int s, int kb, int n0) {  // announces the bytes of a stage and requests its weights
        mbar_expect_tx_on(&full[s], CG * stage_bytes, CG == 2 ? on & (uint32_t)(rank == 0) : on);  // the bytes of both CTAs
        unsigned char* b_dst = base + (size_t)s * stage_bytes + Cfg::kABytes;
        if (CG == 2) tma_load_2d_pair(b_dst, &tm_w, kb * kGemmBK, n0, cluster_addr(&full[s], 0), on);
        else tma_load_2d_on(b_dst, &tm_w, kb * kGemmBK, n0, &full[s], on);
    };
    int ahead = 0;  // k-blocks of the first item whose weights are requested before the kernel in front has ended
    if (warp == 0 && ep.w_static) {
        GemmItem it;
        if (gemm_item(work, num_kb, unit, n_units, 0, it))
            for (; ahead < kStages && it.kb0 + ahead < it.kb1; ++ahead) load_w(ahead, it.kb0 + ahead, it.n0 + rank * (it.width / CG));
    }
    pdl_wait();  // everything above overlaps the end of the kernel in front

    if (warp == 0) {
        int issued = 0;      // k-blocks requested so far, over all items of this unit
        int s = 0, lap = 0;  // their ring position: issued = lap * kStages + s
        bool ok = true;
        GemmItem it;
        for (int local = 0; ok && gemm_item(work, num_kb, unit, n_units, local, it); ++local) {
            const int m0 = (it.m * CG + rank) * kGemmBM, n0 = it.n0 + rank * (it.width / CG);
            for (int kb = it.kb0; kb < it.kb1; ++kb) {
                if (lap > 0) ok = mbar_wait_warp(&empty[s], (uint32_t)((lap - 1) & 1), err, kErrGemmWait, 0, issued, s, 1);
                if (!ok) break;
                if (issued >= ahead) load_w(s, kb, n0);
                unsigned char* a_dst = base + (size_t)s * stage_bytes;
                if (CG == 2) tma_load_2d_pair(a_dst, &tm_a, kb * kGemmBK, m0, cluster_addr(&full[s], 0), on);
                else tma_load_2d_on(a_dst, &tm_a, kb * kGemmBK, m0, &full[s], on);
                ++issued;
                if (++s == kStages) s = 0, ++lap;
            }
        }
        if (lane == 0) {
            if (!ok) give_up();
            else if (CG == 2)  // the leader's last multicast arrivals at this CTA's barriers come before it leaves
                for (int i = max(0, issued - kStages); i < issued; ++i) mbar_drain(&empty[i % kStages], (uint32_t)((i / kStages) & 1));
            if (CG == 2) st_cluster(cluster_addr(requested + rank, 0), issued);
            else *requested = issued;
        }
    } else if (warp == 1) {
        if (rank == 0) {
            const uint32_t base_addr = smem_u32(base);
            int s = 0, lap = 0;  // ring position of the next k-block
            bool ok = true;
            GemmItem it;
            for (int local = 0; ok && gemm_item(work, num_kb, unit, n_units, local, it); ++local) {
                const int buf = local & 1;
                // the epilogue must have read this buffer's previous tile (item local - 2) before it is overwritten
                if (local >= 2) ok = mbar_wait_warp(&acc_empty[buf], (uint32_t)((local / 2 - 1) & 1), err, kErrGemmWait, 3, local, buf, 4);
                if (!ok) break;
                tc_fence_after();
                const uint32_t tmem_d = tmem + (uint32_t)(buf * Cfg::kAccStride), idesc = umma_idesc_bf16(kGemmBM * CG, it.width);
                for (int kb = it.kb0; kb < it.kb1; ++kb) {
                    ok = mbar_wait_warp(&full[s], (uint32_t)(lap & 1), err, kErrGemmWait, 1, kb, s, 2);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t a_addr = base_addr + (uint32_t)s * stage_bytes;
                    const uint64_t a_desc = umma_desc_k128(a_addr), b_desc = umma_desc_k128(a_addr + Cfg::kABytes);
#pragma unroll
                    for (int k = 0; k < kGemmBK / 16; ++k) {  // 16 elements = 32 bytes further along the swizzled row: +2 in the address field
                        const uint32_t acc = ((kb - it.kb0) | k) != 0 ? 1u : 0u;
                        if (CG == 2) tc_mma_bf16_pair(tmem_d, a_desc + (uint64_t)(2 * k), b_desc + (uint64_t)(2 * k), idesc, acc, on);
                        else tc_mma_bf16(tmem_d, a_desc + (uint64_t)(2 * k), b_desc + (uint64_t)(2 * k), idesc, acc, on);
                    }
                    if (CG == 2) tc_commit_pair(&empty[s], on);  // the stage may be refilled once these MMAs have read it
                    else tc_commit(&empty[s], on);
                    if (++s == kStages) s = 0, ++lap;
                }
                if (CG == 2) tc_commit_pair(&acc_full[buf], on);  // arrives when every MMA issued above has finished
                else tc_commit(&acc_full[buf], on);
            }
            if (CG == 2) tc_commit_pair_here(drained, on);
            else tc_commit(drained, on);
            mbar_drain(drained, 0);
            if (!ok && lane == 0) give_up();
        }
    } else {
        const int quarter = warp & 3, first = (warp - 2) / 4 * 32, step = blockDim.x > 192 ? 64 : 32;  // two warps for each quarter take every second 32 columns
        bool ok = true;
        GemmItem it;
        for (int local = 0; ok && gemm_item(work, num_kb, unit, n_units, local, it); ++local) {
            const int buf = local & 1;
            const int m0 = (it.m * CG + rank) * kGemmBM, n0 = it.n0;
            const int row = m0 + quarter * 32 + lane;
            ok = mbar_wait(&acc_full[buf], (uint32_t)((local / 2) & 1), err, kErrGemmWait, 2, local, buf, 3) && *err == kErrNone;
            ok = __all_sync(0xffffffffu, ok);  // tensor-memory loads are warp-wide
            tc_fence_after();
            if (!ok) break;
            const uint32_t acc = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * Cfg::kAccStride);
            const int n_cols = min(it.width, N - n0);
            for (int c = first; c < n_cols; c += step) {
                float v[32];
                tmem_ld32(acc + c, v);
                if (row < M) gemm_epilogue(ep, row, n0 + c, N, v, it.part);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {  // this warp has read its lanes of the buffer
                if (CG == 2) mbar_arrive_cluster(cluster_addr(&acc_empty[buf], 0));
                else mbar_arrive(&acc_empty[buf]);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (CG == 2) cluster_sync_all();  // no CTA leaves while the other's copies, commits or arrivals may still reach it
    if (*abandoned) {  // the same in both CTAs of a pair
        if (threadIdx.x == 0 && rank == 0) {
            const int mine = requested[0], other = requested[CG - 1], last = max(mine, other);
            for (int i = max(0, last - kStages); i < last; ++i) {  // the last filling of each stage
                uint64_t* bar = &full[i % kStages];
                // the leader announces the bytes of both CTAs: make up for a k-block that only one of them has requested
                if (i >= mine) mbar_expect_tx(bar, stage_bytes);
                else if (i >= other) mbar_complete_tx(bar, stage_bytes);
                mbar_drain(bar, (uint32_t)((i / kStages) & 1));
            }
        }
        __syncthreads();
        if (CG == 2) cluster_sync_all();
    }
    if (warp == 1) {
        tc_fence_after();
        if (CG == 2) tmem_dealloc_pair(tmem, 512);
        else tmem_dealloc(tmem, 512);
    }
}

template <int BN, int CG>
static cudaError_t launch_gemm(const CUtensorMap& tm_a, const CUtensorMap& tm_w, int M, int N, int K, const GemmWork& w, const GemmEpi& ep, int epi_warps,
                               cudaStream_t s) {
    const dim3 grid((unsigned)(std::min(g_gemm_ctas / CG, w.tiles * w.parts) * CG));
    return launch_pdl(gemm_tn_kernel<BN, CG>, grid, dim3(64 + 32 * epi_warps), GemmCfg<BN, CG>::kSmem, s, CG, tm_a, tm_w, M, N, K, w, ep);
}

GemmPlan plan_gemm(int M, int N, int K, int max_parts) { return plan_gemm(M, N, K, max_parts, g_gemm_ctas); }

cudaError_t launch_gemm_tn(const CUtensorMap& tm_a, const CUtensorMap& tm_w, int M, int N, int K, const GemmPlan& p, const GemmEpi& ep, cudaStream_t s) {
    if (M <= 0 || N <= 0 || K <= 0) return cudaErrorInvalidValue;
    const GemmWork w{p.m_tiles, p.items, p.parts, p.bn, p.wide, p.narrow};
    const int epi_warps = p.bn == 32 || (ep.mode == kGemmF32 && (ep.ldc & 7) != 0) ? 4 : 8;
    if (p.cg == 1) return launch_gemm<0, 1>(tm_a, tm_w, M, N, K, w, ep, epi_warps, s);
    if (p.bn == 256) return launch_gemm<256, 2>(tm_a, tm_w, M, N, K, w, ep, epi_warps, s);
    if (p.bn == 224) return launch_gemm<224, 2>(tm_a, tm_w, M, N, K, w, ep, epi_warps, s);
    return launch_gemm<192, 2>(tm_a, tm_w, M, N, K, w, ep, epi_warps, s);
}

// The status words of a product on its own, cleared by a kernel whose launch overlaps the end of the kernel in front and under
// which the product's own launch and set-up run (a memset between two products costs both overlaps: 511 x 12288 x 4096
// 54.5 -> 52.6 us a call, 2048 x 22016 x 4096 300 -> 294 us).
__global__ void __launch_bounds__(32) clear_status_kernel(int* status) {
    pdl_launch_dependents();
    pdl_wait();
    if (threadIdx.x < 8) status[threadIdx.x] = 0;
}
cudaError_t launch_clear_status(int* status, cudaStream_t s) { return launch_pdl(clear_status_kernel, dim3(1), dim3(32), 0, s, 1, status); }

// ============================================================================================ row kernels
constexpr int kRowThreads = 256;

// block-wide sums of up to three values; result valid in every thread
template <int NV>
__device__ __forceinline__ void block_sum(float (&v)[NV], float* red /* [NV][8] */) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        v[j] = warp_sum(v[j]);
        if (lane == 0) red[j * 8 + warp] = v[j];
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < kRowThreads / 32; ++w) t += red[j * 8 + w];
        v[j] = t;
    }
    __syncthreads();
}

__global__ void __launch_bounds__(kRowThreads) embed_norm_kernel(const int* tokens, int d, int vocab, const __nv_bfloat16* embed,
                                                                const __nv_bfloat16* gain, float eps, float* x, __nv_bfloat16* xn) {
    __shared__ float red[8];
    pdl_launch_dependents();
    const int r = blockIdx.x;
    int t = tokens[r];
    t = min(max(t, 0), vocab - 1);
    const uint4* e = reinterpret_cast<const uint4*>(embed + (size_t)t * d);  // d is a multiple of 8
    float s[1] = {0.f};
    for (int i = threadIdx.x; i < d / 8; i += kRowThreads) {
        const uint4 v = e[i];
        const float f[8] = {bf_lo(v.x), bf_hi(v.x), bf_lo(v.y), bf_hi(v.y), bf_lo(v.z), bf_hi(v.z), bf_lo(v.w), bf_hi(v.w)};
        float4* dst = reinterpret_cast<float4*>(x + (size_t)r * d + 8 * i);
        dst[0] = make_float4(f[0], f[1], f[2], f[3]);
        dst[1] = make_float4(f[4], f[5], f[6], f[7]);
#pragma unroll
        for (int k = 0; k < 8; ++k) s[0] = fmaf(f[k], f[k], s[0]);
    }
    block_sum<1>(s, red);
    const float inv = 1.0f / sqrtf(s[0] / (float)d + eps);
    for (int i = threadIdx.x; i < d / 8; i += kRowThreads) {
        const uint4 v = e[i], g = reinterpret_cast<const uint4*>(gain)[i];
        uint4 o;
        o.x = pack_bf16(bf_lo(v.x) * inv * bf_lo(g.x), bf_hi(v.x) * inv * bf_hi(g.x));
        o.y = pack_bf16(bf_lo(v.y) * inv * bf_lo(g.y), bf_hi(v.y) * inv * bf_hi(g.y));
        o.z = pack_bf16(bf_lo(v.z) * inv * bf_lo(g.z), bf_hi(v.z) * inv * bf_hi(g.z));
        o.w = pack_bf16(bf_lo(v.w) * inv * bf_lo(g.w), bf_hi(v.w) * inv * bf_hi(g.w));
        reinterpret_cast<uint4*>(xn + (size_t)r * d)[i] = o;
    }
}

// The residual add with the cosine similarity of the hidden state before and after the sublayer (Section 3.2), and
// the RMSNorm that feeds the next sublayer (its statistic is the |y|^2 just computed).
__global__ void __launch_bounds__(kRowThreads) resid_norm_kernel(int d, float* x, const float* c, int parts, size_t part_stride, const __nv_bfloat16* gain, float eps,
                                                                __nv_bfloat16* xn, float* cos_out) {
    __shared__ float red[24];
    pdl_launch_dependents();
    pdl_wait();
    const int r = blockIdx.x;
    float* xr = x + (size_t)r * d;
    const float* cr = c + (size_t)r * d;
    float s[3] = {0.f, 0.f, 0.f};
    for (int i = threadIdx.x; i < d; i += kRowThreads) {
        const float xv = xr[i];
        float o = cr[i];
        for (int p = 1; p < parts; ++p) o += cr[p * part_stride + i];  // a product that came in parts of its reduction dimension
        const float y = xv + o;
        xr[i] = y;
        s[0] = fmaf(xv, y, s[0]);
        s[1] = fmaf(xv, xv, s[1]);
        s[2] = fmaf(y, y, s[2]);
    }
    block_sum<3>(s, red);
    if (threadIdx.x == 0) {
        const double den = fmax(sqrt((double)s[1]) * sqrt((double)s[2]), 1e-30);
        cos_out[r] = (float)((double)s[0] / den);
    }
    if (gain) {
        const float inv = 1.0f / sqrtf(s[2] / (float)d + eps);
        for (int i = threadIdx.x; i < d; i += kRowThreads)
            xn[(size_t)r * d + i] = __float2bfloat16_rn(xr[i] * inv * __bfloat162float(gain[i]));
    }
}

// The same with the row held in registers (rows of at most kRowThreads * 4 * NV elements, a multiple of 4): x and the
// sublayer output are read once, 16 bytes per load, and the sums, the new hidden state and the normalised row all
// come from those registers.
template <int NV>
__global__ void __launch_bounds__(kRowThreads) resid_norm_vec_kernel(int d, float* x, const float* c, int parts, size_t part_stride, const __nv_bfloat16* gain, float eps,
                                                                    __nv_bfloat16* xn, float* cos_out) {
    __shared__ float red[24];
    pdl_launch_dependents();
    pdl_wait();
    const int r = blockIdx.x, nvec = d >> 2;
    float4* xr = reinterpret_cast<float4*>(x + (size_t)r * d);
    const float4* cr = reinterpret_cast<const float4*>(c + (size_t)r * d);
    float4 y[NV], cv[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        const int i = threadIdx.x + v * kRowThreads;
        y[v] = cv[v] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i < nvec) y[v] = xr[i], cv[v] = cr[i];
    }
    for (int p = 1; p < parts; ++p) {  // a product that came in parts of its reduction dimension: added in order
        const float4* cp = reinterpret_cast<const float4*>(c + p * part_stride + (size_t)r * d);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const int i = threadIdx.x + v * kRowThreads;
            if (i < nvec) {
                const float4 o = cp[i];
                cv[v].x += o.x, cv[v].y += o.y, cv[v].z += o.z, cv[v].w += o.w;
            }
        }
    }
    float s[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        const int i = threadIdx.x + v * kRowThreads;
        if (i < nvec) {
            const float4 xv = y[v];
            float4 o;
            o.x = xv.x + cv[v].x, o.y = xv.y + cv[v].y, o.z = xv.z + cv[v].z, o.w = xv.w + cv[v].w;
            s[0] = fmaf(xv.x, o.x, s[0]), s[1] = fmaf(xv.x, xv.x, s[1]), s[2] = fmaf(o.x, o.x, s[2]);
            s[0] = fmaf(xv.y, o.y, s[0]), s[1] = fmaf(xv.y, xv.y, s[1]), s[2] = fmaf(o.y, o.y, s[2]);
            s[0] = fmaf(xv.z, o.z, s[0]), s[1] = fmaf(xv.z, xv.z, s[1]), s[2] = fmaf(o.z, o.z, s[2]);
            s[0] = fmaf(xv.w, o.w, s[0]), s[1] = fmaf(xv.w, xv.w, s[1]), s[2] = fmaf(o.w, o.w, s[2]);
            xr[i] = o;
            y[v] = o;
        }
    }
    block_sum<3>(s, red);
    if (threadIdx.x == 0) {
        const double den = fmax(sqrt((double)s[1]) * sqrt((double)s[2]), 1e-30);
        cos_out[r] = (float)((double)s[0] / den);
    }
    if (gain) {
        const float inv = 1.0f / sqrtf(s[2] / (float)d + eps);
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const int i = threadIdx.x + v * kRowThreads;
            if (i < nvec) {
                const uint2 g = *reinterpret_cast<const uint2*>(gain + (size_t)i * 4);
                const __nv_bfloat162 lo = __floats2bfloat162_rn(y[v].x * inv * bf_lo(g.x), y[v].y * inv * bf_hi(g.x));
                const __nv_bfloat162 hi = __floats2bfloat162_rn(y[v].z * inv * bf_lo(g.y), y[v].w * inv * bf_hi(g.y));
                uint2 o;
                o.x = *reinterpret_cast<const uint32_t*>(&lo);
                o.y = *reinterpret_cast<const uint32_t*>(&hi);
                *reinterpret_cast<uint2*>(xn + (size_t)r * d + (size_t)i * 4) = o;
            }
        }
    }
}

__global__ void __launch_bounds__(32) sumcos_kernel(const float* cos_rows, int stride, int n_rows, double* sumcos, double* host) {
    const float* c = cos_rows + (size_t)blockIdx.x * stride;
    double acc = 0.0;
    for (int r = threadIdx.x; r < n_rows; r += 32) acc += (double)c[r];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (threadIdx.x == 0) sumcos[blockIdx.x] = host[blockIdx.x] = sumcos[blockIdx.x] + acc;
}

cudaError_t launch_embed_norm(const int* tokens, int n_rows, int d, int vocab, const __nv_bfloat16* embed, const __nv_bfloat16* gain,
                              float eps, float* x, __nv_bfloat16* xn, cudaStream_t s) {
    embed_norm_kernel<<<n_rows, kRowThreads, 0, s>>>(tokens, d, vocab, embed, gain, eps, x, xn);
    return cudaGetLastError();
}
cudaError_t launch_resid_norm(int n_rows, int d, float* x, const float* c, int parts, size_t part_stride, const __nv_bfloat16* gain, float eps, __nv_bfloat16* xn,
                              float* cos_out, cudaStream_t s) {
    const int nv = (d + kRowThreads * 4 - 1) / (kRowThreads * 4);
    void (*kernel)(int, float*, const float*, int, size_t, const __nv_bfloat16*, float, __nv_bfloat16*, float*) = resid_norm_vec_kernel<8>;
    if (d % 4 != 0 || nv > 8) kernel = resid_norm_kernel;
    else if (nv <= 1) kernel = resid_norm_vec_kernel<1>;
    else if (nv <= 2) kernel = resid_norm_vec_kernel<2>;
    else if (nv <= 4) kernel = resid_norm_vec_kernel<4>;
    else if (nv <= 5) kernel = resid_norm_vec_kernel<5>;
    return launch_pdl(kernel, dim3(n_rows), dim3(kRowThreads), 0, s, 1, d, x, c, parts, part_stride, gain, eps, xn, cos_out);
}
cudaError_t launch_sumcos(const float* cos_rows, int stride, int n_rows, int n_sub, double* sumcos, double* host, cudaStream_t s) {
    sumcos_kernel<<<n_sub, 32, 0, s>>>(cos_rows, stride, n_rows, sumcos, host);
    return cudaGetLastError();
}

cudaError_t configure_prefill(int max_smem) {
    cudaError_t e;
    (void)max_smem;
    int dev = 0, sms = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if (sms > 0) g_gemm_ctas = sms;
#define ASD_SET_GEMM(BN, CG) \
    if ((e = cudaFuncSetAttribute(gemm_tn_kernel<BN, CG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GemmCfg<BN, CG>::kSmem)) != cudaSuccess) return e
    ASD_SET_GEMM(256, 2);
    ASD_SET_GEMM(224, 2);
    ASD_SET_GEMM(192, 2);
    ASD_SET_GEMM(0, 1);
#undef ASD_SET_GEMM
    return configure_prefill_attention();
}

}  // namespace asd
