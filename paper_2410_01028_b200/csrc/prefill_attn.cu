// Causal attention over the prompt on tcgen05 (see prefill.h).
//
// One CTA = 128 query rows of one head, two CTAs per SM. Scores S = Q K^T of 128 rows x 64 keys and the output O = P V
// live in tensor memory; a thread owns one query row, so maximum, sum and mask need no exchange between threads.
// The probabilities are fp32 and enter the P V product as the sum of three bf16 numbers (p = hi + mid + lo, cut off
// at 8 mantissa bits each, which represents every fp32 probability exactly); with fewer terms the 2^-17 error of P
// flips bf16 roundings of the attention output in about every second row.
//
// What bounds it: the lengths of its MMAs, once two CTAs share an SM (1152 of the 1500 cycles of a tile below; the counter of active tensor
// cycles reads less, 47 % over a launch with its folds and its partly filled second round). Per 64 keys an S tile takes 384 cycles (N = 64 with both operands
// in shared memory is bound by the operand reads: 48 KB at 128 B per cycle) and the three P V products take 256 each; the
// softmax of a row takes about 1400 cycles (450 for S and its maximum, 480 for the exponentials and terms of either half). P is
// handed over in halves of 32 keys, so that the exponentials of one half run while the products of the other do, and S of the
// next tile is ready before the softmax wants it: per tile and CTA 2500 cycles and the fold below, 1500 per SM with two CTAs (2700 when
// a tile was one chain S -> softmax -> P V). Tiles of 64 keys because O (128 columns), S (64) and half a tile's P (64: hi of
// both halves, mid, lo) of two CTAs then fill the 512 columns of tensor memory.
//
// The running maximum of a row is only moved when it has grown by more than 2^8 (the conditional rescaling of FlashAttention-4;
// probabilities up to 256 are as exact as those up to 1): moving it means reading, scaling and writing O in tensor memory,
// which random scores need once or twice per row instead of once per tile. Whether a row moves depends on its own scores alone.
//
// An MMA cuts its sum with the accumulator off towards zero, so a chain of them loses about half an ulp of O at every step:
// 12 steps per key tile, and twice the loss per step that mma.sync has. The terms of a tile are therefore added smallest first (lo and
// mid of both halves, then hi), and before the key tiles 1, 2, 4, 8, ... O and the row
// sums are added to fp32 totals (rounded to nearest) and start anew. No chain is then longer than half of a row's keys, and what is
// lost in it counts by its share of the sum. Error against 64 bits over the attention kernel on mma.sync, 64 to 8192 keys:
// 0.3-0.8 of it (without the totals 0.7-2.4); a bias of values with a mean of one 1.8e-5 after 8192 keys instead of 6.0e-5
// (mma.sync: 3.1e-5). Head size 64 leaves tensor memory for the totals; at 128 they are in scratch memory, and a fold is 64 KB
// each way of L2 traffic that all CTAs make at the same tiles. (Adding in memory, red.add.v4.f32, was slower: 2048 keys 0.127 -> 0.140 ms.)
//
// Measured, 2048 rows of 32 heads of 128, launch to end, against a tile as one chain S -> softmax -> P V with S over the lo terms:
// 0.139 -> 0.123 ms over their own keys, 0.268 -> 0.222 ms on top of 2048 others, 0.521 -> 0.419 ms on top of 6144; heads of 64
// 0.085 -> 0.072, 0.181 -> 0.150, 0.368 -> 0.298 ms. What is left over the tensor core's 0.26 ms (6144) is the second round of CTAs (512 on
// 296 places) and the folds.
#include "common.cuh"
#include "prefill.h"
#include "tcgen05.cuh"

namespace asd {

constexpr int kFaRows = 128, kFaKeys = 64, kFaHalf = kFaKeys / 2, kFaThreads = 192, kFaStages = 2;
constexpr int kFaTmemCols = 256;                       // O: 0-127; S: 128-191; P of half a key tile: 192-255
constexpr int kFaColS = 128, kFaColHi = 192, kFaColMid = 224, kFaColLo = 240;  // hi terms of either half
constexpr int kFaColTotals = 64;                       // head size 64: the totals, behind O

// tiles before which O and the row sums are folded into the totals: 1, 2, 4, 8, ... (absolute key tiles: the same for every row)
constexpr int kFaFirstFold = 1;
__device__ __forceinline__ bool fa_folds(int j) { return j >= kFaFirstFold && (j & (j - 1)) == 0; }

template <int HD>
struct FaCfg {
    static constexpr int kPanels = HD / 64;                      // panels of 64 columns (128 bytes, one swizzle span)
    static constexpr uint32_t kQPanel = kFaRows * 128, kKvPanel = kFaKeys * 128;
    static constexpr uint32_t kQBytes = kPanels * kQPanel, kKvBytes = kPanels * kKvPanel;
    static constexpr size_t kSmem = kQBytes + 2 * kFaStages * kKvBytes + 1024 /* alignment */ + 128 /* barriers */;
};

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ unsigned long long fadd2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
// the upper halves of two words: bf16 pairs cut off from two fp32 numbers (a in the low half)
__device__ __forceinline__ uint32_t upper_halves(uint32_t a, uint32_t b) { return __byte_perm(a, b, 0x7632); }
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15};" ::"r"(r[0]),
        "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]),
        "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(taddr)
        : "memory");
}

__device__ __forceinline__ unsigned long long fsub2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// 32 scores of one row -> probabilities 2^(s c - m c), their sum added to sum2, their three bf16 terms (pairs of keys)
__device__ __forceinline__ void probabilities32(const uint32_t (&s)[32], unsigned long long c2, unsigned long long nmc2, unsigned long long& sum2,
                                                uint32_t (&hi)[16], uint32_t (&mid)[16], uint32_t (&lo)[16]) {
    unsigned long long part = pack2(0.f, 0.f);  // a sum of its own, so that no chain of additions runs over all keys of a row
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        float a, b;
        unpack2(ffma2(pack2(__uint_as_float(s[2 * i]), __uint_as_float(s[2 * i + 1])), c2, nmc2), a, b);
        unsigned long long p = pack2(ex2(a), ex2(b));
        part = fadd2(part, p);
        auto term = [&](uint32_t& w) {  // the upper 8 bits of what is left of both
            unpack2(p, a, b);
            w = upper_halves(__float_as_uint(a), __float_as_uint(b));
            return pack2(__uint_as_float(__float_as_uint(a) & 0xFFFF0000u), __uint_as_float(__float_as_uint(b) & 0xFFFF0000u));
        };
        p = fsub2(p, term(hi[i]));  // exact
        p = fsub2(p, term(mid[i]));  // exact, 8 bits left
        unpack2(p, a, b);
        lo[i] = upper_halves(__float_as_uint(a), __float_as_uint(b));
    }
    sum2 = fadd2(sum2, part);
}

// Warps 0-3: softmax and epilogue, thread = query row. Warp 4: TMA producer. Warp 5: issues the MMAs
// and owns the tensor-memory allocation. Barriers: q_full, k_full / v_full[s] (bytes landed), k_empty / v_empty[s] (the
// MMAs reading the stage have finished), s_full (S of tile j is complete), p_full (the 128 rows' P of half a tile is in tensor
// memory), pv_done (the products with it have finished, and with them every earlier one: O holds the halves so far and P may be
// overwritten). S of tile j + 1 goes over S of tile j, which every thread has read before it reports the first half of P.
template <int HD>
__global__ void __launch_bounds__(kFaThreads, 2)
flash_prefill_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                     __nv_bfloat16* __restrict__ out, float* totals, int n_rows, int pos0, int d_model, int group, float scale_log2, int* err_words) {
    using Cfg = FaCfg<HD>;
    constexpr bool kTmemTotals = HD == 64;
    extern __shared__ unsigned char fa_smem_raw[];
    unsigned char* base = fa_smem_raw + ((1024u - (smem_u32(fa_smem_raw) & 1023u)) & 1023u);
    unsigned char* k_smem = base + Cfg::kQBytes;
    unsigned char* v_smem = k_smem + kFaStages * Cfg::kKvBytes;
    uint64_t* q_full = reinterpret_cast<uint64_t*>(v_smem + kFaStages * Cfg::kKvBytes);
    uint64_t *k_full = q_full + 1, *k_empty = k_full + kFaStages, *v_full = k_empty + kFaStages, *v_empty = v_full + kFaStages;
    uint64_t *s_full = v_empty + kFaStages, *p_full = s_full + 1, *pv_done = p_full + 1, *drained = pv_done + 1;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drained + 1);
    volatile int* err = err_words;

    const int warp = threadIdx.x >> 5;
    const int head = blockIdx.x, kvh = head / group;
    const int r0 = (gridDim.y - 1 - blockIdx.y) * kFaRows;  // the tiles with the most keys start first
    const int last_row = min(r0 + kFaRows, n_rows) - 1;
    const int n_kt = (pos0 + last_row) / kFaKeys + 1;

    if (threadIdx.x == 0) {
        mbar_init(q_full, 1);
        for (int s = 0; s < kFaStages; ++s) mbar_init(&k_full[s], 1), mbar_init(&k_empty[s], 1), mbar_init(&v_full[s], 1), mbar_init(&v_empty[s], 1);
        mbar_init(s_full, 1);
        mbar_init(p_full, kFaRows);
        mbar_init(pv_done, 1);
        mbar_init(drained, 1);
        mbar_fence_init();
    }
    if (warp == 5) {
        tmem_alloc(tmem_slot, kFaTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    pdl_launch_dependents();
    pdl_wait();  // everything above overlaps the end of the kernel before

    const uint32_t on = elect_one();
    if (warp == 4) {
        mbar_expect_tx_on(q_full, Cfg::kQBytes, on);
        for (int p = 0; p < Cfg::kPanels; ++p) tma_load_2d_on(base + p * Cfg::kQPanel, &tm_q, head * HD + p * 64, r0, q_full, on);
        bool ok = true;
        int nk = 0, nv = 0;  // K and V tiles requested so far
        while (nv < n_kt && ok) {
            // K runs one tile ahead of V: S of tile j + 1 is issued right behind P V of tile j
            if (nk < n_kt && nk <= nv + 1) {
                const int s = nk % kFaStages;
                if (nk >= kFaStages) ok = mbar_wait_warp(&k_empty[s], (uint32_t)((nk / kFaStages - 1) & 1), err, kErrAttnWait, 0, nk, s, 1);
                if (!ok) break;
                mbar_expect_tx_on(&k_full[s], Cfg::kKvBytes, on);
                for (int p = 0; p < Cfg::kPanels; ++p)
                    tma_load_2d_on(k_smem + s * Cfg::kKvBytes + p * Cfg::kKvPanel, &tm_k, kvh * HD + p * 64, nk * kFaKeys, &k_full[s], on);
                ++nk;
                if (nk == 1 && n_kt > 1) continue;
            }
            const int s = nv % kFaStages;
            if (nv >= kFaStages) ok = mbar_wait_warp(&v_empty[s], (uint32_t)((nv / kFaStages - 1) & 1), err, kErrAttnWait, 0, nv, s, 2);
            if (!ok) break;
            mbar_expect_tx_on(&v_full[s], Cfg::kKvBytes, on);
            for (int p = 0; p < Cfg::kPanels; ++p)
                tma_load_2d_on(v_smem + s * Cfg::kKvBytes + p * Cfg::kKvPanel, &tm_v, kvh * HD + p * 64, nv * kFaKeys, &v_full[s], on);
            ++nv;
        }
        // the copies land before the CTA gives its shared memory back, also when a role of the CTA gives up
        auto landed = [&](uint64_t* bar, int n) {
            if (n > 0) mbar_drain(bar, (uint32_t)((n - 1) & 1));
        };
        landed(q_full, 1);
        for (int s = 0; s < kFaStages; ++s) landed(&k_full[s], (nk + kFaStages - 1 - s) / kFaStages), landed(&v_full[s], (nv + kFaStages - 1 - s) / kFaStages);
    } else if (warp == 5) {
        constexpr uint32_t idesc_s = umma_idesc_bf16(kFaRows, kFaKeys);
        constexpr uint32_t idesc_o = umma_idesc_bf16(kFaRows, HD) | (1u << 16);  // V is [key][dimension]: N-major
        const uint32_t q_addr = smem_u32(base);
        bool ok = mbar_wait_warp(q_full, 0, err, kErrAttnWait, 1, 0, 0, 3);
        auto scores = [&](int j) {  // S of tile j
            const int s = j % kFaStages;
            ok = ok && mbar_wait_warp(&k_full[s], (uint32_t)((j / kFaStages) & 1), err, kErrAttnWait, 1, j, s, 4);
            if (!ok) return;
            tc_fence_after();
            const uint32_t k_addr = smem_u32(k_smem) + s * Cfg::kKvBytes;
#pragma unroll
            for (int k = 0; k < HD / 16; ++k)
                tc_mma_bf16(tmem + kFaColS, umma_desc_k128(q_addr + (k / 4) * Cfg::kQPanel) + 2 * (k % 4),
                            umma_desc_k128(k_addr + (k / 4) * Cfg::kKvPanel) + 2 * (k % 4), idesc_s, k != 0, on);
            tc_commit(&k_empty[s], on);
            tc_commit(s_full, on);
        };
        scores(0);
        for (int j = 0; j < n_kt && ok; ++j) {
            const int s = j % kFaStages;
            ok = mbar_wait_warp(&v_full[s], (uint32_t)((j / kFaStages) & 1), err, kErrAttnWait, 1, j, s, 5);
            const bool fresh = j == 0 || fa_folds(j);  // O starts anew
            const uint64_t v_desc = umma_desc_mn128(smem_u32(v_smem) + s * Cfg::kKvBytes, Cfg::kKvPanel);
#pragma unroll 1
            for (int h = 0; h < 2 && ok; ++h) {
                ok = mbar_wait_warp(p_full, (uint32_t)h, err, kErrAttnWait, 1, j, s, 6);
                if (!ok) break;
                tc_fence_after();
                auto products = [&](uint32_t a, int half, bool anew) {  // O (+)= one term of the half's P
#pragma unroll
                    for (int k = 0; k < kFaHalf / 16; ++k)  // 16 keys: 8 columns of P, 2048 bytes of V
                        tc_mma_bf16_ts(tmem, tmem + a + 8 * k, v_desc + (uint64_t)(128 * (half * (kFaHalf / 16) + k)), idesc_o, !(anew && k == 0), on);
                };
                products(kFaColLo, h, fresh && h == 0);
                products(kFaColMid, h, false);
                if (h == 1) products(kFaColHi, 0, false), products(kFaColHi + 16, 1, false);  // the largest terms last
                tc_commit(pv_done, on);
                if (h == 0 && j + 1 < n_kt) scores(j + 1);
            }
            tc_commit(&v_empty[s], on);
        }
        // the MMAs end before the tensor memory is freed, also when a role of the CTA gives up
        tc_commit(drained, on);
        mbar_drain(drained, 0);
    } else {
        const int row = r0 + threadIdx.x;
        const int pos = pos0 + min(row, n_rows - 1);  // rows past the prompt (queries of an earlier one) are computed and not stored
        const uint32_t lane_base = tmem + ((uint32_t)(warp * 32) << 16);
        const unsigned long long c2 = pack2(scale_log2, scale_log2);
        float m = 0.f;
        // what has been folded: the columns in totals, the sum of probabilities here; both still want the factor since. The
        // block's part of totals is [HD / 8][128 rows][8], so that the 32 bytes of neighbouring lanes are neighbours.
        float* total = totals + (size_t)r0 * d_model + (size_t)head * (kFaRows * HD) + threadIdx.x * 8;
        float sum_total = 0.f, since = 1.f;
        unsigned long long sum2 = pack2(0.f, 0.f);
        bool ok = true;
        int halves = 0;  // halves of P reported so far
        auto products_done = [&]() {  // of every half reported so far
            if (halves > 0) ok = mbar_wait(pv_done, (uint32_t)((halves - 1) & 1), err, kErrAttnWait, 2, halves, 0, 9) && ok;
            ok = __all_sync(0xffffffffu, ok);  // tensor-memory accesses are warp-wide
            tc_fence_after();
        };
        // total * since + O, 32 columns at a time, to `take`. In scratch memory the totals of 64 columns are requested at a time, the
        // first ones while the products still run; in tensor memory (HD = 64 leaves it 64 columns) they are at hand.
        auto fold = [&](bool first, auto&& take) {
#pragma unroll
            for (int c = 0; c < HD; c += 64) {
                uint32_t w[64], o[32];
                if (!kTmemTotals) {
#pragma unroll
                    for (int i = 0; i < 64; ++i) w[i] = 0u;
                    if (!first) {
#pragma unroll
                        for (int i = 0; i < 64; i += 8) ld_global_v8(total + (c + i) * kFaRows, w + i);
                    }
                }
                if (c == 0) products_done();
                if (!ok) return;
#pragma unroll
                for (int h = 0; h < 64; h += 32) {
                    uint32_t t[32];
                    tmem_ld32_async(lane_base + c + h, o);
                    if (kTmemTotals && !first) tmem_ld32_async(lane_base + kFaColTotals + h, t);
                    tmem_ld_wait(o);
                    if (kTmemTotals && !first) tmem_ld_wait(t);
#pragma unroll
                    for (int i = 0; i < 32; ++i) {
                        const float before = first ? 0.f : __uint_as_float(kTmemTotals ? t[i] : w[h + i]);
                        o[i] = __float_as_uint(fmaf(before, since, __uint_as_float(o[i])));
                    }
                    take(c + h, o);
                }
            }
        };
        // the exponentials of half a tile run while the products of the half before do; then its P takes the place that those have left
        auto report_half = [&](int h, const uint32_t (&s)[32], unsigned long long nmc2) {
            uint32_t hi[16], mid[16], lo[16];
            probabilities32(s, c2, nmc2, sum2, hi, mid, lo);
            products_done();
            if (!ok) return;
            tmem_st16(lane_base + kFaColHi + 16 * h, hi);
            tmem_st16(lane_base + kFaColMid, mid);
            tmem_st16(lane_base + kFaColLo, lo);
            tmem_st_wait();
            tc_fence_before();
            mbar_arrive(p_full);
            ++halves;
        };
        for (int j = 0; j < n_kt; ++j) {
            const bool fresh = fa_folds(j);
            if (fresh) {
                fold(j == kFaFirstFold, [&](int c, const uint32_t (&v)[32]) {
                    if (kTmemTotals) {
                        tmem_st32(lane_base + kFaColTotals + c, v);
                    } else {
#pragma unroll
                        for (int i = 0; i < 32; i += 8) st_global_v8(total + (c + i) * kFaRows, v + i);
                    }
                });
                if (!ok) break;
                float a, b;
                unpack2(sum2, a, b);
                sum_total = fmaf(sum_total, since, a + b);
                sum2 = pack2(0.f, 0.f), since = 1.f;
            }
            ok = mbar_wait(s_full, (uint32_t)(j & 1), err, kErrAttnWait, 2, j, 0, 7);
            ok = __all_sync(0xffffffffu, ok);  // tensor-memory accesses are warp-wide
            if (!ok) break;
            tc_fence_after();
            uint32_t s0[32], s1[32];
            tmem_ld32_async(lane_base + kFaColS, s0);
            tmem_ld32_async(lane_base + kFaColS + 32, s1);
            tmem_ld_wait(s0);
            tmem_ld_wait(s1);
            const int key0 = j * kFaKeys;
            if (key0 + kFaKeys - 1 > pos0 + r0) {  // a tile on the diagonal: the row at position p sees keys <= p
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    if (key0 + i > pos) s0[i] = 0xFF800000u;
                    if (key0 + 32 + i > pos) s1[i] = 0xFF800000u;
                }
            }
            float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
            for (int i = 0; i < 32; i += 2) {
                mx[(i >> 1) & 1] = max3(mx[(i >> 1) & 1], __uint_as_float(s0[i]), __uint_as_float(s0[i + 1]));
                mx[2 + ((i >> 1) & 1)] = max3(mx[2 + ((i >> 1) & 1)], __uint_as_float(s1[i]), __uint_as_float(s1[i + 1]));
            }
            const float tile_max = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
            if (j == 0) {
                m = tile_max;  // finite: key 0 is visible to every row
            }
            // each row decides by its own scores: the others in the warp, rows past the prompt among them, scale by exactly 1
            const bool move = j > 0 && (tile_max - m) * scale_log2 > 8.0f;
            if (__any_sync(0xffffffffu, move)) {
                const float alpha = move ? ex2((m - tile_max) * scale_log2) : 1.0f;
                m = move ? tile_max : m;
                float a, b;
                unpack2(sum2, a, b);
                sum2 = pack2(a * alpha, b * alpha);
                since *= alpha;
                if (!fresh) products_done();
                if (!ok) break;
#pragma unroll 1
                for (int c = fresh ? HD : 0; c < HD; c += 32) {
                    uint32_t o[32];
                    tmem_ld32_async(lane_base + c, o);
                    tmem_ld_wait(o);
#pragma unroll
                    for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                    tmem_st32(lane_base + c, o);
                }
            }
            const float nmc = -m * scale_log2;
            const unsigned long long nmc2 = pack2(nmc, nmc);
            report_half(0, s0, nmc2);
            if (ok) report_half(1, s1, nmc2);
            if (!ok) break;
        }
        if (ok) {
            float a, b;
            unpack2(sum2, a, b);
            const float inv = 1.0f / fmaf(sum_total, since, a + b);
            __nv_bfloat16* dst = out + (size_t)row * d_model + (size_t)head * HD;
            fold(n_kt <= kFaFirstFold, [&](int c, const uint32_t (&v)[32]) {
                if (row < n_rows) {
                    uint32_t w[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i) w[i] = pack_bf16(__uint_as_float(v[2 * i]) * inv, __uint_as_float(v[2 * i + 1]) * inv);
                    st_global_v8(dst + c, w);
                    st_global_v8(dst + c + 16, w + 8);
                }
            });
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 5) {
        tc_fence_after();
        tmem_dealloc(tmem, kFaTmemCols);
    }
}

cudaError_t launch_flash_prefill(const CUtensorMap& tm_q, const CUtensorMap& tm_k, const CUtensorMap& tm_v, __nv_bfloat16* out, float* totals,
                                 int n_rows, int pos0, int d_model, int head_dim, int n_heads, int n_kv_heads, float scale, int* err, cudaStream_t s) {
    if (n_rows <= 0) return cudaErrorInvalidValue;
    const dim3 grid(n_heads, (n_rows + kFaRows - 1) / kFaRows);
    const int group = n_heads / n_kv_heads;
    const float scale_log2 = scale * 1.4426950408889634f;
    if (head_dim == 128)
        return launch_pdl(flash_prefill_kernel<128>, grid, dim3(kFaThreads), FaCfg<128>::kSmem, s, 1, tm_q, tm_k, tm_v, out, totals, n_rows, pos0, d_model, group, scale_log2, err);
    if (head_dim == 64)
        return launch_pdl(flash_prefill_kernel<64>, grid, dim3(kFaThreads), FaCfg<64>::kSmem, s, 1, tm_q, tm_k, tm_v, out, totals, n_rows, pos0, d_model, group, scale_log2, err);
    return cudaErrorInvalidValue;
}

cudaError_t configure_prefill_attention() {
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(flash_prefill_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FaCfg<128>::kSmem)) != cudaSuccess) return e;
    return cudaFuncSetAttribute(flash_prefill_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FaCfg<64>::kSmem);
}

}  // namespace asd
