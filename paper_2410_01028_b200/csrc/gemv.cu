// Fused RMSNorm -> GEMV -> epilogue for M <= 9 activation rows as a launch of its own (asd_fused_gemv).
//
// One CTA per SM owns a contiguous slab of weight rows and streams it exactly once through a ring of shared memory: two
// producer warps copy pieces of up to 16 weight rows x 1024 or 2048 inputs (and what a row has left), one bulk copy per row, eight
// rows each, and run as far ahead as the ring holds. Eight warps multiply: every warp takes the 32-input units u, u + 8, ... of a piece on mma.sync m16n8k16 with the weights
// as the 16-row operand and the activation rows as the 8 columns. A lane reads 16 bytes (8 inputs) of weight rows g and
// g + 8 straight into operand registers, four inputs per MMA; the order of the inputs inside a dot product is free, so the
// same lane supplies the same 8 inputs of activation row g. Two more warps add the eight warps' sums of a group of rows and
// run the epilogue while the others multiply the next group. Many rows of up to 768 inputs come in copies of 16 whole rows, and a warp
// has a group to itself (BY_WARP), with the same sums in the same order.
//
// Sums: the 16 x 8 result of every MMA starts from zero and the results are added on the CUDA cores; a warp's sums of a
// group go to shared memory every kGemvEpoch inputs, where the eight warps' sums are added as a tree and then to the row's
// total. A sum of 16 products is nearly exact and no chain of additions is long (error against 64 bits 8.8e-8 of the result at
// 13760 inputs; 9.1e-8 with the chains of the kernel before). Chunks of 1024 inputs, epochs and groups depend on the
// matrix and the SM count alone: row m of an M-row call is bit-identical to the same row of a one-row call. Rows of weights
// are 64 bytes apart modulo 128 in shared memory (but for copies of whole rows), so the eight lanes of a 16-byte read phase (two
// rows) meet no conflict.
//
// What bounds it: the weight stream and, for small matrices, launch, first bytes and last sums; a piece costs every role some
// hundred cycles of index arithmetic and barriers (a producer also about 60 for each copy), so small pieces were bound by those and not by
// DRAM. Launch after launch in CUDA graphs over matrices that L2 does not hold, us with the weights loaded straight into operand registers
// by 16 warps -> with this ring, one producer warp, divisions in every step and pieces of 1024 inputs at most for short rows -> now:
//   1 row    256 -> 32000 6.1 -> 15.5 -> 5.5, 688 -> 30000 11.6 -> 14.4 -> 9.4, 1032 -> 20000 12.2 -> 16.4 -> 11.5, 2056 -> 12000 14.2 -> 15.2 -> 12.2,
//            2048 -> 6144 norm 9.3 -> 7.3 -> 7.0, 4096 -> 22016 SwiGLU 34.7 -> 29.5 -> 29.5 (6.1 TB/s), 2000 -> 12000 13.0 -> 11.8 -> 12.1
//   5 rows   256 -> 32000 7.5 -> 15.5 -> 5.5, 13760 -> 5120 residual 36.0 -> 32.3 -> 32.0, 22016 -> 8192 residual 69.6 -> 69.4 -> 65.4
//   9 rows   1032 -> 20000 16.6 -> 18.4 -> 13.5, 4096 -> 22016 SwiGLU 40.4 -> 36.1 -> 30.5, 11008 -> 4096 residual 32.4 -> 25.9 -> 25.3
// and behind an RMSNorm of long rows (norm_long): 2 rows 16384 -> 4096 29.3 -> 36.3 -> 28.6, 4 rows 22016 -> 8192 73.7 -> 79.1 -> 70.1, 5 rows 11008 ->
// 4096 26.1 -> 27.9 -> 24.6, 6 rows 16384 -> 4096 37.1 -> 48.0 -> 34.8. Of 300 shapes of one to nine rows none is slower than with operand
// registers; against the ring with one producer three of 256 to 2048 inputs are 2 to 3 % slower (three to five rows of 2048 -> 6144 norm 7.4 -> 7.6).
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "gemv.h"
#include "ring.cuh"

namespace asd {

constexpr int kGemvChunk = 1024;     // inputs whose products are added in pairs first
constexpr int kGemvEpoch = 4096;     // inputs whose products are added in registers (a multiple of a piece's)
constexpr int kGemvMaxStages = 16;
constexpr int kGemvBlockRows = 256;  // most weight rows of a CTA whose totals are in shared memory at a time
constexpr int kGemvThreads = (kGemvWarps + 4) * 32;  // multiplying warps, two producers, two epilogue warps
constexpr int kGemvHead = 1024;      // bytes in front: barriers, flag, sums of squares
constexpr int kErrGemvWait = 21;

// n / d for n * d < 2^32, with magic = 2^32 / d + 1 (0 for d = 1): a division takes a warp 150 to 250 cycles, and every role
// would make two for each group of rows
__device__ __forceinline__ int gemv_div(int n, unsigned magic) { return magic ? (int)__umulhi((unsigned)n, magic) : n; }

// first row of CTA b; the boundaries are even so that gate_i and up_i stay together
__device__ __forceinline__ int gemv_row(const GemvParams& p, int b) {
    return min(p.n_rows, 2 * (b * p.cta_pairs + gemv_div(b * p.cta_more, p.div_grid)));  // 2 * (b * pairs / CTAs)
}

__device__ __forceinline__ void mma_zero(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}

// Signal arrival of this CTA; returns true in every thread of the last CTA to arrive.
__device__ __forceinline__ bool last_cta_arrives(unsigned* counter, int* flag_smem) {
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned t;  // one release and acquire at GPU scope, cumulative over the CTA's writes, which the barrier has ordered before it
        asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(t) : "l"(counter) : "memory");
        *flag_smem = (t == gridDim.x - 1) ? 1 : 0;
    }
    __syncthreads();
    return *flag_smem != 0;
}

// The order in which every role walks a CTA's rows: blocks of rows, windows of the activations, groups of at most 16 rows, epochs
// of inputs, pieces. A warp whose wait has run out leaves (the calls return false, and so does the walk): it signals nothing any
// more, so that whoever needs its signal leaves as well, and no ring stage, window or sums are filled again before they have
// landed and been read.
//   window(first_use, k0, k1)                     the activations k0 .. k1 are wanted
//   piece(row, rows, k0, len, win0)               rows x inputs of one ring stage
//   epoch(local_row, row, rows, k0, k1, win_end)  the sums of inputs k0 .. k1 of a group are complete; win_end: nothing else
//                                                 reads the window
template <class Window, class Piece, class Epoch>
__device__ __forceinline__ bool gemv_walk(const GemvParams& p, int row0, int row1, Window&& window, Piece&& piece, Epoch&& epoch) {
    for (int blk = 0; blk < p.n_blk; ++blk) {
        const int blk0 = blk == 0 ? row0 : row0 + (row1 - row0) * blk / p.n_blk / 2 * 2;
        const int rows = (blk + 1 == p.n_blk ? row1 : row0 + (row1 - row0) * (blk + 1) / p.n_blk / 2 * 2) - blk0;
        const int pairs = (rows + 1) >> 1;
        if (rows <= 0) break;  // fewer pairs of rows than CTAs
        const int least = gemv_div(pairs, p.div_groups), more = pairs - least * p.groups;
        for (int w0 = 0; w0 < p.n_in; w0 += p.win) {
            const int w1 = min(p.n_in, w0 + p.win);
            if ((blk == 0 || p.win < p.n_in) && !window(blk + w0 == 0, w0, w1)) return false;
            for (int o = 0, r0 = 0, n, part = 0; o < p.groups; ++o, r0 += n) {  // group o: pairs o * pairs / groups and on
                part += more;
                n = min(rows - r0, 2 * (least + (part >= p.groups)));
                if (part >= p.groups) part -= p.groups;
                for (int e0 = w0; e0 < w1; e0 += kGemvEpoch) {
                    const int e1 = min(w1, e0 + kGemvEpoch);
                    for (int k0 = e0, len; k0 < e1; k0 += len) {
                        len = min(p.seg, e1 - k0);
                        if (e1 - k0 - len <= p.tail) len = e1 - k0;
                        if (!piece(blk0 + r0, n, k0, len, w0)) return false;
                    }
                    if (!epoch(r0, blk0 + r0, n, e0, e1, o + 1 == p.groups && e1 == w1)) return false;
                }
            }
        }
    }
    return true;
}

// Every stride-th group of a CTA's rows, from the first on (a block of all rows: the groups are those of the walk)
struct GemvGroups {
    int o, row, rows;  // the group, its first weight row and their number
    __device__ __forceinline__ GemvGroups(const GemvParams& p, int row0, int row1, int first, int stride)
        : o(first), row(0), rows(0), row0(row0), row1(row1), stride(stride), groups(p.groups) {
        const int pairs = (row1 - row0 + 1) >> 1;
        least = gemv_div(pairs, p.div_groups), more = pairs - least * groups;
        leap = gemv_div(stride * pairs, p.div_groups), part_leap = stride * pairs - leap * groups;
        at = gemv_div(first * pairs, p.div_groups), part = first * pairs - at * groups;
        settle();
    }
    __device__ __forceinline__ void next() {
        o += stride, at += leap, part += part_leap;
        if (part >= groups) part -= groups, ++at;
        settle();
    }

private:
    int row0, row1, stride, groups, least, more, leap, part_leap, at, part;
    __device__ __forceinline__ void settle() { row = row0 + 2 * at, rows = min(row1 - row, 2 * (least + (part + more >= groups))); }
};

// RMSNorm of the activation rows into the window of inputs w0 .. w1, by the multiplying warps: R rows of up to U x 1024 inputs at a
// time are read once, all loads in flight together, and normalised from registers; what lies behind (one row) is read twice, 8 loads of a
// thread at a time. Thread t adds the squares of inputs 4 t + 1024 u in this order whatever R and U.
template <int R, int U, bool kTail>
__device__ __forceinline__ void norm_rows(const GemvParams& p, __nv_bfloat16* xs, float* red, bool first, int w0, int w1) {
    constexpr int kThreads = kGemvWarps * 32, kStep = kThreads * 4, kBatch = R == 1 ? 8 : 16 / R, kHeld = U > 0 ? U : 1;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, n_in = p.n_in;
    const float* xf = reinterpret_cast<const float*>(p.x);
    auto load = [&](int m, int i) { return *reinterpret_cast<const ulonglong2*>(xf + (size_t)m * n_in + i); };
    auto inverse = [&](int m) {  // of the row's root mean square
        const float* r = red + m * kGemvWarps;
        const float s = ((r[0] + r[1]) + (r[2] + r[3])) + ((r[4] + r[5]) + (r[6] + r[7]));
        return 1.0f / sqrtf(s / (float)n_in + p.eps);
    };
    auto put = [&](int m, int i, const ulonglong2& a, unsigned long long inv, const uint2& gn) {
        float lo0, hi0, lo1, hi1;
        unpack2(fmul2(fmul2(a.x, inv), bf2_to_f2(gn.x)), lo0, hi0);
        unpack2(fmul2(fmul2(a.y, inv), bf2_to_f2(gn.y)), lo1, hi1);
        const __nv_bfloat162 lo = __floats2bfloat162_rn(lo0, hi0), hi = __floats2bfloat162_rn(lo1, hi1);
        *reinterpret_cast<uint2*>(xs + (size_t)m * p.xs_ld + (i - w0)) = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
    };
    auto gain = [&](int i) { return *reinterpret_cast<const uint2*>(p.gain + i); };
    static_assert(kGemvWarps == 8, "sums of squares of eight warps");
    auto load_batch = [&](ulonglong2 (&a)[kBatch][R], int m0, int i, int end) {
#pragma unroll
        for (int b = 0; b < kBatch; ++b)
#pragma unroll
            for (int r = 0; r < R; ++r) {
                a[b][r] = make_ulonglong2(0ull, 0ull);
                if (m0 + r < p.M && i + kStep * b < end) a[b][r] = load(m0 + r, i + kStep * b);
            }
    };
    auto fill = [&](int m0, int i, const unsigned long long (&inv)[R]) {  // inputs i, i + 1024, ... of these rows
        for (; i < w1; i += kStep * kBatch) {
            ulonglong2 a[kBatch][R];
            load_batch(a, m0, i, w1);
#pragma unroll
            for (int b = 0; b < kBatch; ++b)
                if (i + kStep * b < w1) {
                    const uint2 gn = gain(i + kStep * b);
#pragma unroll
                    for (int r = 0; r < R; ++r)
                        if (m0 + r < p.M) put(m0 + r, i + kStep * b, a[b][r], inv[r], gn);
                }
        }
    };
    if (first) {  // (w0 == 0)
        uint2 g[kHeld];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            g[u] = make_uint2(0u, 0u);
            if (4 * t + kStep * u < n_in) g[u] = gain(4 * t + kStep * u);
        }
        for (int m0 = 0; m0 < p.M; m0 += R) {
            ulonglong2 v[R][kHeld];
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    v[r][u] = make_ulonglong2(0ull, 0ull);
                    if (m0 + r < p.M && 4 * t + kStep * u < n_in) v[r][u] = load(m0 + r, 4 * t + kStep * u);
                }
            unsigned long long ss[R][2] = {};
            auto add = [&](unsigned long long (&q)[2], const ulonglong2& a) { q[0] = ffma2(a.x, a.x, q[0]), q[1] = ffma2(a.y, a.y, q[1]); };
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int u = 0; u < U; ++u) add(ss[r], v[r][u]);
            if constexpr (kTail)
                for (int i = 4 * t + kStep * U; i < n_in; i += kStep * kBatch) {
                    ulonglong2 a[kBatch][R];
                    load_batch(a, m0, i, n_in);
#pragma unroll
                    for (int b = 0; b < kBatch; ++b)
#pragma unroll
                        for (int r = 0; r < R; ++r) add(ss[r], a[b][r]);
                }
            float s[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                float a, b, c, d;
                unpack2(ss[r][0], a, b);
                unpack2(ss[r][1], c, d);
                s[r] = (a + b) + (c + d);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int r = 0; r < R; ++r) s[r] += __shfl_xor_sync(0xffffffffu, s[r], o);
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (lane == 0 && m0 + r < p.M) red[(m0 + r) * kGemvWarps + warp] = s[r];
            bar_sync(1, kThreads);
            const float inv_lane = inverse(min(m0 + min(lane, R - 1), p.M - 1));  // a row per lane: one chain of square root and division
            unsigned long long inv[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float f = __shfl_sync(0xffffffffu, inv_lane, r);
                inv[r] = pack2(f, f);
                if (m0 + r < p.M) {
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (4 * t + kStep * u < w1) put(m0 + r, 4 * t + kStep * u, v[r][u], inv[r], g[u]);
                }
            }
            if constexpr (kTail) fill(m0, 4 * t + kStep * U, inv);
        }
    } else {
        for (int m0 = 0; m0 < p.M; m0 += R) {
            unsigned long long inv[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float f = inverse(min(m0 + r, p.M - 1));
                inv[r] = pack2(f, f);
            }
            fill(m0, w0 + 4 * t, inv);
        }
    }
}

// The same for R rows too long to hold in registers, from row m0 on: read twice, 12 loads of a thread in flight (8 and 20: up to 5 % and 7 %
// slower). Eight warps are two for each scheduler, so what counts is the number of instructions: packed arithmetic, groups of exactly
// R rows, no bounds in whole batches. (Five rows of 11008 inputs took 10 us in the loops above; L2 gives them twice in 4.5.) Same sums as above.
template <int R>
__device__ __forceinline__ void norm_long(const GemvParams& p, __nv_bfloat16* xs, float* red, int m0, bool first, int w0, int w1) {
    constexpr int kThreads = kGemvWarps * 32, kStep = kThreads * 4, kBatch = 12 / R;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, n_in = p.n_in;
    const float* x = reinterpret_cast<const float*>(p.x) + (size_t)m0 * n_in + 4 * t;
    auto load = [&](ulonglong2 (&a)[kBatch][R], int i, int end, bool whole) {
#pragma unroll
        for (int b = 0; b < kBatch; ++b)
#pragma unroll
            for (int r = 0; r < R; ++r) {
                a[b][r] = make_ulonglong2(0ull, 0ull);
                if (whole || i + kStep * b + 4 * t < end) a[b][r] = *reinterpret_cast<const ulonglong2*>(x + (size_t)r * n_in + i + kStep * b);
            }
    };
    auto inverse = [&](int m) {
        const float* q = red + m * kGemvWarps;
        return 1.0f / sqrtf((((q[0] + q[1]) + (q[2] + q[3])) + ((q[4] + q[5]) + (q[6] + q[7]))) / (float)n_in + p.eps);
    };
    if (first) {
        unsigned long long ss[R][2] = {};
        auto add = [&](int i, bool whole) {
            ulonglong2 a[kBatch][R];
            load(a, i, n_in, whole);
#pragma unroll
            for (int b = 0; b < kBatch; ++b)
#pragma unroll
                for (int r = 0; r < R; ++r) ss[r][0] = ffma2(a[b][r].x, a[b][r].x, ss[r][0]), ss[r][1] = ffma2(a[b][r].y, a[b][r].y, ss[r][1]);
        };
        int i = 0;
        for (; i + kStep * kBatch <= n_in; i += kStep * kBatch) add(i, true);
        if (i < n_in) add(i, false);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            float a, b, c, d;
            unpack2(ss[r][0], a, b);
            unpack2(ss[r][1], c, d);
            const float s = warp_sum((a + b) + (c + d));
            if (lane == 0) red[(m0 + r) * kGemvWarps + warp] = s;
        }
        bar_sync(1, kThreads);
    }
    const float inv_lane = inverse(m0 + min(lane, R - 1));  // a row per lane: one chain of square root and division
    unsigned long long inv[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const float v = __shfl_sync(0xffffffffu, inv_lane, r);
        inv[r] = pack2(v, v);
    }
    __nv_bfloat16* to = xs + (size_t)m0 * p.xs_ld + 4 * t - w0;
    auto fill = [&](int i, bool whole) {
        ulonglong2 a[kBatch][R];
        load(a, i, w1, whole);
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            if (!whole && i + kStep * b + 4 * t >= w1) continue;
            const uint2 g = *reinterpret_cast<const uint2*>(p.gain + 4 * t + i + kStep * b);
            const unsigned long long g0 = bf2_to_f2(g.x), g1 = bf2_to_f2(g.y);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                float lo0, hi0, lo1, hi1;
                unpack2(fmul2(fmul2(a[b][r].x, inv[r]), g0), lo0, hi0);
                unpack2(fmul2(fmul2(a[b][r].y, inv[r]), g1), lo1, hi1);
                const __nv_bfloat162 y0 = __floats2bfloat162_rn(lo0, hi0), y1 = __floats2bfloat162_rn(lo1, hi1);
                *reinterpret_cast<uint2*>(to + (size_t)r * p.xs_ld + i + kStep * b) =
                    make_uint2(*reinterpret_cast<const uint32_t*>(&y0), *reinterpret_cast<const uint32_t*>(&y1));
            }
        }
    };
    int i = w0;
    for (; i + kStep * kBatch <= w1; i += kStep * kBatch) fill(i, true);
    if (i < w1) fill(i, false);
}

template <int N>
using Units = std::integral_constant<int, N>;

// BY_WARP: a group of rows is one warp's alone
template <int NB, int EPI, bool NORM, bool BY_WARP>
__global__ void __launch_bounds__(kGemvThreads, 1) gemv_kernel(const __grid_constant__ GemvParams p) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int M = p.M, n_in = p.n_in;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem_raw);  // [stages] bytes landed
    uint64_t* empty = full + kGemvMaxStages;                 // [stages] read by the multiplying warps
    uint64_t* acc_full = empty + kGemvMaxStages;             // [2] a group's sums of an epoch are in psum
    uint64_t* acc_empty = acc_full + 2;                      // [2] and have been read
    uint64_t* x_full = acc_empty + 2;                        // bf16 activations of a window landed
    int* flag = reinterpret_cast<int*>(x_full + 1);
    volatile int* gone = flag + 1;                           // a warp of this CTA has left
    float* red = reinterpret_cast<float*>(flag + 6);         // [kMaxRows][kGemvWarps] sums of squares
    float* psum = reinterpret_cast<float*>(smem_raw + kGemvHead);  // [2][kGemvWarps][group_rows * M]
    float* tot = psum + 2 * kGemvWarps * p.group_rows * M;         // [max_rows][M], when a row has more than one epoch
    __nv_bfloat16* xs = reinterpret_cast<__nv_bfloat16*>(smem_raw + p.off_xs);  // [M][xs_ld]
    unsigned char* ring = smem_raw + p.off_ring;
    volatile int* err = p.err;
    auto wait = [&](uint64_t* bar, int phase, int role, int item, int slot, int tag) {
        return mbar_wait_warp(bar, (uint32_t)(phase & 1), err, kErrGemvWait, role, item, slot, tag, gone);
    };
    bool ok = true;  // this warp has not left
    auto missing = [&]() {  // what is missing reads as NaN, and so does whatever else the CTA has written
        const int r0 = gemv_row(p, blockIdx.x), rows = gemv_row(p, blockIdx.x + 1) - r0;
        for (int i = lane; i < rows * M; i += 32) {
            const int m = i / rows, at = r0 + i - m * rows;
            if (EPI != kEpiSwiglu) reinterpret_cast<float*>(p.out)[(size_t)m * p.n_rows + at] = NAN;
            else if (at % 2 == 0) reinterpret_cast<__nv_bfloat16*>(p.out)[(size_t)m * (p.n_rows >> 1) + (at >> 1)] = __float2bfloat16_rn(NAN);
        }
    };

    if (tid == 0) {
        for (int s = 0; s < p.n_stages; ++s) mbar_init(&full[s], BY_WARP ? 1 : 2), mbar_init(&empty[s], BY_WARP ? 1 : kGemvWarps);
        for (int b = 0; b < 2; ++b) mbar_init(&acc_full[b], kGemvWarps), mbar_init(&acc_empty[b], 2);
        mbar_init(x_full, 1);
        *gone = 0;
        mbar_fence_init();
    }
    const int cta_row0 = gemv_row(p, blockIdx.x), cta_row1 = gemv_row(p, blockIdx.x + 1);
    pdl_launch_dependents();
    __syncthreads();
    pdl_wait();

    if (warp < kGemvWarps) {
        // ------------------------------------------------------------------------------------ multiply
        const int g = lane >> 2, q = lane & 3;
        int s = 0, lap = 0, n_x = 0, n_epoch = 0;
        float acc[NB][4];
        auto zero = [&]() {
#pragma unroll
            for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[nb][e] = 0.f;
        };
        // Sums of up to 1024 inputs from c0 on over the units of warp w, a lane's weight rows at wa and wb: its four units in pairs, each
        // with sums of its own
        const __nv_bfloat16* xr[NB];
        auto chunk = [&](const unsigned char* wa, const unsigned char* wb, int c0, int len, int w, auto units, bool whole, float (&sum)[NB][4]) {
            float t[2][NB][4] = {};
#pragma unroll
            for (int v = 0; v < decltype(units)::value; ++v) {
                const int u = c0 + (v * kGemvWarps + w) * 32;  // first input of the unit
                const bool in = whole || u + q * 8 < len;  // past the end of a ragged row lies whatever the stage held before
                uint4 a = make_uint4(0u, 0u, 0u, 0u), b = a;
                if (in) a = *reinterpret_cast<const uint4*>(wa + u * 2), b = *reinterpret_cast<const uint4*>(wb + u * 2);
#pragma unroll
                for (int nb = 0; nb < NB; ++nb) {
                    uint4 xv = make_uint4(0u, 0u, 0u, 0u);
                    if (in) xv = *reinterpret_cast<const uint4*>(xr[nb] + u);
                    float d0[4], d1[4];
                    mma_zero(d0, a.x, b.x, a.y, b.y, xv.x, xv.y);
                    mma_zero(d1, a.z, b.z, a.w, b.w, xv.z, xv.w);
#pragma unroll
                    for (int e = 0; e < 4; ++e) t[v & 1][nb][e] += d0[e] + d1[e];
                }
            }
#pragma unroll
            for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                for (int e = 0; e < 4; ++e) sum[nb][e] += t[0][nb][e] + t[1][nb][e];
        };
        zero();
        auto window = [&](bool first, int w0, int w1) {
            ++n_x;
            if (!NORM) return wait(x_full, n_x - 1, 0, n_x, 0, 1);
            if (!first) bar_sync(1, kGemvWarps * 32);  // the window before has been read
            // Registers hold 15 to 24 groups of four inputs of a thread, 8 of one row: six to eight rows of up to 3072 inputs all together, others of them five at a time,
            // 4096 five, 5120 three or two. (Six to eight rows in two batches, the second one's loads behind the first one's sums: 6 rows of 2048 -> 6144 8.6 us for
            // 8.4, 7 of 3000 -> 9000 13.0 for 12.4; nine together 2504 -> 1564 7.7 for 7.5.) Behind one row only is there a loop over what does not fit (nine
            // rows of 2056 -> 6145 with one 12.3 us, without 11.7).
            if (BY_WARP) {  // (at most 768 inputs)
                if (M == 1) norm_rows<1, 1, false>(p, xs, red, first, w0, w1);
                else norm_rows<5, 1, false>(p, xs, red, first, w0, w1);
            } else if (M == 1) norm_rows<1, 8, true>(p, xs, red, first, w0, w1);
            else if (n_in > 5120) {  // rows too long to hold in registers, in even shares of at most five
                if (M == 2) norm_long<2>(p, xs, red, 0, first, w0, w1);
                else if (M == 3 || M == 6) {
                    norm_long<3>(p, xs, red, 0, first, w0, w1);
                    if (M == 6) norm_long<3>(p, xs, red, 3, first, w0, w1);
                } else if (M == 5) norm_long<5>(p, xs, red, 0, first, w0, w1);
                else {
                    norm_long<4>(p, xs, red, 0, first, w0, w1);
                    if (M == 7) norm_long<3>(p, xs, red, 4, first, w0, w1);
                    if (M == 8) norm_long<4>(p, xs, red, 4, first, w0, w1);
                    if (M == 9) norm_long<5>(p, xs, red, 4, first, w0, w1);
                }
            } else if (M == 2) norm_rows<2, 5, false>(p, xs, red, first, w0, w1);
            else if (n_in <= 3072 && (M <= 5 || M == 9)) norm_rows<5, 3, false>(p, xs, red, first, w0, w1);
            else if (n_in <= 3072) norm_rows<8, 3, false>(p, xs, red, first, w0, w1);
            else if (n_in <= 4096) norm_rows<5, 4, false>(p, xs, red, first, w0, w1);
            else norm_rows<3, 5, false>(p, xs, red, first, w0, w1);
            bar_sync(1, kGemvWarps * 32);
            return true;
        };
        float s_warp[NB][2][3] = {};  // residual, by_warp: this lane's share of the sums of its activation rows
        // Short rows, many of them: a warp has every eighth group (and stage: it never waits for a phase while another warp has yet to see the
        // one before) to itself, with the sums of the eight shares kept apart and added as below, and runs their epilogue.
        auto rows_by_warp = [&]() {
            float* const out = reinterpret_cast<float*>(p.out);
#pragma unroll
            for (int nb = 0; nb < NB; ++nb) xr[nb] = xs + (size_t)min(nb * 8 + g, M - 1) * p.xs_ld + q * 8;
            float x0[NB][4];  // residual: the hidden state of the group
            auto request = [&](const GemvGroups& grp, float (&x)[NB][4]) {
#pragma unroll
                for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int m = nb * 8 + 2 * q + (e & 1), r = g + (e >> 1) * 8;
                        x[nb][e] = 0.f;
                        if (EPI == kEpiResidual && grp.o < p.groups && m < M && r < grp.rows) x[nb][e] = out[(size_t)m * p.n_rows + grp.row + r];
                    }
            };
            GemvGroups grp(p, cta_row0, cta_row1, warp, kGemvWarps);
            s = warp;
            while (grp.o < p.groups) {
                const int row = grp.row, rows = grp.rows;
                request(grp, x0);
                if (!wait(&full[s], lap, 0, grp.o, s, 6)) return false;
                const unsigned char* st = ring + (size_t)s * p.stage_bytes + q * 16;
                const unsigned char *wa = st + min(g, rows - 1) * p.pitch, *wb = st + min(g + 8, rows - 1) * p.pitch;
                float sum[kGemvWarps][NB][4] = {};
#pragma unroll
                for (int w = 0; w < kGemvWarps; ++w) {
                    if (n_in <= 256) chunk(wa, wb, 0, n_in, w, Units<1>(), false, sum[w]);
                    else if (n_in <= 512) chunk(wa, wb, 0, n_in, w, Units<2>(), false, sum[w]);
                    else chunk(wa, wb, 0, n_in, w, Units<3>(), false, sum[w]);
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&empty[s]);
#pragma unroll
                for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int m = nb * 8 + 2 * q + (e & 1), r = g + (e >> 1) * 8;
                        const bool mine = m < M && r < rows;
                        const float v = ((sum[0][nb][e] + sum[1][nb][e]) + (sum[2][nb][e] + sum[3][nb][e])) +
                                        ((sum[4][nb][e] + sum[5][nb][e]) + (sum[6][nb][e] + sum[7][nb][e]));
                        if (EPI == kEpiPlain) {
                            if (mine) out[(size_t)m * p.n_rows + row + r] = v;
                        } else if (EPI == kEpiSwiglu) {
                            const float up = __shfl_xor_sync(0xffffffffu, v, 4);
                            if (mine && (r & 1) == 0)
                                reinterpret_cast<__nv_bfloat16*>(p.out)[(size_t)m * (p.n_rows >> 1) + ((row + r) >> 1)] =
                                    __float2bfloat16_rn(v / (1.0f + expf(-v)) * up);
                        } else if (mine) {
                            const float y0 = x0[nb][e] + v;
                            out[(size_t)m * p.n_rows + row + r] = y0;
                            float* sw = s_warp[nb][e & 1];
                            sw[0] = fmaf(x0[nb][e], y0, sw[0]), sw[1] = fmaf(x0[nb][e], x0[nb][e], sw[1]), sw[2] = fmaf(y0, y0, sw[2]);
                        }
                    }
                grp.next();
                s += kGemvWarps;
                if (s >= p.n_stages) s = warp, ++lap;
            }
            return true;
        };
        if constexpr (BY_WARP) ok = window(true, 0, n_in) && rows_by_warp();
        else ok = gemv_walk(
            p, cta_row0, cta_row1, window,
            [&](int, int rows, int k0, int len, int w0) {
                if (!wait(&full[s], lap, 0, k0, s, 2)) return false;
                const unsigned char* st = ring + (size_t)s * p.stage_bytes + q * 16;
                const unsigned char *wa = st + min(g, rows - 1) * p.pitch, *wb = st + min(g + 8, rows - 1) * p.pitch;
#pragma unroll
                for (int nb = 0; nb < NB; ++nb) xr[nb] = xs + (size_t)min(nb * 8 + g, M - 1) * p.xs_ld + (k0 - w0) + q * 8;
                int c0 = 0;  // sums of 1024 inputs at a time, whatever the length of a piece
                for (; c0 + kGemvChunk <= len; c0 += kGemvChunk) chunk(wa, wb, c0, len, warp, Units<4>(), true, acc);
                if (c0 + 512 < len) chunk(wa, wb, c0, len, warp, Units<4>(), false, acc);
                else if (c0 < len) chunk(wa, wb, c0, len, warp, Units<2>(), false, acc);
                __syncwarp();
                if (lane == 0) mbar_arrive(&empty[s]);
                if (++s == p.n_stages) s = 0, ++lap;
                return true;
            },
            [&](int, int, int rows, int, int, bool) {
                const int b = n_epoch & 1;
                if (n_epoch >= 2 && !wait(&acc_empty[b], n_epoch / 2 - 1, 0, n_epoch, b, 3)) return false;
                ++n_epoch;
                float* dst = psum + (size_t)(b * kGemvWarps + warp) * p.group_rows * M;
#pragma unroll
                for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int m = nb * 8 + 2 * q + (e & 1), r = g + (e >> 1) * 8;
                        if (m < M && r < rows) dst[r * M + m] = acc[nb][e];
                    }
                zero();
                __syncwarp();
                if (lane == 0) mbar_arrive(&acc_full[b]);
                return true;
            });
        if (!ok) {
            *gone = 1;
            if (NORM)  // the barriers of the windows to come
                for (const int all = p.win < n_in ? p.n_blk * ((n_in + p.win - 1) / p.win) : 1; n_x < all; ++n_x)
                    bar_sync(1, kGemvWarps * 32), bar_sync(1, kGemvWarps * 32);
            if (BY_WARP) missing();
        }
        if (EPI == kEpiResidual && BY_WARP) {  // the warps' sums, added in order
#pragma unroll
            for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int j = 0; j < 3; ++j) {
                        float v = ok ? s_warp[nb][i][j] : NAN;
#pragma unroll
                        for (int o = 4; o < 32; o *= 2) v += __shfl_xor_sync(0xffffffffu, v, o);
                        const int m = nb * 8 + 2 * q + i;
                        if (g == 0 && m < M) psum[(warp * M + m) * 3 + j] = v;
                    }
            bar_sync(1, kGemvWarps * 32);
            if (tid < 3 * M) {
                float v = 0.f;
#pragma unroll
                for (int w = 0; w < kGemvWarps; ++w) v += psum[w * M * 3 + tid];
                p.partials[((size_t)blockIdx.x * kMaxRows + tid / 3) * 4 + tid % 3] = v;
            }
        }
    } else if (warp < kGemvWarps + 2) {
        // ------------------------------------------------------------------------------------ weights -> ring
        const int r8 = (warp - kGemvWarps) * 8;  // each of the two copies eight rows of a piece
        int s = 0, lap = 0;
        auto copy_group = [&](const GemvGroups& grp, int stage) {
            const uint32_t bytes = (uint32_t)(grp.rows * n_in * 2);
            mbar_expect_tx(&full[stage], bytes);
            tma_load_1d(ring + (size_t)stage * p.stage_bytes, p.W + (size_t)grp.row * n_in, bytes, &full[stage]);
        };
        // Groups of short rows: the first lap by the lanes of the first warp, a stage each, then every second one by either warp
        auto groups_of_rows = [&]() {
            if (r8 == 0 && lane < p.n_stages && lane < p.groups) copy_group(GemvGroups(p, cta_row0, cta_row1, lane, 2), lane);
            __syncwarp();
            s = warp - kGemvWarps, lap = 1;
            for (GemvGroups grp(p, cta_row0, cta_row1, p.n_stages + s, 2); grp.o < p.groups; grp.next()) {
                if (!wait(&empty[s], lap - 1, 1, grp.o, s, 7)) return false;
                if (lane == 0) copy_group(grp, s);
                s += 2;
                if (s >= p.n_stages) s = warp - kGemvWarps, ++lap;
            }
            return true;
        };
        if constexpr (BY_WARP) ok = groups_of_rows();
        else ok = gemv_walk(
            p, cta_row0, cta_row1, [&](bool, int, int) { return true; },
            [&](int row, int rows, int k0, int len, int) {
                if (lap > 0 && !wait(&empty[s], lap - 1, 1, k0, s, 4)) return false;
                // (the first lap beside an RMSNorm is the first one's alone: at full speed the weights keep the activations waiting; one and two
                // short rows are there first. us alone / both: one row 2048 -> 6144 7.4 / 7.0, 4096 -> 12288 18.3 / 18.6, 6000 -> 9000 19.8 / 20.2)
                const bool alone = NORM && lap == 0 && (M > 2 || n_in > 3072);
                const int r0 = alone && r8 > 0 ? rows : r8, mine = max(min(rows - r0, alone ? 16 : 8), 0);
                if (lane == 0) mbar_expect_tx(&full[s], (uint32_t)(mine * len * 2));
                __syncwarp();
                // (whole rows that lie in the ring as in memory: one copy)
                const int copies = p.whole ? min(mine, 1) : mine, bytes = p.whole ? mine * len * 2 : len * 2;
                if (lane < copies)
                    tma_load_1d(ring + (size_t)s * p.stage_bytes + (r0 + lane) * p.pitch, p.W + (size_t)(row + r0 + lane) * n_in + k0, (uint32_t)bytes, &full[s]);
                if (++s == p.n_stages) s = 0, ++lap;
                return true;
            },
            [&](int, int, int, int, int, bool) { return true; });
        if (!ok) *gone = 1;
        // what is in flight lands before the CTA leaves, also when this warp leaves early: at most the last piece of every stage, for
        // the ones before have been read
        const int next = lap * p.n_stages + s, end = BY_WARP ? min(next, p.groups) : next;
        for (int i = max(0, next - p.n_stages); i < end; i += BY_WARP ? 2 : 1)
            mbar_drain(&full[i % p.n_stages], (uint32_t)((i / p.n_stages) & 1));
    } else {
        // ------------------------------------------------------------------------------------ sums of the warps, epilogue
        const int et = tid - (kGemvWarps + 2) * 32, r = et & 15, m_first = et >> 4;  // weight row of the group, first activation row
        float* const out = reinterpret_cast<float*>(p.out);
        float s_loc[3][3] = {};  // residual: this thread's share of the sums of rows m_first + 4 i
        int n_epoch = 0, n_x = 0;
        auto request_x = [&](int w0, int w1) {  // bf16 activations of a window
            if (NORM || warp != kGemvWarps + 2) return;
            ++n_x;
            if (lane == 0) mbar_expect_tx(x_full, (uint32_t)(M * (w1 - w0) * 2));
            __syncwarp();
            if (lane < M) tma_load_1d(xs + (size_t)lane * p.xs_ld, reinterpret_cast<const __nv_bfloat16*>(p.x) + (size_t)lane * n_in + w0, (uint32_t)(w1 - w0) * 2, x_full);
        };
        int blocks_left = p.n_blk;
        if (cta_row1 > cta_row0) request_x(0, min(n_in, p.win));
        if constexpr (!BY_WARP) ok = gemv_walk(
            p, cta_row0, cta_row1, [&](bool, int, int) { return true; }, [&](int, int, int, int, int) { return true; },
            [&](int local, int row, int rows, int e0, int e1, bool win_end) {
                const bool last = e1 == n_in;
                float x0[3] = {0.f, 0.f, 0.f};
                if (EPI == kEpiResidual && last) {
#pragma unroll
                    for (int i = 0; i < 3; ++i)
                        if (r < rows && m_first + 4 * i < M) x0[i] = out[(size_t)(m_first + 4 * i) * p.n_rows + row + r];
                }
                const int b = n_epoch & 1;
                if (!wait(&acc_full[b], n_epoch / 2, 2, n_epoch, b, 5)) return false;
                ++n_epoch;
                // every multiplying warp has read the window
                if (win_end && p.win < n_in) {
                    if (!last) request_x(e1, min(n_in, e1 + p.win));
                    else if (--blocks_left > 0) request_x(0, p.win);
                }
                float v[3];
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    const int m = m_first + 4 * i;
                    v[i] = 0.f;
                    if (r < rows && m < M) {
                        const float* src = psum + (size_t)b * kGemvWarps * p.group_rows * M + r * M + m;
                        float w[kGemvWarps];
#pragma unroll
                        for (int j = 0; j < kGemvWarps; ++j) w[j] = src[j * p.group_rows * M];
#pragma unroll
                        for (int st = 1; st < kGemvWarps; st *= 2)
#pragma unroll
                            for (int j = 0; j < kGemvWarps; j += 2 * st) w[j] += w[j + st];
                        v[i] = w[0];
                        if (e0 > 0) v[i] = tot[(local + r) * M + m] + v[i];
                        if (!last) tot[(local + r) * M + m] = v[i];
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&acc_empty[b]);
                if (last) {
#pragma unroll
                    for (int i = 0; i < 3; ++i) {
                        const int m = m_first + 4 * i;
                        const bool mine = r < rows && m < M;
                        if (EPI == kEpiPlain) {
                            if (mine) out[(size_t)m * p.n_rows + row + r] = v[i];
                        } else if (EPI == kEpiSwiglu) {
                            const float up = __shfl_xor_sync(0xffffffffu, v[i], 1);
                            if (mine && (r & 1) == 0)
                                reinterpret_cast<__nv_bfloat16*>(p.out)[(size_t)m * (p.n_rows >> 1) + ((row + r) >> 1)] =
                                    __float2bfloat16_rn(v[i] / (1.0f + expf(-v[i])) * up);
                        } else if (mine) {
                            const float y0 = x0[i] + v[i];
                            out[(size_t)m * p.n_rows + row + r] = y0;
                            s_loc[i][0] = fmaf(x0[i], y0, s_loc[i][0]);
                            s_loc[i][1] = fmaf(x0[i], x0[i], s_loc[i][1]);
                            s_loc[i][2] = fmaf(y0, y0, s_loc[i][2]);
                        }
                    }
                }
                return true;
            });
        if (!ok) {
            *gone = 1;
            missing();
#pragma unroll
            for (int i = 0; i < 3; ++i) s_loc[i][0] = s_loc[i][1] = s_loc[i][2] = NAN;
        }
        if (n_x > 0) mbar_drain(x_full, (uint32_t)((n_x - 1) & 1));
        if (EPI == kEpiResidual && !BY_WARP) {
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    float v = s_loc[i][j];
#pragma unroll
                    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                    if (r == 0 && m_first + 4 * i < M) p.partials[((size_t)blockIdx.x * kMaxRows + m_first + 4 * i) * 4 + j] = v;
                }
        }
    }
    // whoever has set the error word comes here afterwards: no call leaves it set
    if (!ok) {
        __syncwarp();
        if (lane == 0) *err = kErrNone;
    }

    if (EPI == kEpiResidual) {
        if (last_cta_arrives(p.counter, flag)) {
            // one warp per activation row: lanes add the per-CTA partials b = lane, lane+32, ... in order, then an
            // xor butterfly in double precision (fixed order, independent of the row count)
            if (warp < M) {
                double sxy = 0, sxx = 0, syy = 0;
                for (unsigned b = lane; b < gridDim.x; b += 32) {
                    const float4 v = __ldcg(reinterpret_cast<const float4*>(p.partials + ((size_t)b * kMaxRows + warp) * 4));
                    sxy += (double)v.x, sxx += (double)v.y, syy += (double)v.z;
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    sxy += __shfl_xor_sync(0xffffffffu, sxy, o);
                    sxx += __shfl_xor_sync(0xffffffffu, sxx, o);
                    syy += __shfl_xor_sync(0xffffffffu, syy, o);
                }
                if (lane == 0) {
                    const double c = sxy / fmax(sqrt(sxx) * sqrt(syy), 1e-30);
                    p.cos_out[warp] = (float)c;
                }
            }
            if (tid == 0) *p.counter = 0u;
        }
    }
}

// ============================================================================================ host side
// The plan of one launch. The activations stay in shared memory whole, or in the longest windows (multiples of an epoch) that
// leave the ring kGemvRing bytes: the ring has to cover the memory latency and the prologue, a window costs a copy from L2
// that the ring covers.
constexpr size_t kGemvRing = 96 * 1024;
// Rows of up to 768 inputs are copied 16 at a time, as they lie in memory (their reads conflict in pairs: one row of 1000 -> 4000 4.6 us in
// copies by rows, 4.7 whole; 1024 -> 32000 13.5 and 14.5); a ring then has the eight stages that a group per warp needs with nine
// activation rows. A group per warp from 50 weight rows per SM on, four groups: 9472 x 256 6.0 -> 3.1 us, 9472 x 688 6.2 -> 4.8, but
// 4096 x 688 (two groups) 4.1 -> 4.6.
constexpr int kGemvWhole = 768, kGemvByWarp = 49;
static size_t plan_gemv(int max_smem, int sms, GemvParams* p) {
    const size_t M = p->M;
    auto magic = [](int d) { return d > 1 ? (unsigned)((1ull << 32) / (unsigned)d + 1) : 0u; };
    const int n_pairs = p->n_rows / 2 + p->n_rows % 2;
    p->cta_pairs = n_pairs / sms, p->cta_more = n_pairs % sms, p->div_grid = magic(sms);
    int max_rows = 2 * (p->cta_pairs + (p->cta_more > 0));
    p->whole = p->n_in <= kGemvWhole;
    p->by_warp = p->whole && max_rows >= kGemvByWarp && max_rows <= 32768;
    p->n_blk = p->by_warp ? 1 : (max_rows + kGemvBlockRows - 1) / kGemvBlockRows;
    if (p->n_blk > 1) max_rows = (max_rows + p->n_blk - 1) / p->n_blk + 2;  // block boundaries are even
    const int pairs = (max_rows + 1) / 2;
    p->groups = (pairs + 7) / 8, p->div_groups = magic(p->groups);
    p->group_rows = 2 * ((pairs + p->groups - 1) / p->groups);
    const size_t psum = (size_t)2 * kGemvWarps * p->group_rows * M * 4;
    const size_t tot = p->n_in > kGemvEpoch ? (size_t)(max_rows + 2) * M * 4 : 0;
    p->off_xs = (int)((kGemvHead + psum + tot + 127) / 128 * 128);
    auto window_bytes = [&](int win) { return M * ((size_t)(win + 63) / 64 * 128 + 64); };
    const size_t room = (size_t)max_smem - p->off_xs;
    p->win = p->n_in;
    if (window_bytes(p->win) + kGemvRing > room) {
        p->win = kGemvEpoch;
        while (p->win + kGemvEpoch < p->n_in && window_bytes(p->win + kGemvEpoch) + kGemvRing <= room) p->win += kGemvEpoch;
        p->win = std::min(p->win, p->n_in);
    }
    p->xs_ld = (p->win + 63) / 64 * 64 + 32;
    p->off_ring = (int)((p->off_xs + window_bytes(p->win) + 127) / 128 * 128);
    // The longer the pieces, the better the stream (copies of 1, 2 and 4 KB: 3.2, 5.4 and 6.2 TB/s), the shorter, the sooner it starts and
    // the less of it is left at the end: 4 KB from 4096 inputs on, where the ring then holds three (two from 8192 on). us with 2 KB -> 4 KB: one row
    // of 4096 -> 22016 33.8 -> 31.5, five of 13760 -> 5120 36.9 -> 36.1, one of 2048 -> 6144 10.0 -> 10.2, nine of 2056 -> 6145 12.3 -> 11.9 (the
    // only one of these short rows that gains).
    // The last piece of a row is up to half as long again (one row of 1032 -> 20000 16.4 -> 11.5 us, 6152 -> 8000 20.5 -> 18.1) where the ring keeps its
    // stages, or four (11008 -> 4096 with two stages for three 20.1 -> 20.8).
    auto ring = [&](int seg, bool tail) {
        const int left = p->n_in % seg;
        p->seg = seg;
        p->tail = tail && left <= seg / 2 && p->n_in % kGemvEpoch > left ? left : 0;
        p->pitch = p->whole ? p->n_in * 2 : (std::min(p->n_in, seg + p->tail) + 63) / 64 * 128 + 64;
        p->stage_bytes = p->group_rows * p->pitch;
        p->n_stages = std::min<int>(kGemvMaxStages, (max_smem - p->off_ring) / p->stage_bytes);
        return p->n_stages;
    };
    auto best = [&](int seg) {
        const int plain = ring(seg, false);
        return ring(seg, true) >= std::min(plain, 4) ? p->n_stages : ring(seg, false);
    };
    if (p->whole) ring(p->n_in, false);
    else if (p->n_in < 4096 || best(2048) < (p->n_in >= 8192 ? 2 : 3)) best(1024);
    if (p->by_warp) p->n_stages = p->n_stages / kGemvWarps * kGemvWarps;  // a stage is one warp's
    return (size_t)p->off_ring + (size_t)p->n_stages * p->stage_bytes;
}

using GemvKernel = void (*)(const GemvParams);
template <int NB, bool BY_WARP>
static GemvKernel gemv_pick(int epi, bool norm) {
    switch (epi) {
        case kEpiPlain: return norm ? gemv_kernel<NB, kEpiPlain, true, BY_WARP> : gemv_kernel<NB, kEpiPlain, false, BY_WARP>;
        case kEpiSwiglu: return norm ? gemv_kernel<NB, kEpiSwiglu, true, BY_WARP> : gemv_kernel<NB, kEpiSwiglu, false, BY_WARP>;
    }
    return norm ? gemv_kernel<NB, kEpiResidual, true, BY_WARP> : gemv_kernel<NB, kEpiResidual, false, BY_WARP>;
}
static GemvKernel gemv_pick(int M, int epi, bool norm, bool by_warp) {
    if (M > 8) return by_warp ? gemv_pick<2, true>(epi, norm) : gemv_pick<2, false>(epi, norm);
    return by_warp ? gemv_pick<1, true>(epi, norm) : gemv_pick<1, false>(epi, norm);
}

cudaError_t launch_gemv(GemvParams p, int epi, bool norm, int max_smem, int sms, cudaStream_t s) {
    const size_t smem = plan_gemv(max_smem, sms, &p);
    if (p.n_stages < 2) return cudaErrorInvalidValue;
    return launch_pdl(gemv_pick(p.M, epi, norm, p.by_warp), dim3(sms), dim3(kGemvThreads), smem, s, 1, p);
}

cudaError_t configure_gemv(int max_smem) {
    for (int M : {1, kMaxRows})
        for (int epi : {kEpiPlain, kEpiSwiglu, kEpiResidual})
            for (bool norm : {false, true})
                for (bool by_warp : {false, true}) {
                    const cudaError_t e = cudaFuncSetAttribute(gemv_pick(M, epi, norm, by_warp), cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
                    if (e != cudaSuccess) return e;
                }
    return cudaSuccess;
}

}  // namespace asd
