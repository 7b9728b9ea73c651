// Fused RMSNorm -> GEMV -> epilogue for M <= 9 activation rows as a launch of its own (asd_fused_gemv).
//
// One CTA per SM owns a contiguous slab of weight rows and streams it exactly once through a ring of shared memory: a
// producer warp copies pieces of up to 16 weight rows x 1024 or 2048 inputs, one bulk copy per row, and runs as far ahead as the
// ring holds. Eight warps multiply: every warp takes the 32-input units u, u + 8, ... of a piece on mma.sync m16n8k16 with the weights
// as the 16-row operand and the activation rows as the 8 columns. A lane reads 16 bytes (8 inputs) of weight rows g and
// g + 8 straight into operand registers, four inputs per MMA; the order of the inputs inside a dot product is free, so the
// same lane supplies the same 8 inputs of activation row g. Two more warps add the eight warps' sums of a group of rows and
// run the epilogue while the others multiply the next group.
//
// Sums: the 16 x 8 result of every MMA starts from zero and the results are added on the CUDA cores; a warp's sums of a
// group go to shared memory every kGemvEpoch inputs, where the eight warps' sums are added as a tree and then to the row's
// total. A sum of 16 products is nearly exact and no chain of additions is long (error against 64 bits 8.8e-8 of the result at
// 13760 inputs; 9.1e-8 with the chains of the kernel before). Chunks of 1024 inputs, epochs and groups depend on the
// matrix and the SM count alone: row m of an M-row call is bit-identical to the same row of a one-row call. Rows of weights
// are 64 bytes apart modulo 128 in shared memory, so the eight lanes of a 16-byte read phase (two rows) meet no conflict.
//
// What bounds it: the weight stream and, for small matrices, launch, first bytes and last sums. With the weights loaded straight into
// operand registers (16 warps, 4 to 8 KB in flight each) the stream waited for the RMSNorm in front of it and shared its
// scoreboards with the products. Launch after launch over matrices that L2 does not hold,
// us before -> now: 1 row 2048 -> 6144 9.6 -> 7.7, 4096 -> 22016 SwiGLU 36.8 -> 31.7 (5.7 TB/s), 8192 -> 24576 69.3 -> 63.7 (6.3 TB/s);
// 5 rows 1024 -> 12000 11.6 -> 9.1, 13760 -> 5120 residual 36.2 -> 32.7; 9 rows 2056 -> 6145 16.0 -> 12.9, 11008 -> 4096 residual 32.6 -> 26.6,
// 13760 -> 5120 44.8 -> 38.5, 4096 -> 22016 44.8 -> 43.2; 26 shapes of one to nine rows: none slower. Behind an RMSNorm, 32 shapes of one and
// five rows: 1.01 to 1.5 times as fast but for five rows of more than 11000 inputs (11008 -> 4096 30.2 -> 31.4, 13760 -> 5120 44.2 -> 44.7, 22016 ->
// 8192 79.7 -> 90.2), whose norm reads the rows twice with eight warps where it had sixteen.
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
constexpr int kGemvThreads = (kGemvWarps + 3) * 32;  // multiplying warps, producer, two epilogue warps
constexpr int kGemvHead = 1024;      // bytes in front: barriers, flag, sums of squares
constexpr int kErrGemvWait = 21;

// first row of CTA b; the boundaries are even so that gate_i and up_i stay together
__host__ __device__ __forceinline__ int gemv_row(int n_rows, int grid, int b) {
    const int n_pairs = (n_rows + 1) >> 1;
    const int r = 2 * (int)((long long)b * n_pairs / grid);
    return r < n_rows ? r : n_rows;
}

__device__ __forceinline__ void mma_zero(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}

// Signal arrival of this CTA; returns true in every thread of the last CTA to arrive.
__device__ __forceinline__ bool last_cta_arrives(unsigned* counter, int* flag_smem) {
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned t = atomicAdd(counter, 1u);
        *flag_smem = (t == gridDim.x - 1) ? 1 : 0;
    }
    __syncthreads();
    const bool last = *flag_smem != 0;
    if (last) __threadfence();
    return last;
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
        const int blk0 = row0 + (row1 - row0) * blk / p.n_blk / 2 * 2;
        const int rows = (blk + 1 == p.n_blk ? row1 : row0 + (row1 - row0) * (blk + 1) / p.n_blk / 2 * 2) - blk0;
        const int pairs = (rows + 1) >> 1;
        if (rows <= 0) break;  // fewer pairs of rows than CTAs
        for (int w0 = 0; w0 < p.n_in; w0 += p.win) {
            const int w1 = min(p.n_in, w0 + p.win);
            if ((blk == 0 || p.win < p.n_in) && !window(blk + w0 == 0, w0, w1)) return false;
            for (int o = 0; o < p.groups; ++o) {
                const int r0 = 2 * (o * pairs / p.groups), n = min(rows, 2 * ((o + 1) * pairs / p.groups)) - r0;
                for (int e0 = w0; e0 < w1; e0 += kGemvEpoch) {
                    const int e1 = min(w1, e0 + kGemvEpoch);
                    for (int k0 = e0; k0 < e1; k0 += p.seg)
                        if (!piece(blk0 + r0, n, k0, min(p.seg, e1 - k0), w0)) return false;
                    if (!epoch(r0, blk0 + r0, n, e0, e1, o + 1 == p.groups && e1 == w1)) return false;
                }
            }
        }
    }
    return true;
}

// RMSNorm of the activation rows into the window of inputs w0 .. w1, by the multiplying warps: R rows of up to U x 1024 inputs at a
// time are read once, all loads in flight together, and normalised from registers; what lies behind, and every window after
// the first, is read twice, 8 to 16 loads of a thread at a time. Thread t adds the squares of inputs
// 4 t + 1024 u in this order whatever R and U.
template <int R, int U, bool kTail>
__device__ __forceinline__ void norm_rows(const GemvParams& p, __nv_bfloat16* xs, float* red, bool first, int w0, int w1) {
    constexpr int kThreads = kGemvWarps * 32, kStep = kThreads * 4, kBatch = R == 1 ? 8 : 16 / R, kHeld = U > 0 ? U : 1;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, n_in = p.n_in;
    const float* xf = reinterpret_cast<const float*>(p.x);
    auto load = [&](int m, int i) { return *reinterpret_cast<const float4*>(xf + (size_t)m * n_in + i); };
    auto inverse = [&](int m) {  // of the row's root mean square
        const float* r = red + m * kGemvWarps;
        const float s = ((r[0] + r[1]) + (r[2] + r[3])) + ((r[4] + r[5]) + (r[6] + r[7]));
        return 1.0f / sqrtf(s / (float)n_in + p.eps);
    };
    auto put = [&](int m, int i, const float4& a, float inv, const uint2& gn) {
        uint2 o;
        const __nv_bfloat162 lo = __floats2bfloat162_rn(a.x * inv * bf_lo(gn.x), a.y * inv * bf_hi(gn.x));
        const __nv_bfloat162 hi = __floats2bfloat162_rn(a.z * inv * bf_lo(gn.y), a.w * inv * bf_hi(gn.y));
        o.x = *reinterpret_cast<const uint32_t*>(&lo);
        o.y = *reinterpret_cast<const uint32_t*>(&hi);
        *reinterpret_cast<uint2*>(xs + (size_t)m * p.xs_ld + (i - w0)) = o;
    };
    auto gain = [&](int i) { return *reinterpret_cast<const uint2*>(p.gain + i); };
    static_assert(kGemvWarps == 8, "sums of squares of eight warps");
    auto load_batch = [&](float4 (&a)[kBatch][R], int m0, int i, int end) {
#pragma unroll
        for (int b = 0; b < kBatch; ++b)
#pragma unroll
            for (int r = 0; r < R; ++r) {
                a[b][r] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (m0 + r < p.M && i + kStep * b < end) a[b][r] = load(m0 + r, i + kStep * b);
            }
    };
    auto fill = [&](int m0, int i, const float (&inv)[R]) {  // inputs i, i + 1024, ... of these rows
        for (; i < w1; i += kStep * kBatch) {
            float4 a[kBatch][R];
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
            float4 v[R][kHeld];
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    v[r][u] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (m0 + r < p.M && 4 * t + kStep * u < n_in) v[r][u] = load(m0 + r, 4 * t + kStep * u);
                }
            float4 ss[R];
            auto add = [&](float4& t4, const float4& a) {
                t4.x = fmaf(a.x, a.x, t4.x), t4.y = fmaf(a.y, a.y, t4.y), t4.z = fmaf(a.z, a.z, t4.z), t4.w = fmaf(a.w, a.w, t4.w);
            };
#pragma unroll
            for (int r = 0; r < R; ++r) {
                ss[r] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int u = 0; u < U; ++u) add(ss[r], v[r][u]);
            }
            if constexpr (kTail)
                for (int i = 4 * t + kStep * U; i < n_in; i += kStep * kBatch) {
                    float4 a[kBatch][R];
                    load_batch(a, m0, i, n_in);
#pragma unroll
                    for (int b = 0; b < kBatch; ++b)
#pragma unroll
                        for (int r = 0; r < R; ++r) add(ss[r], a[b][r]);
                }
            float s[R];
#pragma unroll
            for (int r = 0; r < R; ++r) s[r] = (ss[r].x + ss[r].y) + (ss[r].z + ss[r].w);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int r = 0; r < R; ++r) s[r] += __shfl_xor_sync(0xffffffffu, s[r], o);
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (lane == 0 && m0 + r < p.M) red[(m0 + r) * kGemvWarps + warp] = s[r];
            bar_sync(1, kThreads);
            const float inv_lane = inverse(min(m0 + min(lane, R - 1), p.M - 1));  // a row per lane: one chain of square root and division
            float inv[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                inv[r] = __shfl_sync(0xffffffffu, inv_lane, r);
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
            float inv[R];
#pragma unroll
            for (int r = 0; r < R; ++r) inv[r] = inverse(min(m0 + r, p.M - 1));
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

template <int NB, int EPI, bool NORM>
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

    if (tid == 0) {
        for (int s = 0; s < p.n_stages; ++s) mbar_init(&full[s], 1), mbar_init(&empty[s], kGemvWarps);
        for (int b = 0; b < 2; ++b) mbar_init(&acc_full[b], kGemvWarps), mbar_init(&acc_empty[b], 2);
        mbar_init(x_full, 1);
        *gone = 0;
        mbar_fence_init();
    }
    pdl_launch_dependents();
    __syncthreads();
    pdl_wait();

    const int cta_row0 = gemv_row(p.n_rows, gridDim.x, blockIdx.x), cta_row1 = gemv_row(p.n_rows, gridDim.x, blockIdx.x + 1);
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
        zero();
        ok = gemv_walk(
            p, cta_row0, cta_row1,
            [&](bool first, int w0, int w1) {
                ++n_x;
                if (!NORM) return wait(x_full, n_x - 1, 0, n_x, 0, 1);
                if (!first) bar_sync(1, kGemvWarps * 32);  // the window before has been read
                // Without a loop over what lies behind, the kernels of up to 5120 inputs run faster as well (one row of 4096 -> 11008 SwiGLU 17.8 ->
                // 16.2 us, nine of 2056 -> 6145 12.3 -> 11.7); five rows of 22016 -> 8192 with one load at a time 102 us, in batches 90.
                if (M == 1) norm_rows<1, 8, true>(p, xs, red, first, w0, w1);
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
                }
                else if (M == 2) norm_rows<2, 5, false>(p, xs, red, first, w0, w1);
                else if (n_in <= 3072) norm_rows<5, 3, false>(p, xs, red, first, w0, w1);
                else if (n_in <= 4096) norm_rows<5, 4, false>(p, xs, red, first, w0, w1);
                else norm_rows<3, 5, false>(p, xs, red, first, w0, w1);
                bar_sync(1, kGemvWarps * 32);
                return true;
            },
            [&](int, int rows, int k0, int len, int w0) {
                if (!wait(&full[s], lap, 0, k0, s, 2)) return false;
                const unsigned char* st = ring + (size_t)s * p.stage_bytes + q * 16;
                const unsigned char *wa = st + min(g, rows - 1) * p.pitch, *wb = st + min(g + 8, rows - 1) * p.pitch;
                // Sums of 1024 inputs at a time, whatever the length of a piece; a warp's four units in pairs, each with sums of its own
                const __nv_bfloat16* xr[NB];
#pragma unroll
                for (int nb = 0; nb < NB; ++nb) xr[nb] = xs + (size_t)min(nb * 8 + g, M - 1) * p.xs_ld + (k0 - w0) + q * 8;
                auto chunk = [&](int c0, auto whole) {
                    float t[2][NB][4] = {};
#pragma unroll
                    for (int v = 0; v < kGemvChunk / (kGemvWarps * 32); ++v) {
                        const int u = c0 + (v * kGemvWarps + warp) * 32;  // first input of the unit
                        const bool in = decltype(whole)::value || u + q * 8 < len;  // past the end of a ragged row lies whatever the stage held before
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
                        for (int e = 0; e < 4; ++e) acc[nb][e] += t[0][nb][e] + t[1][nb][e];
                };
                int c0 = 0;
                for (; c0 + kGemvChunk <= len; c0 += kGemvChunk) chunk(c0, std::true_type());
                if (c0 < len) chunk(c0, std::false_type());
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
        }
    } else if (warp == kGemvWarps) {
        // ------------------------------------------------------------------------------------ weights -> ring
        int s = 0, lap = 0;
        ok = gemv_walk(
            p, cta_row0, cta_row1, [&](bool, int, int) { return true; },
            [&](int row, int rows, int k0, int len, int) {
                if (lap > 0 && !wait(&empty[s], lap - 1, 1, k0, s, 4)) return false;
                if (lane == 0) mbar_expect_tx(&full[s], (uint32_t)(rows * len * 2));
                __syncwarp();
                if (lane < rows)
                    tma_load_1d(ring + (size_t)s * p.stage_bytes + lane * p.pitch, p.W + (size_t)(row + lane) * n_in + k0, (uint32_t)len * 2, &full[s]);
                if (++s == p.n_stages) s = 0, ++lap;
                return true;
            },
            [&](int, int, int, int, int, bool) { return true; });
        if (!ok) *gone = 1;
        // what is in flight lands before the CTA leaves, also when this warp leaves early: at most the last piece of every stage, for
        // the ones before have been read
        for (int i = max(0, (lap - 1) * p.n_stages + s); i < lap * p.n_stages + s; ++i)
            mbar_drain(&full[i % p.n_stages], (uint32_t)((i / p.n_stages) & 1));
    } else {
        // ------------------------------------------------------------------------------------ sums of the warps, epilogue
        const int et = tid - (kGemvWarps + 1) * 32, r = et & 15, m_first = et >> 4;  // weight row of the group, first activation row
        float* const out = reinterpret_cast<float*>(p.out);
        float s_loc[3][3] = {};  // residual: this thread's share of the sums of rows m_first + 4 i
        int n_epoch = 0, n_x = 0;
        auto request_x = [&](int w0, int w1) {  // bf16 activations of a window
            if (NORM || warp != kGemvWarps + 1) return;
            ++n_x;
            if (lane == 0) mbar_expect_tx(x_full, (uint32_t)(M * (w1 - w0) * 2));
            __syncwarp();
            if (lane < M) tma_load_1d(xs + (size_t)lane * p.xs_ld, reinterpret_cast<const __nv_bfloat16*>(p.x) + (size_t)lane * n_in + w0, (uint32_t)(w1 - w0) * 2, x_full);
        };
        int blocks_left = p.n_blk;
        if (cta_row1 > cta_row0) request_x(0, min(n_in, p.win));
        ok = gemv_walk(
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
        if (!ok) {  // what is missing reads as NaN, and so does whatever else the CTA has written
            *gone = 1;
            for (int i = lane; i < (cta_row1 - cta_row0) * M; i += 32) {
                const int m = i / (cta_row1 - cta_row0), at = cta_row0 + i - m * (cta_row1 - cta_row0);
                if (EPI != kEpiSwiglu) out[(size_t)m * p.n_rows + at] = NAN;
                else if (at % 2 == 0) reinterpret_cast<__nv_bfloat16*>(p.out)[(size_t)m * (p.n_rows >> 1) + (at >> 1)] = __float2bfloat16_rn(NAN);
            }
#pragma unroll
            for (int i = 0; i < 3; ++i) s_loc[i][0] = s_loc[i][1] = s_loc[i][2] = NAN;
        }
        if (n_x > 0) mbar_drain(x_full, (uint32_t)((n_x - 1) & 1));
        if (EPI == kEpiResidual) {
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
static size_t plan_gemv(int max_smem, int sms, GemvParams* p) {
    const size_t M = p->M;
    int max_rows = 2 * (((p->n_rows + 1) / 2 + sms - 1) / sms);  // (a loop over gemv_row costs the host two microseconds)
    p->n_blk = (max_rows + kGemvBlockRows - 1) / kGemvBlockRows;
    if (p->n_blk > 1) max_rows = (max_rows + p->n_blk - 1) / p->n_blk + 2;  // block boundaries are even
    const int pairs = (max_rows + 1) / 2;
    p->groups = (pairs + 7) / 8;
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
    for (p->seg = p->n_in >= 4096 ? 2048 : 1024;; p->seg = 1024) {
        p->pitch = (std::min(p->n_in, p->seg) + 63) / 64 * 128 + 64;
        p->stage_bytes = p->group_rows * p->pitch;
        p->n_stages = std::min<int>(kGemvMaxStages, (max_smem - p->off_ring) / p->stage_bytes);
        if (p->seg == 1024 || p->n_stages >= (p->n_in >= 8192 ? 2 : 3)) break;
    }
    return (size_t)p->off_ring + (size_t)p->n_stages * p->stage_bytes;
}

template <int NB>
static void (*gemv_pick(int epi, bool norm))(const GemvParams) {
    switch (epi) {
        case kEpiPlain: return norm ? gemv_kernel<NB, kEpiPlain, true> : gemv_kernel<NB, kEpiPlain, false>;
        case kEpiSwiglu: return norm ? gemv_kernel<NB, kEpiSwiglu, true> : gemv_kernel<NB, kEpiSwiglu, false>;
    }
    return norm ? gemv_kernel<NB, kEpiResidual, true> : gemv_kernel<NB, kEpiResidual, false>;
}

cudaError_t launch_gemv(GemvParams p, int epi, bool norm, int max_smem, int sms, cudaStream_t s) {
    const size_t smem = plan_gemv(max_smem, sms, &p);
    if (p.n_stages < 2) return cudaErrorInvalidValue;
    return launch_pdl(p.M > 8 ? gemv_pick<2>(epi, norm) : gemv_pick<1>(epi, norm), dim3(sms), dim3(kGemvThreads), smem, s, 1, p);
}

cudaError_t configure_gemv(int max_smem) {
    for (int epi : {kEpiPlain, kEpiSwiglu, kEpiResidual})
        for (bool norm : {false, true}) {
            cudaError_t e = cudaFuncSetAttribute(gemv_pick<1>(epi, norm), cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
            if (e == cudaSuccess) e = cudaFuncSetAttribute(gemv_pick<2>(epi, norm), cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

}  // namespace asd
