// Fused RMSNorm -> GEMV -> epilogue for M <= 9 activation rows as a launch of its own (asd_fused_gemv).
//
// One CTA per SM owns a contiguous slab of weight rows and streams it exactly once with 16-byte read-only loads. The
// products run on mma.sync m16n8k16 with the weights as the 16-row operand and the activation rows as the 8 columns:
// a lane loads 16 bytes (8 inputs) of weight rows g and g + 8 straight into operand registers, four inputs per MMA; the
// order of the inputs inside a dot product is free, so the same lane supplies the same 8 inputs of activation row g from
// shared memory. The 16 x 8 result of every MMA starts from zero and the results are added on the CUDA cores, first the
// eight of a segment in pairs, then to the running fp32 sums, which go to shared memory every eight segments: a sum of 16
// products is nearly exact and no chain of additions is long, so the result is no further from 64 bits than sums of fp32
// FMAs were (0.8-1.0e-7 against 0.8-1.1e-7, 2048 to 22016 inputs).
//
// Work items: the CTA's rows are cut into groups of at most 16, a group's inputs into segments of kGemvSeg, and the
// segments of a group are dealt to `split` sub-items (segment s to sub-item s mod split), so that the CTA's 16 warps have
// equal shares whatever the number of rows. A warp walks its sub-items with the weights of two segments in registers:
// a segment's eight loads per lane are reissued as soon as its MMAs have read the registers, so one to two segments (4-8 KB)
// per warp are in flight. (Four segments of half the length would keep more in flight, but the loads then share
// the warp's scoreboards and a wait for one segment waits for the next as well: 85 us instead of 64 us at 22016 x 8192.)
// Every sub-item keeps its sums in one place of shared memory and the epilogue adds the sub-items in order. Groups, segments
// and split depend on the matrix and the SM count alone: row m of an M-row call is bit-identical to the same row of a
// one-row call. The activations sit in shared memory as bf16, all of them or window by window when they do not fit.
//
// What bounds it: from about 50 MB on the stream and its start and end, below the chain launch -> x -> RMSNorm -> stream ->
// epilogue. With fp32 FMAs in the place of the MMAs the kernel was issue-bound from two rows on (widening, and shuffles of
// 2 M sums per 2048 weights): 13760 -> 5120 with five rows 54 -> 36 us (one row 33 -> 33), 4096 -> 22016 with nine rows 84 ->
// 47 us (one row 34 -> 36), 22016 -> 8192 with nine rows 185 -> 85 us.
//
// Epilogues
//   plain    : out[m][r] = a                                   (fp32)
//   swiglu   : t[m][i] = bf16(silu(gate_i) * up_i), gate_i and up_i neighbouring rows
//   residual : y = x + a in place; per-row <x,y>, |x|^2, |y|^2 by one warp per activation row, and the last CTA to
//              arrive turns the per-CTA partials into the cosine similarity of the hidden state before and after the
//              sublayer (summand of C_l, Section 3.2)
#pragma once
#include <limits.h>

#include "common.cuh"

namespace asd {

constexpr int kGemvSeg = 128;        // inputs per segment: 256 bytes of a weight row, eight loads per lane
constexpr int kGemvRun = 2;          // segments in a row that go to one sub-item: 512 bytes of each weight row
constexpr int kGemvDepth = 2;        // segments of a warp in registers
constexpr int kGemvBlockRows = 256;  // most weight rows whose sums are in shared memory at a time
constexpr int kGemvMaxSub = 48;      // sub-items of a block
constexpr int kGemvPad = 32;         // bf16 between activation rows: 64 bytes, conflict-free 16-byte operand reads

// first row of CTA b; the boundaries are even so that gate_i and up_i stay together
__host__ __device__ __forceinline__ int gemv_row(int n_rows, int grid, int b) {
    const int n_pairs = (n_rows + 1) >> 1;
    const int r = 2 * (int)((long long)b * n_pairs / grid);
    return r < n_rows ? r : n_rows;
}
// bytes in front of the activation window for M rows: reduction scratch, sums of the sub-items, hidden state before and after
__host__ __device__ __forceinline__ int gemv_fixed_smem(int M, int max_sub, int max_rows) {
    return kGemvWarps * kMaxRows * 4 * 4 + 32 + max_sub * 16 * M * 8 + (max_rows + 1) / 2 * 2 * M * 8;
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

template <int M, int EPI, bool NORM>
__global__ void __launch_bounds__(kGemvThreads, 1) gemv_kernel(const __grid_constant__ GemvParams p) {
    constexpr int NB = (M + 7) / 8;  // column blocks of 8 activation rows
    constexpr int kSteps = kGemvSeg / 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    pdl_launch_dependents();
    pdl_wait();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, q = lane & 3;
    const int n_in = p.n_in;
    const int n_seg = (n_in + kGemvSeg - 1) / kGemvSeg;
    const int cta_row0 = gemv_row(p.n_rows, gridDim.x, blockIdx.x), cta_row1 = gemv_row(p.n_rows, gridDim.x, blockIdx.x + 1);
    const int win_segs = p.win_segs, n_win = (n_seg + win_segs - 1) / win_segs;
    const int ld = win_segs * kGemvSeg + kGemvPad;  // bf16 per activation row in shared memory

    float* red = reinterpret_cast<float*>(smem_raw);              // [kGemvWarps][kMaxRows * 4]
    int* flag = reinterpret_cast<int*>(red + kGemvWarps * kMaxRows * 4);
    float2* psum = reinterpret_cast<float2*>(flag + 8);           // [max_sub][16][M]: (sum of whole runs of eight segments, sum of the rest)
    float2* xy = psum + p.max_sub * 16 * M;  // [max_rows][M]: hidden state before and after
    __nv_bfloat16* xs = reinterpret_cast<__nv_bfloat16*>(xy + (p.max_rows + 1) / 2 * 2 * M);  // [M][ld]

    float s_loc[3] = {0.f, 0.f, 0.f};  // residual: this lane's share of the sums of row `warp`
    const int n_blk = p.n_blk;
    for (int blk = 0; blk < n_blk; ++blk) {
        const int blk0 = cta_row0 + (cta_row1 - cta_row0) * blk / n_blk / 2 * 2;
        const int rows = (blk + 1 == n_blk ? cta_row1 : cta_row0 + (cta_row1 - cta_row0) * (blk + 1) / n_blk / 2 * 2) - blk0;
        if (rows <= 0) break;  // fewer pairs of rows than CTAs
        const int groups = (rows + 15) / 16, split = p.split, n_sub = groups * split;
        for (int win = 0; win < n_win; ++win) {
            const int seg0 = win * win_segs, win_end = min(seg0 + win_segs, n_seg);
            // load cursor over the (sub-item, segment) pairs of this warp inside the window, and the lane's weight rows there
            int sub = warp, seg = 0;
            const __nv_bfloat16 *wa = nullptr, *wb = nullptr;
            auto open = [&]() {  // the first segment of sub-item `sub` in the window (windows begin at multiples of split)
                const int o = sub / split;
                const int ra = o * rows / groups + g, rb = (o + 1) * rows / groups;
                seg = seg0 + (sub - o * split) * kGemvRun;
                wa = ra < rb ? p.W + (size_t)(blk0 + ra) * n_in + q * 8 : nullptr;
                wb = ra + 8 < rb ? p.W + (size_t)(blk0 + ra + 8) * n_in + q * 8 : nullptr;
            };
            auto settle = [&]() {  // past the end of a sub-item: on to this warp's next one
                while (seg >= win_end && sub < n_sub) {
                    sub += kGemvWarps;
                    if (sub < n_sub) open();
                }
            };
            uint4 buf[kGemvDepth][2 * kSteps];                       // rows g and g + 8, two steps of 32 inputs
            int at_sub[kGemvDepth], at_k[kGemvDepth];  // what the buffer holds (sub-item >= n_sub: nothing)
            auto fetch = [&](uint4 (&w)[2 * kSteps], int& ws, int& wk) {
                ws = sub, wk = seg * kGemvSeg;
                if (sub < n_sub) {
                    const int left = n_in - 8 * q - wk;  // inputs from this lane's first one to the end of the row
#pragma unroll
                    for (int i = 0; i < kSteps; ++i) {
                        w[2 * i] = (wa && i * 32 < left) ? ldg_stream(wa + wk + i * 32) : make_uint4(0, 0, 0, 0);
                        w[2 * i + 1] = (wb && i * 32 < left) ? ldg_stream(wb + wk + i * 32) : make_uint4(0, 0, 0, 0);
                    }
                    seg += (seg + 1) % kGemvRun ? 1 : (split - 1) * kGemvRun + 1;
                    settle();
                }
            };
            if (sub < n_sub) open(), settle();
            // the weights do not depend on the activations: get the first ones moving before the prologue (one segment beside an
            // RMSNorm of several rows, which needs registers as well), the others before the wait at its end
            constexpr int kEarly = !NORM || M == 1 ? kGemvDepth : 1;
#pragma unroll
            for (int d = 0; d < kEarly; ++d) fetch(buf[d], at_sub[d], at_k[d]);

            // ---- activations of this window -> bf16 rows in shared memory (RMSNorm fused here)
            if (blk + win > 0) __syncthreads();  // the previous window and the previous block's sums have been read
            if (n_win > 1 || blk == 0) {
                const int k0 = seg0 * kGemvSeg, k1 = min(n_in, win_end * kGemvSeg), k_pad = (win_end - seg0) * kGemvSeg;
                if (NORM) {
                    const float* xf = reinterpret_cast<const float*>(p.x);
                    // Up to five rows: all of them at a time, several loads of a row in flight together for one and two, and rows that
                    // fit the registers are read once. More rows go through the registers three at a time and are read again
                    // from L1 and L2 for their normalisation: beside the weights of a segment there is no room for all of them (seven
                    // and nine rows of 64 shapes 9 and 10 % faster, five rows 1 % slower that way).
                    constexpr int U = M == 1 ? 4 : (M == 2 ? 2 : 1), R = M <= 5 ? M : 3;
                    const bool in_regs = M <= 5 && n_in <= kGemvThreads * 4 * U && n_win == 1;
                    float4 v[U][R];
#pragma unroll
                    for (int u = 0; u < U; ++u)  // threads behind the end of the row store zeros
#pragma unroll
                        for (int m = 0; m < R; ++m) v[u][m] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (win == 0 && blk == 0) {
#pragma unroll
                        for (int m0 = 0; m0 < M; m0 += R) {
                            float ss[R];
#pragma unroll
                            for (int m = 0; m < R; ++m) ss[m] = 0.f;
                            for (int i0 = tid * 4; i0 < n_in; i0 += kGemvThreads * 4 * U) {
#pragma unroll
                                for (int u = 0; u < U; ++u)
#pragma unroll
                                    for (int m = 0; m < R; ++m) {
                                        const int i = i0 + u * kGemvThreads * 4;
                                        v[u][m] = make_float4(0.f, 0.f, 0.f, 0.f);
                                        if (i < n_in && m0 + m < M) v[u][m] = *reinterpret_cast<const float4*>(xf + (size_t)(m0 + m) * n_in + i);
                                    }
#pragma unroll
                                for (int u = 0; u < U; ++u)
#pragma unroll
                                    for (int m = 0; m < R; ++m) {
                                        ss[m] = fmaf(v[u][m].x, v[u][m].x, ss[m]);
                                        ss[m] = fmaf(v[u][m].y, v[u][m].y, ss[m]);
                                        ss[m] = fmaf(v[u][m].z, v[u][m].z, ss[m]);
                                        ss[m] = fmaf(v[u][m].w, v[u][m].w, ss[m]);
                                    }
                            }
#pragma unroll
                            for (int m = 0; m < R; ++m) {
                                if (m0 + m >= M) continue;
                                ss[m] = warp_sum(ss[m]);
                                if (lane == 0) red[warp * (kMaxRows * 4) + m0 + m] = ss[m];
                            }
                        }
                        __syncthreads();
                    }
#pragma unroll
                    for (int m0 = 0; m0 < M; m0 += R) {
                        float inv_m[R];
#pragma unroll
                        for (int m = 0; m < R; ++m) {
                            float s = 0.f;
#pragma unroll
                            for (int w = 0; w < kGemvWarps; ++w) s += red[w * (kMaxRows * 4) + min(m0 + m, M - 1)];
                            inv_m[m] = 1.0f / sqrtf(s / (float)n_in + p.eps);
                        }
                        auto put = [&](int i, const float4* row_v) {  // inputs i .. i + 3 of these rows
                            uint2 gv = make_uint2(0u, 0u);
                            if (i < k1) gv = *reinterpret_cast<const uint2*>(p.gain + i);
                            const float g0 = bf_lo(gv.x), g1 = bf_hi(gv.x), g2 = bf_lo(gv.y), g3 = bf_hi(gv.y);
#pragma unroll
                            for (int m = 0; m < R; ++m) {
                                if (m0 + m >= M) continue;
                                const __nv_bfloat162 lo = __floats2bfloat162_rn(row_v[m].x * inv_m[m] * g0, row_v[m].y * inv_m[m] * g1);
                                const __nv_bfloat162 hi = __floats2bfloat162_rn(row_v[m].z * inv_m[m] * g2, row_v[m].w * inv_m[m] * g3);
                                uint2 o;
                                o.x = *reinterpret_cast<const uint32_t*>(&lo);
                                o.y = *reinterpret_cast<const uint32_t*>(&hi);
                                *reinterpret_cast<uint2*>(xs + (size_t)(m0 + m) * ld + (i - k0)) = o;
                            }
                        };
                        if (in_regs) {
#pragma unroll
                            for (int u = 0; u < U; ++u) {
                                const int i = tid * 4 + u * kGemvThreads * 4;
                                if (i < k_pad) put(i, v[u]);
                            }
                        } else {
                            for (int i = k0 + tid * 4; i < k0 + k_pad; i += kGemvThreads * 4) {
                                float4 r[R];
#pragma unroll
                                for (int m = 0; m < R; ++m) {
                                    r[m] = make_float4(0.f, 0.f, 0.f, 0.f);
                                    if (i < k1 && m0 + m < M) r[m] = *reinterpret_cast<const float4*>(xf + (size_t)(m0 + m) * n_in + i);
                                }
                                put(i, r);
                            }
                        }
                    }
                } else {
                    const __nv_bfloat16* xb = reinterpret_cast<const __nv_bfloat16*>(p.x);
                    for (int i = k0 + tid * 8; i < k0 + k_pad; i += kGemvThreads * 8) {
                        uint4 v[M];
#pragma unroll
                        for (int m = 0; m < M; ++m) {
                            v[m] = make_uint4(0u, 0u, 0u, 0u);
                            if (i < k1) v[m] = *reinterpret_cast<const uint4*>(xb + (size_t)m * n_in + i);
                        }
#pragma unroll
                        for (int m = 0; m < M; ++m) *reinterpret_cast<uint4*>(xs + (size_t)m * ld + (i - k0)) = v[m];
                    }
                }
            }
#pragma unroll
            for (int d = kEarly; d < kGemvDepth; ++d) fetch(buf[d], at_sub[d], at_k[d]);
            __syncthreads();

            // ---- stream
            const __nv_bfloat16* xrow[NB];
#pragma unroll
            for (int nb = 0; nb < NB; ++nb) xrow[nb] = xs + (size_t)min(nb * 8 + g, M - 1) * ld + q * 8 - seg0 * kGemvSeg;
            float acc[NB][4];
            int open_sub = -1, done = 0;  // the sub-item whose sums are in acc, and how many of its segments are in all its sums
            auto flush = [&]() {
                float2* slot = psum + (size_t)open_sub * 16 * M;
#pragma unroll
                for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int m = nb * 8 + 2 * q + (e & 1);
                        if (m < M) slot[(g + (e >> 1) * 8) * M + m].y = acc[nb][e];
                    }
            };
            while (at_sub[0] < n_sub) {
#pragma unroll
                for (int d = 0; d < kGemvDepth; ++d) {
                    if (at_sub[d] < n_sub) {
                        if (at_sub[d] != open_sub) {
                            if (open_sub >= 0) flush();
                            open_sub = at_sub[d];
                            float2* slot = psum + (size_t)open_sub * 16 * M;
                            done = seg0 / split;  // windows hold equal numbers of segments of every sub-item
#pragma unroll
                            for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                                for (int e = 0; e < 4; ++e) {  // later windows go on from the sums of the earlier ones
                                    const int m = nb * 8 + 2 * q + (e & 1);
                                    acc[nb][e] = 0.f;
                                    if (m < M && win > 0) acc[nb][e] = slot[(g + (e >> 1) * 8) * M + m].y;
                                    if (m < M && win == 0) slot[(g + (e >> 1) * 8) * M + m].x = 0.f;
                                }
                        }
                        float t[NB][kSteps][4];
#pragma unroll
                        for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                            for (int i = 0; i < kSteps; ++i) {
                                const uint4 xv = *reinterpret_cast<const uint4*>(xrow[nb] + at_k[d] + i * 32);
                                const uint4 &a = buf[d][2 * i], &b = buf[d][2 * i + 1];
                                float u[4];
                                mma_zero(t[nb][i], a.x, b.x, a.y, b.y, xv.x, xv.y);
                                mma_zero(u, a.z, b.z, a.w, b.w, xv.z, xv.w);
#pragma unroll
                                for (int e = 0; e < 4; ++e) t[nb][i][e] += u[e];
                            }
                        fetch(buf[d], at_sub[d], at_k[d]);
#pragma unroll
                        for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
#pragma unroll
                                for (int w = 1; w < kSteps; w *= 2)
#pragma unroll
                                    for (int i = 0; i < kSteps; i += 2 * w) t[nb][i][e] += t[nb][i + w][e];
                                acc[nb][e] += t[nb][0][e];
                            }
                        if ((++done & 7) == 0) {
                            float2* slot = psum + (size_t)open_sub * 16 * M;
#pragma unroll
                            for (int nb = 0; nb < NB; ++nb)
#pragma unroll
                                for (int e = 0; e < 4; ++e) {
                                    const int m = nb * 8 + 2 * q + (e & 1);
                                    if (m < M) slot[(g + (e >> 1) * 8) * M + m].x += acc[nb][e];
                                    acc[nb][e] = 0.f;
                                }
                        }
                    }
                }
            }
            if (open_sub >= 0) flush();
        }
        __syncthreads();

        // ---- epilogue: one (row or pair, activation row) per thread and turn
        auto total = [&](int r, int m) {  // sum of row r of this block, sub-items in order
            int o = r * groups / rows;  // the group of row r, or the one before it
            if ((o + 1) * rows / groups <= r) ++o;
            const float2* s = psum + ((size_t)o * split * 16 + (r - o * rows / groups)) * M + m;
            float v = 0.f;
            for (int j = 0; j < split; ++j) v += s[(size_t)j * 16 * M].x + s[(size_t)j * 16 * M].y;
            return v;
        };
        if (EPI == kEpiSwiglu) {
            for (int i = tid; i < rows / 2 * M; i += kGemvThreads) {
                const int m = i / (rows / 2), r = 2 * (i - m * (rows / 2));
                const float va = total(r, m), vb = total(r + 1, m);
                reinterpret_cast<__nv_bfloat16*>(p.out)[(size_t)m * (p.n_rows >> 1) + ((blk0 + r) >> 1)] =
                    __float2bfloat16_rn(va / (1.0f + expf(-va)) * vb);
            }
        } else {
            for (int i = tid; i < rows * M; i += kGemvThreads) {
                const int m = i / rows, r = i - m * rows;
                float* out = reinterpret_cast<float*>(p.out) + (size_t)m * p.n_rows + blk0 + r;
                if (EPI == kEpiPlain) {
                    *out = total(r, m);
                } else {
                    const float x0 = *out, y0 = x0 + total(r, m);
                    *out = y0;
                    xy[r * M + m] = make_float2(x0, y0);
                }
            }
            if (EPI == kEpiResidual) {
                __syncthreads();
                if (warp < M)
                    for (int r = lane; r < rows; r += 32) {
                        const float2 v = xy[r * M + warp];
                        s_loc[0] = fmaf(v.x, v.y, s_loc[0]);
                        s_loc[1] = fmaf(v.x, v.x, s_loc[1]);
                        s_loc[2] = fmaf(v.y, v.y, s_loc[2]);
                    }
            }
        }
    }

    if (EPI == kEpiResidual) {
        if (warp < M) {
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const float v = warp_sum(s_loc[j]);
                if (lane == 0) p.partials[((size_t)blockIdx.x * kMaxRows + warp) * 4 + j] = v;
            }
        }
        if (last_cta_arrives(p.counter, flag)) {
            // one warp per activation row: lanes add the per-CTA partials b = lane, lane+32, ... in order, then an
            // xor butterfly in double precision (fixed order, independent of the row count)
            if (warp < M) {
                double sxy = 0, sxx = 0, syy = 0;
                for (unsigned b = lane; b < gridDim.x; b += 32) {
                    sxy += (double)__ldcg(p.partials + ((size_t)b * kMaxRows + warp) * 4 + 0);
                    sxx += (double)__ldcg(p.partials + ((size_t)b * kMaxRows + warp) * 4 + 1);
                    syy += (double)__ldcg(p.partials + ((size_t)b * kMaxRows + warp) * 4 + 2);
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

}  // namespace asd
