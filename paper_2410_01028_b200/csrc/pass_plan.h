// How the persistent pass kernel divides a block's shared memory: plain C++, shared by the kernel and the host code that
// launches it.
#pragma once
#include <stddef.h>

#include <algorithm>

#include "../../include/asd.h"

#ifdef __CUDACC__
#define ASD_HOST_DEVICE __host__ __device__
#else
#define ASD_HOST_DEVICE
#endif

namespace asd {

constexpr int kPassMaxRows = 16;  // rows of one pass (prefill feeds the prompt 16 rows at a time)
constexpr int kSlotBytes = 8192;  // one ring slot: 16 weight rows x 256 bf16 inputs, or one 64-key K/V box
constexpr int kSegK = 256;        // inputs per ring item (8 column blocks of 32; the last item of a row may hold fewer)
constexpr int kXsPad = 32;        // bf16 elements of padding per activation row (64 bytes: conflict-free 16-byte reads)
constexpr int kAttnChunk = 128;   // keys per attention work item; chunks are aligned to absolute positions
constexpr int kBoxKeys = 64;      // keys per K/V box (one ring slot)
constexpr int kMaxSlots = 48;     // ring slots that barriers and generations are set aside for (a block holds 28)
constexpr int kXsBudget = 40960;  // most shared memory the attention scratch of all warp groups may take

// 256-input segments whose activations (M rows, bf16, padded rows) fit the shared-memory window
ASD_HOST_DEVICE inline int pass_wseg(int M, int xs_bytes) {
    const int w = (xs_bytes / M - kXsPad * 2) / (kSegK * 2);
    return w < 1 ? 1 : w;
}

// Shared memory of a group of attention warps: the queries of eight columns [column][head_dim] and their probabilities as three bf16 terms
// [term][column][128 keys], rows 16 bytes longer than they are (the eight rows of a matrix then lie in different banks), then the warps' maxima and sums.
constexpr int kAttnCols = 8;  // (row, head of the group) pairs per step: the N of m16n8k16
constexpr int kAttnPRow = kAttnChunk * 2 + 16;
ASD_HOST_DEVICE inline int attn_cols(int M, int group) { return M * group < kAttnCols ? M * group : kAttnCols; }
ASD_HOST_DEVICE inline int attn_scratch_bytes(int M, int group, int hd) {
    return attn_cols(M, group) * (2 * hd + 16 + 3 * kAttnPRow) + 2 * 4 * kAttnCols * 4;
}

// Shared-memory plan of a pass of M rows: ring slots, barriers, reduction scratch, per-pair partial sums, activation window /
// attention scratch.
struct PassPlan {
    int ns, attn_groups, off_bars, off_misc, off_psum, off_reg_a, xs_bytes;
    size_t smem;
};

inline bool plan_pass(int num_sms, size_t max_smem, const asd_config& c, int M, PassPlan* pl) {
    const int kvd = c.n_kv_heads * c.head_dim;
    const long long max_rows = std::max<long long>(std::max(c.vocab, 2 * c.d_ffn), std::max(c.d_model + 2 * kvd, c.d_model));
    const long long np_max = ((max_rows + 1) / 2 + num_sms - 1) / num_sms + 2;
    if ((max_rows + 1) / 2 * num_sms >= (1LL << 31)) return false;  // the kernel splits a matrix's pairs over the CTAs in 32-bit arithmetic
    // per-pair partial sums; when a CTA has fewer than 8 groups of 8 pairs up to 15 warps keep copies (at most 15 / groups
    // copies of at most 8 * groups pairs: 120 pairs in all)
    const size_t psum = ((size_t)std::max<long long>(np_max, 120) * 2 * M * 4 + 15) & ~(size_t)15;
    const size_t misc = ((size_t)16 * kPassMaxRows * 4 * 4 + 32 + kMaxSlots * 4 + 8 * 4 * 4 + kPassMaxRows * 4 + 8 * 16 * 2 + 15) & ~(size_t)15;  // reduction scratch, flags, slot generations, split table, tokens, warp sets
    const size_t attn_scratch = (size_t)attn_scratch_bytes(M, c.n_heads / c.n_kv_heads, c.head_dim);
    // Activation window: the longest reduction dimension (in segments of 256 inputs) cut into as few windows as leave
    // the ring 20 slots. Every further window costs a stage of a multi-row pass a block-wide refill, every slot less
    // costs bandwidth (one row, 7B shape: 24 slots 0.402 ms per 4 layers, 21: 0.409, 16: 0.422, 12: 0.481); 20 was the
    // best trade for three and four rows (measured again with 22 and 24 after the kernel had changed: four and five rows
    // 0.7 % slower). Windows do not get shorter than a row of d_model while that leaves 16 slots: the RMSNorm stages want
    // their rows whole (six to nine rows: 1-2.5 % faster than with W_d's row cut into equal parts). One row always fits whole.
    const size_t seg_max = ((size_t)std::max(c.d_model, c.d_ffn) + kSegK - 1) / kSegK;
    const size_t seg_norm = ((size_t)c.d_model + kSegK - 1) / kSegK;  // the RMSNorm stages want their rows whole in the window
    const long long fixed = 1024 + (long long)(psum + misc) + 2 * kMaxSlots * 8;
    size_t wseg_plan = seg_max;
    auto leaves_ring = [&](size_t wseg, long long slots) {
        const size_t bytes = (size_t)M * (wseg * kSegK + kXsPad) * 2;
        return (long long)max_smem - fixed - (long long)((bytes + 15) & ~(size_t)15) >= slots * kSlotBytes;
    };
    for (size_t nw = 1; nw <= seg_max; ++nw) {
        wseg_plan = (seg_max + nw - 1) / nw;
        if (leaves_ring(wseg_plan, 20)) break;
    }
    // not shorter than a row of d_model while the ring keeps 16 slots: the RMSNorm stages want their rows whole
    if (wseg_plan < seg_norm && leaves_ring(seg_norm, 16)) wseg_plan = seg_norm;
    const int xs_bytes = (int)((size_t)M * (wseg_plan * kSegK + kXsPad) * 2);
    const size_t xs = (size_t)M * ((size_t)pass_wseg(M, xs_bytes) * kSegK + kXsPad) * 2;
    // Up to three groups of four warps work on attention items: as many as their scratch fits its budget and as the ring feeds, a K and a V
    // tile for each. Scratch is set aside for the groups that work and no others: at head size 256, where the ring feeds one, three
    // would take the slots that 16 rows with a vocabulary above 141000 need.
    const int tile_slots = (kAttnChunk / kBoxKeys) * std::max(1, c.head_dim / 64);
    int groups = (int)std::max<size_t>(1, std::min<size_t>(3, (size_t)kXsBudget / attn_scratch)), ns = 0;
    size_t reg_a = 0;
    for (;; --groups) {
        reg_a = (std::max(xs, groups * attn_scratch) + 15) & ~(size_t)15;
        ns = (int)std::min<long long>(kMaxSlots, ((long long)max_smem - fixed - (long long)reg_a) / kSlotBytes);
        if (groups == 1 || ns >= groups * 2 * tile_slots) break;
    }
    if (ns < 2 * tile_slots || ns < 8) return false;
    pl->ns = ns;
    pl->xs_bytes = xs_bytes;
    pl->attn_groups = groups;
    pl->off_bars = ns * kSlotBytes;
    pl->off_misc = pl->off_bars + 2 * kMaxSlots * 8;
    pl->off_psum = pl->off_misc + (int)misc;
    pl->off_reg_a = pl->off_psum + (int)psum;
    pl->smem = (size_t)pl->off_reg_a + reg_a + 1024;
    return pl->smem <= max_smem;
}

}  // namespace asd
