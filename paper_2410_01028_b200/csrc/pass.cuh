// One persistent kernel per decoder pass (decode, draft, verify, row pass of a short prompt).
//
// Why: at batch 1 a pass is ~200 dependent sublayer stages of 5-30 us each. Launching them one by one leaves
// HBM idle at every boundary (launch latency, RMSNorm prologue, drain). Weights, however, never depend on
// activations. So here one CTA per SM stays resident for the whole pass (cooperative launch) and is split in
// two roles:
//   * a producer warp walks this CTA's share of EVERY stage's weights (and of the old part of the KV cache)
//     in order and keeps a shared-memory ring of 8 KB slots full with TMA copies (cp.async.bulk, and
//     cp.async.bulk.tensor with 128-byte swizzle for K/V boxes). It never waits for activations, so HBM keeps
//     streaming across stage boundaries, grid barriers and prologues. Weights are stored in HBM in exactly
//     the order the ring consumes them (see "packed weights" below), so a CTA's slab of a stage is one
//     contiguous byte range;
//   * 15 consumer warps wait for the previous stage of all CTAs (a grid barrier on a monotonically increasing
//     counter, bounded spin), stage the activations in shared memory (RMSNorm fused), multiply the ring slots
//     on the tensor cores, and run the epilogue: RoPE + KV append, SwiGLU, residual add + cosine
//     similarity (summand of C_l, Section 3.2), LM-head argmax + greedy acceptance (Section 1).
// Sublayers in the skip mask (the draft model D, Algorithm 1) simply do not appear in the stage table: no
// weights are streamed and no K/V is touched for them.
//
// Packed weights: a matrix [n_rows, n_in] is cut into PAIRS of rows (the two rotary partners of a q/k head,
// gate_i and up_i, or two neighbouring rows) and SEGMENTS of 256 inputs. CTA b owns pairs [b*P/G, (b+1)*P/G)
// and groups them into GROUPS of eight pairs (the last group may hold fewer). One ring item = one group x one
// segment of 256 inputs = up to 16 rows x 512 bytes = one 8 KB slot, stored as up to 8 column blocks of 32 inputs
// (rows x 64 bytes each; the last segment of a row simply has fewer blocks). The CTA's slab is
// segment-major (for seg: for group), so consecutive ring items belong to different consumer warps and are
// consumed as soon as they land, and no padding crosses HBM for input sizes that are multiples of 32.
//
// The products run on the tensor cores (mma.sync m16n8k16, bf16 in, fp32 accumulate): the 16 weight rows of an item
// are the A operand, the activation rows the 8 columns of the B operand (two B tiles for more than 8 rows), so one
// step serves any row count up to 8 and the arithmetic of a row does not depend on how many rows share the pass. tcgen05 is not used here on
// purpose: its smallest tile (64 weight rows) does not fit a 148-way row split that leaves ~28 rows of the
// d x d matrices to a CTA, and its A operand would need the activations padded to 64+ rows in shared memory.
//
// Reduction order is fixed and independent of the row count M: an item's 16 steps go round four
// accumulators that are added in pairs at the end, segments are added in ascending order. Attention chunks are aligned
// to absolute positions and merged in a fixed order. Row m of a (k+1)-row verify pass is therefore bit-identical to
// a 1-row decode pass at the same position, so speculative output equals autoregressive output bit for bit.
#pragma once
#include <limits.h>

#include <type_traits>

#include "common.cuh"
#include "pass_plan.h"
#include "ring.cuh"

namespace asd {

constexpr int kPassConsumerWarps = 15;
constexpr int kPassConsumers = kPassConsumerWarps * 32;
constexpr int kPassThreads = kPassConsumers + 32;  // + one producer warp
constexpr unsigned kProducerNapNs = 50;             // the producer warp's sleep after a round without a free slot
constexpr int kAttnDoneBar = 8;  // named barriers 8 to 10: a group of attention warps has read its value tile
constexpr int kFinishBar = 7;  // named barrier: a CTA's cosines are done (1: consumer warps, 2 to 4: groups of attention warps)
// Passes of one and two rows read the embeddings in the first sublayer and finish their cosines beside the LM head; in the code of more rows
// both cost more (registers) than the two hand-offs that they save: five rows of the tiny decoder 136 -> 139 us, 16 rows 5 %.
template <int M>
constexpr bool kFewRows = M <= 2;

enum StageType : int { kStEmbed = 0, kStQkv, kStAttn, kStOproj, kStGateUp, kStDown, kStLmHead, kStFinish };

struct StageDesc {
    int type, layer;
    int n_rows, n_in;
    const unsigned char* W;             // packed weights of this stage (items of up to 8 KB, see above)
    const __nv_bfloat16* gain;
    __nv_bfloat16 *k_cache, *v_cache;   // this layer's cache [max_seq, kv_dim]
    const CUtensorMap *tm_k, *tm_v;     // tensor maps over the same
    int resid_slot;                     // residual stages: which block of per-CTA partial sums they write
    int src_stage;                      // index of the stage that wrote the hidden state this stage reads (tagged handoff)
};

// where the cosine similarity of one residual stage goes (filled in by the finish stage of the pass)
struct ResidOut {
    float* cos_out;  // [kPassMaxRows] cosine of this sublayer, per row
    double* sumcos;  // running sum over prompt rows
};

struct PassParams {
    int pos0;
    const int* tokens;                // the rows' tokens in device memory, or null:
    int inline_tokens[kMaxRows];      // a single-step call's tokens come with the launch
    const __nv_bfloat16* embed;
    int d_model, vocab, kv_dim, head_dim, n_heads, n_kv_heads, d_ffn;
    int hd_shift;  // log2(head_dim) when head_dim is a power of two, else 0 (divisions instead of shifts)
    float eps, inv_d, attn_scale;  // inv_d: 1 / d_model
    const float *rope_cos, *rope_sin;
    float* x;
    __nv_bfloat16 *q, *a, *t;
    uint2 *xl, *al, *tl;  // tagged handoff (one-row passes): hidden state [d], attention output [d/2], SwiGLU output [f/2] as (value, tag) words
    uint2 *ql, *kl, *vl;  // tagged handoff: this pass's query [d], key and value [kv_dim], one bf16 per word
    uint2 *pl_acc, *pl_ml;  // tagged handoff: attention partial results per (head, chunk): [head_dim] sums and (maximum before the scale, sum of weights)
    uint32_t pass_tag;     // tag of stage 0 of this pass; stage s writes pass_tag + s
    int embed_direct;      // 1: the first sublayer reads the rows' embeddings itself (see pass_kernel)
    int use_ll;            // 1: launch the kernel variant that hands activations over through the tagged buffers (host: one row, d_model <= 5760)
    float *part_acc, *part_ml;
    int chunk_stride;
    float* partials;        // [n_resid + 1][gridDim.x][kPassMaxRows][4] per-CTA partial sums (last block: LM head)
    const ResidOut* resid;  // [n_resid] outputs of the residual stages of this pass, in stage order
    int n_resid;
    unsigned* fin_counter;
    unsigned* grid_bar;
    unsigned bar_base;
    unsigned* merge_bar;    // grid barrier in front of the merge of an attention stage (passes without tags), and its value before the pass
    unsigned merge_base;
    unsigned bar_extra_last;  // test hook: arrivals the finish stage's barrier waits for beyond the grid size (0 in normal use)
    long long wait_cycles;    // cycle budget of every bounded wait of the pass
    int* err;
    const StageDesc* stages;
    int n_stages, finish_stage;  // finish_stage: index of the finish stage; the LM head may follow it
    int* argmax_out;
    float* margin_out;  // [M] top-1 minus top-2 logit of every row (the confidence that ends a draft run early), or null
    int* accept_out;   // greedy verification: accepted drafts, then the tokens (null: none)
    int* host_out;     // pinned host memory for what the caller waits for (kHost... below), or null
    int host_stamp;    // names this pass there
    float* logits_out;
    float* logits_host;  // pinned host memory for the same logits [M][vocab], or null
    int acc_sim;
    const double* sim_base;  // the sums behind C_l [2][L], and their copy in pinned host memory
    double* sim_host;
    long long* trace;  // optional [n_stages][kTraceEntries][gridDim.x] device timestamps (ns) and cycle counts, or null
    // shared-memory plan (bytes from the 1024-aligned base)
    int ns;            // ring slots
    unsigned ns_magic; // 2^32 / ns + 1, for exact division of ring item numbers by ns
    int attn_groups;   // 1 to 3 groups of 4 warps work on attention items
    int off_bars, off_misc, off_psum, off_reg_a;
    int xs_bytes;      // bytes of the activation window (as few windows per stage as leave the ring 20 slots)
};

// Words of host_out: the accept block or the last row's token, the last row's margin, the error words, the pass's stamp
constexpr int kHostMargin = 12, kHostErr = 16, kHostStamp = 24;

__device__ __forceinline__ int pass_token(const PassParams& p, int m) { return p.tokens ? __ldcg(p.tokens + m) : p.inline_tokens[m]; }

constexpr int kTraceEntries = 12;  // per stage and CTA: 0-7 consumer side, 8-10 producer side (first / last copy issued, stall cycles), 11 descriptor read
constexpr int kGrpPairs = 8;   // pairs of weight rows per ring item: 16 rows, the M of one m16n8k16 tensor-core step
constexpr int kGrpRows = 2 * kGrpPairs;
constexpr int kSegBlocks = kSegK / 32;  // column blocks of 32 inputs per full segment
constexpr int kNarrowRow = 512;  // rows up to this length are normalised by a warp each (passes of several rows)

// D (16x8, fp32) += A (16x16, bf16, row) * B (16x8, bf16, col): one warp-wide tensor-core step
__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                               uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

struct PassSmem {
    unsigned char* ring;
    uint64_t *full, *empty;
    float* red;   // [16][kPassMaxRows*4]
    int* flag;    // [8]
    volatile unsigned* consumed;  // [kMaxSlots] generations of each ring slot that consumers have finished with
    const int* split;             // [8][4] per stage type: this CTA's first pair, pair count, groups of 16 rows, warp sets per group
    const unsigned short* warp_set;  // [8][16] per stage type and warp: warp set | first group << 8 (divisions that a stage would start with)
    const int* tok;               // [16] the rows' tokens, clamped to the vocabulary
    float* psum;
    unsigned char* reg_a;
};

__device__ __forceinline__ void stage_pair_rows(int type, const PassParams& p, int pair, int& ra, int& rb) {
    if (type == kStQkv) {
        const int half = p.head_dim >> 1;
        const int nq = p.d_model >> 1, nk = p.kv_dim >> 1;
        int base, pp;
        if (pair < nq) {
            base = 0;
            pp = pair;
        } else if (pair < nq + nk) {
            base = p.d_model;
            pp = pair - nq;
        } else {
            base = p.d_model + p.kv_dim;
            pp = pair - nq - nk;
        }
        const int head = p.hd_shift ? (pp >> (p.hd_shift - 1)) : pp / half, j = pp - head * half;
        ra = base + head * p.head_dim + j;
        rb = ra + half;
    } else {
        ra = 2 * pair;
        rb = 2 * pair + 1;
    }
}

// CTA b owns pairs [pair0, pair0 + np) of a matrix. W_gu is split at even pair indices (align = 2): two neighbouring
// SwiGLU outputs share one tagged word of the handoff buffer and must come from the same CTA.
__device__ __forceinline__ void cta_pairs(int n_rows, int type, int& pair0, int& np) {
    const int n_pairs = (n_rows + 1) >> 1;
    const int align = (type == kStGateUp) ? 2 : 1;
    const unsigned units = (unsigned)(n_pairs / align);  // units * gridDim.x < 2^32 (the host refuses larger matrices): 32-bit divisions
    pair0 = (int)(blockIdx.x * units / gridDim.x) * align;
    const int pair1 = (blockIdx.x + 1 == gridDim.x) ? n_pairs : (int)((blockIdx.x + 1) * units / gridDim.x) * align;
    np = pair1 - pair0;
}

// Attention work items (kv head, 128-key chunk), head-major; CTA b takes the contiguous range
// [b*T/G, (b+1)*T/G): mostly chunks of one head, so queries and DRAM pages are reused.
__device__ __forceinline__ int attn_local_items(const PassParams& p, int M, int& n_chunks, int& first) {
    n_chunks = (p.pos0 + M - 1) / kAttnChunk + 1;
    const unsigned total = (unsigned)(p.n_kv_heads * n_chunks);  // heads * chunks * CTAs stays far below 2^32
    first = (int)(blockIdx.x * total / gridDim.x);
    return (int)((blockIdx.x + 1) * total / gridDim.x) - first;
}

// ============================================================================================ ring protocol
// mbarrier waits are by phase PARITY, which is only unambiguous when the waiter is at most one phase away from
// the barrier. Consumer warps and producer lanes skip through the ring (each takes every n-th item), so a
// waiter can reach generation g of a slot while generation g-1 has not even landed. Every wait therefore
// first checks a plain per-slot counter of consumed generations (monotonic, no aliasing) and only then the
// barrier, which by then is at most one phase away.
__device__ __forceinline__ void ring_locate(const PassParams& p, uint32_t g, int& slot, uint32_t& gen) {
    gen = fast_div(g, p.ns_magic);
    slot = (int)(g - gen * (uint32_t)p.ns);
}

__device__ __forceinline__ bool ring_spin_consumed(const PassParams& p, const PassSmem& sm, int slot, uint32_t gen, int code,
                                                   int stage, uint32_t g, int tag) {
    if (sm.consumed[slot] >= gen) return true;
    volatile int* err = p.err;
    const long long t0 = clock64();
    for (unsigned spin = 1;; ++spin) {
        if (sm.consumed[slot] >= gen) return true;
        if ((spin & 255u) != 0) continue;
        if (*err != kErrNone) return false;
        if (clock64() - t0 > p.wait_cycles) {
            if (atomicCAS(p.err, kErrNone, code) == kErrNone) {
                p.err[1] = stage, p.err[2] = (int)g, p.err[3] = slot, p.err[4] = blockIdx.x, p.err[5] = threadIdx.x;
                p.err[6] = tag, p.err[7] = -1;
            }
            return false;
        }
    }
}

// consumer: wait until ring item g has landed in its slot
__device__ __forceinline__ void ring_wait_full(const PassParams& p, const PassSmem& sm, uint32_t g, int slot, uint32_t gen, int stage, int tag) {
    if (gen > 0 && !ring_spin_consumed(p, sm, slot, gen, kErrFullWait, stage, g, tag)) return;
    mbar_wait(&sm.full[slot], gen & 1, p.err, kErrFullWait, stage, g, slot, tag, p.wait_cycles);
}
// consumer: one thread, after all readers of the slot are done (warp or group barrier before the call, which with the arrival's
// release orders their loads before the slot is handed back)
__device__ __forceinline__ void ring_release(const PassSmem& sm, int slot, uint32_t gen) {
    sm.consumed[slot] = gen + 1;
    mbar_arrive(&sm.empty[slot]);
}
__device__ __forceinline__ long long global_ns() {
    long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}
// producer side of the timeline (lane 0 of the producer warp): when it issued its first and last copy of the stage
// and how many cycles it waited for free slots in between
__device__ __forceinline__ void producer_trace(const PassParams& p, int stage, long long t_first, long long stall_cycles) {
    if (!p.trace || (threadIdx.x & 31) != 0) return;
    long long* t = p.trace + (size_t)stage * kTraceEntries * gridDim.x + blockIdx.x;
    t[(size_t)8 * gridDim.x] = t_first;
    t[(size_t)9 * gridDim.x] = global_ns();
    t[(size_t)10 * gridDim.x] = stall_cycles;
}

// ============================================================================================ producer
// The whole producer warp feeds the ring: lane l takes ring items l, l+32, ... of each stage. The lanes poll in ONE
// converged loop (each lane looks at the slot of its own next item, the lanes whose slot is free issue their copy
// and move on), so the warp costs its scheduler a dozen instructions per round however many lanes are waiting, and
// a freed slot is refilled within one round. (Asking L2 for the items beyond the ring with
// cp.async.bulk.prefetch.L2 while the ring is full was measured twice and slows the pass down, by 17 % at 32 items
// ahead and more at larger distances; the ring alone is the prefetch buffer.)
struct ProdState {
    int s, type, idx, n_items;
    uint32_t gi;  // ring index of item 0 of the stage
    // GEMV stage: this CTA's slab is contiguous and already in ring order (segment-major, octets inside)
    const unsigned char* slab;
    int np, n_oct, row_blocks;
    // attention stage
    const CUtensorMap *tm_k, *tm_v;
    int n_chunks, first;
};

// move to the next stage that streams anything for this lane; false when the pass has no more
template <int M>
__device__ __forceinline__ bool prod_next_stage(const PassParams& p, const PassSmem& sm, ProdState& c, int lane) {
    for (;;) {
        c.gi += (uint32_t)c.n_items;
        c.n_items = 0;
        if (++c.s >= p.n_stages) return false;
        const StageDesc st = p.stages[c.s];
        c.type = st.type;
        if (st.type == kStEmbed || st.type == kStFinish) continue;
        if (st.type == kStAttn) {
            const int n_local = attn_local_items(p, M, c.n_chunks, c.first);
            const int nhb = p.head_dim > 64 ? p.head_dim / 64 : 1;
            c.n_items = n_local * 2 * (kAttnChunk / kBoxKeys) * nhb;
            c.tm_k = st.tm_k, c.tm_v = st.tm_v;
        } else {
            const int pair0 = sm.split[st.type * 4 + 0];
            c.np = sm.split[st.type * 4 + 1];
            c.n_oct = sm.split[st.type * 4 + 2];
            c.n_items = c.n_oct * ((st.n_in + kSegK - 1) / kSegK);
            c.row_blocks = (st.n_in + 31) >> 5;  // 32-input column blocks per row
            c.slab = st.W + (size_t)pair0 * c.row_blocks * 128;
        }
        c.idx = lane;
        if (c.idx < c.n_items) return true;
    }
}

// Where item c.idx of the lane's current stage lives: a K/V box (tensor map + coordinates) or a run of weight bytes.
struct ItemSrc {
    const CUtensorMap* map;  // non-null: K/V box at (x, y)
    int x, y;
    const unsigned char* ptr;
    uint32_t bytes;
};
__device__ __forceinline__ ItemSrc item_source(const PassParams& p, const ProdState& c) {
    ItemSrc s;
    if (c.type == kStAttn) {
        const int nhb = p.head_dim > 64 ? p.head_dim / 64 : 1;
        const int box_cols = p.head_dim > 64 ? 64 : p.head_dim;
        const int tile_slots = (kAttnChunk / kBoxKeys) * nhb;
        const int j = c.idx / (2 * tile_slots), r = c.idx - j * 2 * tile_slots;
        const int which = r / tile_slots, t = r - which * tile_slots;
        const int rg = t / nhb, hb = t - rg * nhb;
        const int item = c.first + j;
        const int kvh = item / c.n_chunks, chunk = item - kvh * c.n_chunks;
        s.map = which ? c.tm_v : c.tm_k;
        s.x = kvh * p.head_dim + hb * 64;
        s.y = chunk * kAttnChunk + rg * kBoxKeys;
        s.ptr = nullptr;
        s.bytes = (uint32_t)kBoxKeys * box_cols * 2u;
    } else {
        const int seg = c.idx / c.n_oct, o = c.idx - seg * c.n_oct;
        const int nblk = min(kSegBlocks, c.row_blocks - seg * kSegBlocks);  // column blocks of this segment
        const int rows = 2 * min(kGrpPairs, c.np - kGrpPairs * o);
        s.map = nullptr;
        s.x = s.y = 0;
        s.ptr = c.slab + (size_t)seg * c.np * (kSegK * 4) + (size_t)o * nblk * (kGrpRows * 64);
        s.bytes = (uint32_t)(nblk * rows * 64);
    }
    return s;
}

template <int M>
__device__ void pass_producer(const PassParams& p, const PassSmem& sm) {
    const int lane = threadIdx.x & 31;
    volatile int* err = p.err;
    uint32_t issued[2] = {0, 0};
    int n_issued = 0;
    const uint64_t pol_stream = make_policy_evict_first();  // weights are read once per pass: do not let them age in L2
    ProdState c{};
    c.s = -1;
    bool active = prod_next_stage<M>(p, sm, c, lane);
    long long t_progress = clock64();
    long long tp_first = (p.trace && lane == 0) ? global_ns() : 0, stall = 0, t_blocked = 0;
    bool blocked = false;
    for (unsigned round = 1; __any_sync(0xffffffffu, active); ++round) {
        bool copied = false;
        if (active) {
            const uint32_t g = c.gi + (uint32_t)c.idx;
            int slot;
            uint32_t gen;
            ring_locate(p, g, slot, gen);
            // the slot may be overwritten once generation gen-1 of it has been consumed (counter first: the barrier's
            // phase parity alone is ambiguous for a waiter that is more than one phase behind)
            const bool free_now = gen == 0 || (sm.consumed[slot] >= gen && mbar_try_wait(&sm.empty[slot], (gen - 1) & 1));
            if (free_now) {
                if (p.trace && lane == 0 && blocked) stall += clock64() - t_blocked;
                blocked = false;
                unsigned char* dst = sm.ring + (size_t)slot * kSlotBytes;
                const ItemSrc src = item_source(p, c);
                mbar_expect_tx(&sm.full[slot], src.bytes);
                if (src.map) tma_load_2d(dst, src.map, src.x, src.y, &sm.full[slot]);
                else tma_load_1d_hint(dst, src.ptr, src.bytes, &sm.full[slot], pol_stream);
                issued[1] = issued[0], issued[0] = g, ++n_issued;
                copied = true;
                t_progress = clock64();
                c.idx += 32;
                if (c.idx >= c.n_items) {
                    if (p.trace && lane == 0) {
                        producer_trace(p, c.s, tp_first, stall);
                        stall = 0;
                    }
                    active = prod_next_stage<M>(p, sm, c, lane);
                    if (p.trace && lane == 0) tp_first = global_ns();
                }
            } else {
                if (p.trace && lane == 0 && !blocked) t_blocked = clock64();
                blocked = true;
                if ((round & 255u) == 0) {  // the error word lives in global memory: look at it only now and then
                    if (*err != kErrNone) {
                        active = false;
                    } else if (clock64() - t_progress > p.wait_cycles) {
                        if (atomicCAS(p.err, kErrNone, kErrEmptyWait) == kErrNone) {
                            p.err[1] = c.s, p.err[2] = (int)g, p.err[3] = slot, p.err[4] = blockIdx.x, p.err[5] = threadIdx.x;
                            p.err[6] = M, p.err[7] = (int)((gen - 1) & 1);
                        }
                        active = false;
                    }
                }
            }
        }
        // A round in which no lane found a free slot: sleep a moment instead of polling again at once. The warp shares
        // its scheduler with three consumer warps, and a refill that starts some tens of nanoseconds later costs
        // nothing against a memory latency of microseconds.
        if (!__any_sync(0xffffffffu, copied)) __nanosleep(kProducerNapNs);
        __syncwarp();
    }
    // If the pass was abandoned, copies may still be in flight into this CTA's shared memory: let this lane's
    // last two copies land (bounded) before the CTA exits (the ring holds at most two items of a lane).
    if (*err != kErrNone) {
        for (int k = 0; k < 2 && k < n_issued; ++k) {
            int slot;
            uint32_t gen;
            ring_locate(p, issued[k], slot, gen);
            const long long t0 = clock64();
            while (!mbar_try_wait(&sm.full[slot], gen & 1) && clock64() - t0 < 20000000LL) {
            }
        }
    }
}

// per-stage timeline of every CTA (debugging aid): 0 = stage entered, 1 = inputs ready, 2 = streaming done, 3 = stage left
__device__ __forceinline__ void trace_mark(const PassParams& p, int stage, int k) {
    if (p.trace && threadIdx.x == 0) p.trace[((size_t)stage * kTraceEntries + k) * gridDim.x + blockIdx.x] = global_ns();
}

// ============================================================================================ grid barrier
__device__ __forceinline__ void consumers_sync() { bar_sync(1, kPassConsumers); }

// n: the stages that this arrival ends
__device__ __forceinline__ void grid_arrive(unsigned* counter, unsigned n = 1u) {
    consumers_sync();
    // one release at GPU scope: cumulative over the writes of the whole CTA, which the barrier above ordered before it
    if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(counter), "r"(n) : "memory");
}
__device__ __forceinline__ void grid_poll(const PassParams& p, const unsigned* counter, unsigned target) {  // one thread
    volatile int* err = p.err;
    const long long t0 = clock64();
    // every poll is a round trip to L2; the error word and the clock are looked at only now and then
    for (unsigned spin = 1; (int)(ld_acquire_gpu(counter) - target) < 0; ++spin) {
        if ((spin & 63u) != 0) continue;
        if (*err != kErrNone) break;
        if (clock64() - t0 > p.wait_cycles) {
            if (atomicCAS(p.err, kErrNone, kErrGridWait) == kErrNone) {
                p.err[1] = counter == p.grid_bar ? (int)((target - p.bar_base) / gridDim.x) : -1, p.err[2] = (int)ld_acquire_gpu(counter);
                p.err[3] = (int)target, p.err[4] = blockIdx.x;
            }
            break;
        }
    }
}
__device__ __forceinline__ void grid_wait(const PassParams& p, const unsigned* counter, unsigned target) {
    if (threadIdx.x == 0) grid_poll(p, counter, target);
    consumers_sync();
}

// consumers only: true in every thread of the last CTA to arrive on a global counter
__device__ __forceinline__ bool last_cta_consumers(unsigned* counter, int* flag_smem) {
    consumers_sync();
    if (threadIdx.x == 0) {
        unsigned t;  // cumulative over the CTA's writes, like the grid barrier's arrival
        asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(t) : "l"(counter) : "memory");
        *flag_smem = (t == gridDim.x - 1) ? 1 : 0;
    }
    consumers_sync();
    return *flag_smem != 0;
}

// A stage of a pass without tags starts by waiting for the previous stage of all CTAs, but for the first RMSNorm where it reads the
// embeddings itself and the LM head, in front of which the finish stage has waited. Whatever does not depend on activations (the
// stage descriptor, index arithmetic, RMSNorm gains) is done before this wait. extra: arrivals beyond the grid's (test hook).
__device__ __forceinline__ void stage_begin(const PassParams& p, int s, unsigned extra = 0u) {
    if (s > 0) grid_wait(p, p.grid_bar, p.bar_base + (unsigned)s * gridDim.x + extra);
    trace_mark(p, s, 1);
}

// LM head: (largest logit, its lowest index, second-largest logit) of two disjoint index sets combined
__device__ __forceinline__ void top2_merge(float& v, int& i, float& s, float ov, int oi, float os) {
    s = fmaxf(fminf(v, ov), fmaxf(s, os));
    if (ov > v || (ov == v && oi < i)) {
        v = ov;
        i = oi;
    }
}

// ============================================================================================ tagged handoff
// One-row passes (decode, draft) spend a third of their time between weight streams,
// and most of that in round trips to L2: a stage's last output is stored, a fence and an atomic arrive at the grid
// barrier, every CTA polls the barrier word, and only then loads the activations. Here the activations carry their
// own "ready" mark instead: every 4-byte value (one fp32 of the hidden state, or two bf16 of the attention / SwiGLU
// output) is stored together with a 4-byte tag as ONE 8-byte word (8-byte scalar stores are single-copy atomic), the
// tag naming the pass and the stage that wrote it. A consumer simply loads the words it needs and repeats the load
// until every tag is the one it expects: one round trip after the slowest producer's store, no fence, no barrier.
// A buffer is only overwritten by a stage that itself needed ALL outputs of a later stage than every reader's, so no
// reader can still be waiting for the old contents (same ordering a barrier would give, carried by the data).
// The attention stage takes part: W_qkv's epilogue leaves q and this pass's k and v as tagged words (one bf16 each), a
// (head, chunk) item leaves its partial result as tagged words, and the warps without items merge the heads, chunk by chunk as
// the words arrive. q, k, v and the partial results of a layer are overwritten by the next
// layer's stages, which a CTA only reaches through W_o's stage, i.e. after every head's merged output (and with it
// every read of q, k, v and of the partial results) exists.
__device__ __forceinline__ void ll_store(uint2* dst, uint32_t data, uint32_t tag) {
    const unsigned long long v = ((unsigned long long)tag << 32) | (unsigned long long)data;
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(dst), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long ll_load1(const uint2* src) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(src) : "memory");
    return v;
}
__device__ __forceinline__ void ll_load2(const uint2* src, unsigned long long& a, unsigned long long& b) {  // 16-byte aligned
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(src) : "memory");
}
__device__ __forceinline__ bool ll_ready(unsigned long long v, uint32_t tag) { return (uint32_t)(v >> 32) == tag; }
// after a load that found a stale tag: go on waiting? (bounded like every other wait of the kernel)
__device__ __forceinline__ bool ll_keep_waiting(const PassParams& p, unsigned& spins, long long& t0, int stage) {
    if (spins == 0) t0 = clock64();
    if ((++spins & 31u) != 0) return true;
    volatile int* err = p.err;
    if (*err != kErrNone) return false;
    if (clock64() - t0 > p.wait_cycles) {
        if (atomicCAS(p.err, kErrNone, kErrGridWait) == kErrNone) {
            p.err[1] = stage, p.err[2] = -1, p.err[3] = -1, p.err[4] = blockIdx.x, p.err[5] = threadIdx.x, p.err[6] = 77, p.err[7] = 0;
        }
        return false;
    }
    return true;
}

// ============================================================================================ GEMV stage
// RMSNorm of M whole rows into the activation window (two or more rows; rows of at most 12 x 480 elements), for most
// row counts a function of its own so that its registers are its own: the rows are taken in batches of up to six, all loads of a
// batch in flight together, and what was loaded for the statistics is normalised from registers, so a batch costs one
// memory round trip. The arithmetic of a row is the one of the other paths: thread t adds the squares of its chunks
// t, t + 480, t + 960 element by element, lanes by butterfly, warps in index order.
// Four elements of a row of the hidden state: from x, or (emb given) from the embedding of the row's token.
__device__ __forceinline__ float4 load_row4(const float* xf, const __nv_bfloat16* emb, const int* tok, int m, int n_in, int i) {
    if (!emb) return __ldcg(reinterpret_cast<const float4*>(xf + (size_t)m * n_in + i));
    const uint2 e = *reinterpret_cast<const uint2*>(emb + (size_t)tok[m] * n_in + i);
    return make_float4(bf_lo(e.x), bf_hi(e.x), bf_lo(e.y), bf_hi(e.y));
}
template <int M>
__device__ __forceinline__ float4 load_row4_of(const float* xf, const __nv_bfloat16* emb, const int* tok, int m, int n_in, int i) {
    return load_row4(xf, kFewRows<M> ? emb : nullptr, tok, m, n_in, i);
}
template <int M>
__device__ __forceinline__ void norm_rows_body(const float* xf, const __nv_bfloat16* emb, const int* tok, const __nv_bfloat16* gain, int n_in, int wlen,
                                               int xstride, float inv_d, float eps, __nv_bfloat16* xs, float* red) {
    constexpr int kBatches = (M + 5) / 6, kRB = (M + kBatches - 1) / kBatches;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint2 gv[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int i = (tid + c * kPassConsumers) * 4;
        gv[c] = make_uint2(0u, 0u);
        if (i < n_in) gv[c] = *reinterpret_cast<const uint2*>(gain + i);
    }
#pragma unroll
    for (int m0 = 0; m0 < M; m0 += kRB) {
        float4 v[kRB][3];
#pragma unroll
        for (int u = 0; u < kRB; ++u)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int i = (tid + c * kPassConsumers) * 4;
                v[u][c] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (m0 + u < M && i < n_in) v[u][c] = load_row4_of<M>(xf, emb, tok, m0 + u, n_in, i);
            }
#pragma unroll
        for (int u = 0; u < kRB; ++u)
            if (m0 + u < M) {
                float s = 0.f;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const int i = (tid + c * kPassConsumers) * 4;
                    if (i < n_in) {
                        s = fmaf(v[u][c].x, v[u][c].x, s);
                        s = fmaf(v[u][c].y, v[u][c].y, s);
                        s = fmaf(v[u][c].z, v[u][c].z, s);
                        s = fmaf(v[u][c].w, v[u][c].w, s);
                    }
                }
                s = warp_sum(s);
                if (lane == 0) red[warp * (kPassMaxRows * 4) + m0 + u] = s;
            }
        bar_sync(1, kPassConsumers);
#pragma unroll
        for (int u = 0; u < kRB; ++u)
            if (m0 + u < M) {
                const int m = m0 + u;
                float s = 0.f;
#pragma unroll
                for (int w = 0; w < kPassConsumerWarps; ++w) s += red[w * (kPassMaxRows * 4) + m];
                const float inv = __frsqrt_rn(fmaf(s, inv_d, eps));
                const unsigned long long inv2 = pack2(inv, inv);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const int i = (tid + c * kPassConsumers) * 4;
                    if (i < wlen) {  // (past n_in everything is zero)
                        float a0, a1, a2, a3;
                        unpack2(fmul2(fmul2(pack2(v[u][c].x, v[u][c].y), inv2), bf2_to_f2(gv[c].x)), a0, a1);
                        unpack2(fmul2(fmul2(pack2(v[u][c].z, v[u][c].w), inv2), bf2_to_f2(gv[c].y)), a2, a3);
                        const __nv_bfloat162 lo = __floats2bfloat162_rn(a0, a1), hi = __floats2bfloat162_rn(a2, a3);
                        *reinterpret_cast<uint2*>(xs + (size_t)m * xstride + i) =
                            make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
                    }
                }
            }
    }
    for (int i = kPassConsumers * 12 + tid * 4; i < wlen; i += kPassConsumers * 4)  // zero padding past 5760
        for (int m = 0; m < M; ++m) *reinterpret_cast<uint2*>(xs + (size_t)m * xstride + i) = make_uint2(0u, 0u);
}

// The same for rows of at most 512 elements, which a warp holds in four loads: a row per warp, all rows side by side, and no block-wide
// barrier in between: a stage's RMSNorm of five rows of 256 elements 2.8 -> 1.0 us, a pass of five rows of the tiny decoder 151 -> 134 us. The
// longest row is what four loads of a lane hold; the function above spreads longer ones over the block. The sums are those of that function: lane l of group g has the element group of thread 32 g + l, the groups'
// butterflies are added in ascending order.
template <int M>
__device__ __forceinline__ void norm_rows_narrow(const float* xf, const __nv_bfloat16* emb, const int* tok, const __nv_bfloat16* gain, int n_in, int wlen,
                                                 int xstride, float inv_d, float eps, __nv_bfloat16* xs) {
    constexpr int kGroups = kNarrowRow / 128;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint2 gv[kGroups];
#pragma unroll
    for (int g = 0; g < kGroups; ++g) {
        const int i = (g * 32 + lane) * 4;
        gv[g] = make_uint2(0u, 0u);
        if (i < n_in) gv[g] = *reinterpret_cast<const uint2*>(gain + i);
    }
#pragma unroll 1
    for (int m = warp; m < M; m += kPassConsumerWarps) {
        float4 v[kGroups];
#pragma unroll
        for (int g = 0; g < kGroups; ++g) {
            const int i = (g * 32 + lane) * 4;
            v[g] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (i < n_in) v[g] = load_row4_of<M>(xf, emb, tok, m, n_in, i);
        }
        float s = 0.f;
#pragma unroll
        for (int g = 0; g < kGroups; ++g) {
            float q = 0.f;
            q = fmaf(v[g].x, v[g].x, q);
            q = fmaf(v[g].y, v[g].y, q);
            q = fmaf(v[g].z, v[g].z, q);
            q = fmaf(v[g].w, v[g].w, q);
            s += warp_sum(q);
        }
        const float inv = __frsqrt_rn(fmaf(s, inv_d, eps));
#pragma unroll
        for (int g = 0; g < kGroups; ++g) {
            const int i = (g * 32 + lane) * 4;
            if (i < wlen) {
                const __nv_bfloat162 lo = __floats2bfloat162_rn(v[g].x * inv * bf_lo(gv[g].x), v[g].y * inv * bf_hi(gv[g].x));
                const __nv_bfloat162 hi = __floats2bfloat162_rn(v[g].z * inv * bf_lo(gv[g].y), v[g].w * inv * bf_hi(gv[g].y));
                uint2 o;
                o.x = *reinterpret_cast<const uint32_t*>(&lo);
                o.y = *reinterpret_cast<const uint32_t*>(&hi);
                *reinterpret_cast<uint2*>(xs + (size_t)m * xstride + i) = o;
            }
        }
    }
}

// Called as a function by most row counts; with five and six rows the call itself (measured) costs more than the
// registers it frees.
template <int M>
__device__ __noinline__ void norm_rows_call(const float* xf, const __nv_bfloat16* emb, const int* tok, const __nv_bfloat16* gain, int n_in, int wlen,
                                            int xstride, float inv_d, float eps, __nv_bfloat16* xs, float* red) {
    norm_rows_body<M>(xf, emb, tok, gain, n_in, wlen, xstride, inv_d, eps, xs, red);
}
template <int M>
__device__ __forceinline__ void norm_rows_into_window(const float* xf, const __nv_bfloat16* emb, const int* tok, const __nv_bfloat16* gain, int n_in, int wlen,
                                                      int xstride, float inv_d, float eps, __nv_bfloat16* xs, float* red) {
    if (n_in <= kNarrowRow) norm_rows_narrow<M>(xf, emb, tok, gain, n_in, wlen, xstride, inv_d, eps, xs);
    else if constexpr (M == 5 || M == 6) norm_rows_body<M>(xf, emb, tok, gain, n_in, wlen, xstride, inv_d, eps, xs, red);
    else norm_rows_call<M>(xf, emb, tok, gain, n_in, wlen, xstride, inv_d, eps, xs, red);
}

// Epilogues of a GEMV stage with three or more activation rows, as functions of their own (their registers are their
// own; everything they need comes as scalar arguments, so nothing is re-read from the parameter block or the stage
// table). The (weight row or pair, activation row) items of the CTA are spread over all consumer threads instead of
// giving a thread all M rows of its pair. Every item is computed exactly as the one-row path computes it, and the
// sums that cross threads keep that path's shape (the cosine sums of activation row m: the lanes of a warp hold 32
// consecutive weight rows and are added by the same butterfly, the warps' sums are added in ascending order of the
// weight rows), so row m of an M-row pass stays bit-identical to a one-row pass. pre0 / pre1: what the first item of
// the thread (W_qkv: rotary factors) or of the warp (residual stages: old hidden state) needs from global memory,
// requested by the caller ahead of the weight stream.
__device__ __forceinline__ float psum_total(const float* psum, int idx, int S, int copy_stride) {
    float v = psum[idx];  // the copies of a partial sum (warp sets that shared a group) in the order 0, 1, ..., four loads in flight
#pragma unroll 1
    for (int k = 1; k < S; k += 4) {
        float c[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) c[i] = k + i < S ? psum[(k + i) * copy_stride + idx] : 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (k + i < S) v += c[i];
    }
    return v;
}

// residual add + cosine sums: item (m, j) = activation row m, weight rows 32 j .. 32 j + 31 of this CTA, one warp each
template <int M>
__device__ __noinline__ void epi_resid_rows(float* out, const float* psum, float* red, float* partials_dst, int n_rows, int pair0, int np,
                                            int S, float pre0) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int copy_stride = np * 2 * M;
    const int W = (np * 2 + 31) >> 5;
    for (int it = warp; it < M * W; it += kPassConsumerWarps) {
        const int m = it / W, j = it - m * W, e = j * 32 + lane, row = 2 * pair0 + e;
        float sxy = 0.f, sxx = 0.f, syy = 0.f;
        if (e < np * 2 && row < n_rows) {
            const float xv = (it == warp) ? pre0 : __ldcg(out + (size_t)m * n_rows + row);
            const float y = xv + psum_total(psum, e * M + m, S, copy_stride);
            out[(size_t)m * n_rows + row] = y;
            sxy = fmaf(xv, y, 0.f);
            sxx = fmaf(xv, xv, 0.f);
            syy = fmaf(y, y, 0.f);
        }
        sxy = warp_sum(sxy);
        sxx = warp_sum(sxx);
        syy = warp_sum(syy);
        if (lane == 0) red[it * 4 + 0] = sxy, red[it * 4 + 1] = sxx, red[it * 4 + 2] = syy;
    }
    bar_sync(1, kPassConsumers);
    if (tid < M * 3) {
        const int m = tid / 3, q = tid - m * 3;
        float tot = 0.f;
        for (int j = 0; j < W; ++j) tot += red[(m * W + j) * 4 + q];
        partials_dst[m * 4 + q] = tot;
    }
}

// W_qkv: rotary embedding of the q and k pairs, bf16 rounding, q to its buffer and k, v to the cache rows pos0 + m
template <int M>
__device__ __noinline__ void epi_qkv_rows(const float* psum, int pair0, int np, int S, int pos0, int d_model, int kv_dim, int head_dim,
                                          const float* rope_cos, const float* rope_sin, __nv_bfloat16* q, __nv_bfloat16* kc,
                                          __nv_bfloat16* vc, float pre0, float pre1) {
    const int tid = threadIdx.x;
    const int copy_stride = np * 2 * M;
    const int half = head_dim >> 1, nq = d_model >> 1, nk = kv_dim >> 1;
    for (int it = tid; it < np * M; it += kPassConsumers) {
        const int m = it / np, pl = it - m * np, pair = pair0 + pl;
        const int base = pair < nq ? 0 : (pair < nq + nk ? d_model : d_model + kv_dim);
        const int pp = pair < nq ? pair : (pair < nq + nk ? pair - nq : pair - nq - nk);
        const int head = pp / half, jr = pp - head * half;
        const int ra = base + head * head_dim + jr, rb = ra + half;
        float va = psum_total(psum, (pl * 2 + 0) * M + m, S, copy_stride), vb = psum_total(psum, (pl * 2 + 1) * M + m, S, copy_stride);
        const int pos = pos0 + m;
        if (ra < d_model + kv_dim) {  // q or k: rotate the pair (j, j + head_dim/2) by pos * theta_j
            const float c = (it == tid) ? pre0 : rope_cos[(size_t)pos * half + jr];
            const float sn = (it == tid) ? pre1 : rope_sin[(size_t)pos * half + jr];
            const float r0 = __fmaf_rn(va, c, -__fmul_rn(vb, sn));
            const float r1 = __fmaf_rn(vb, c, __fmul_rn(va, sn));
            va = r0;
            vb = r1;
        }
        const __nv_bfloat16 ha = __float2bfloat16_rn(va), hb = __float2bfloat16_rn(vb);
        if (ra < d_model) {
            q[(size_t)m * d_model + ra] = ha;
            q[(size_t)m * d_model + rb] = hb;
        } else if (ra < d_model + kv_dim) {
            kc[(size_t)pos * kv_dim + (ra - d_model)] = ha;
            kc[(size_t)pos * kv_dim + (rb - d_model)] = hb;
        } else {
            vc[(size_t)pos * kv_dim + (ra - d_model - kv_dim)] = ha;
            vc[(size_t)pos * kv_dim + (rb - d_model - kv_dim)] = hb;
        }
    }
}

// W_gu: SwiGLU of every (pair, row), bf16 rounding
template <int M>
__device__ __noinline__ void epi_gateup_rows(const float* psum, int pair0, int np, int S, __nv_bfloat16* t_out, int t_stride) {
    const int copy_stride = np * 2 * M;
    for (int it = threadIdx.x; it < np * M; it += kPassConsumers) {
        const int m = it / np, pl = it - m * np;
        const float va = psum_total(psum, (pl * 2 + 0) * M + m, S, copy_stride), vb = psum_total(psum, (pl * 2 + 1) * M + m, S, copy_stride);
        const float t = va / (1.0f + expf(-va)) * vb;
        t_out[(size_t)m * t_stride + (pair0 + pl)] = __float2bfloat16_rn(t);
    }
}

// LM head: the warps are dealt to the activation rows (warp w serves rows w mod G, w mod G + G, ...); a row's (largest
// logit, its lowest index, second-largest logit) does not depend on the order of the comparisons. lmp: this CTA's
// block of the per-CTA results.
template <int M>
__device__ __noinline__ void epi_lmhead_rows(const float* psum, float* red, int pair0, int np, int S, int n_rows, float* logits_out, float* lmp) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int copy_stride = np * 2 * M;
    constexpr int G = M < kPassConsumerWarps ? M : kPassConsumerWarps;
    const int g = warp % G, wi = warp / G, nw = (kPassConsumerWarps - g + G - 1) / G;
    for (int m = g; m < M; m += G) {
        float bv = -INFINITY, sv = -INFINITY;
        int bi = INT_MAX;
        for (int pl = wi * 32 + lane; pl < np; pl += nw * 32) {
            const int ra = 2 * (pair0 + pl), rb = ra + 1;
            const bool has_b = rb < n_rows;
            const float va = psum_total(psum, (pl * 2 + 0) * M + m, S, copy_stride), vb = psum_total(psum, (pl * 2 + 1) * M + m, S, copy_stride);
            if (logits_out) {
                logits_out[(size_t)m * n_rows + ra] = va;
                if (has_b) logits_out[(size_t)m * n_rows + rb] = vb;
            }
            if (va > bv) {  // rows come in ascending order: an equal logit keeps the lower index
                sv = bv, bv = va, bi = ra;
            } else {
                sv = fmaxf(sv, va);
            }
            if (has_b) {
                if (vb > bv) {
                    sv = bv, bv = vb, bi = rb;
                } else {
                    sv = fmaxf(sv, vb);
                }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            const float os = __shfl_xor_sync(0xffffffffu, sv, o);
            top2_merge(bv, bi, sv, ov, oi, os);
        }
        if (lane == 0) {
            red[warp * (kPassMaxRows * 4) + m * 4 + 0] = bv;
            red[warp * (kPassMaxRows * 4) + m * 4 + 1] = __int_as_float(bi);
            red[warp * (kPassMaxRows * 4) + m * 4 + 2] = sv;
        }
    }
    bar_sync(1, kPassConsumers);
    if (tid < M) {
        float v = -INFINITY, sc = -INFINITY;
        int i = INT_MAX;
        for (int w = tid % G; w < kPassConsumerWarps; w += G)
            top2_merge(v, i, sc, red[w * (kPassMaxRows * 4) + tid * 4 + 0], __float_as_int(red[w * (kPassMaxRows * 4) + tid * 4 + 1]),
                       red[w * (kPassMaxRows * 4) + tid * 4 + 2]);
        lmp[tid * 4 + 0] = v;
        lmp[tid * 4 + 1] = __int_as_float(i);
        lmp[tid * 4 + 2] = sc;
    }
}

template <int M, bool LL>
__device__ void gemv_stage(const PassParams& p, const StageDesc& st, const PassSmem& sm, uint32_t& gi, int stage) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int type = st.type;
    const bool norm = (type == kStQkv || type == kStGateUp || type == kStLmHead);
    const int n_in = st.n_in, n_rows = st.n_rows;
    // this CTA's share of the matrix (computed once per launch: the split costs three integer divisions)
    const int pair0 = sm.split[type * 4 + 0], np = sm.split[type * 4 + 1];
    const int n_seg = (n_in + kSegK - 1) / kSegK;
    const int n_oct = sm.split[type * 4 + 2];  // groups of 16 rows (8 pairs; the last group may hold fewer)
    const int wseg = pass_wseg(M, p.xs_bytes);
    const int xstride = wseg * kSegK + kXsPad;  // bf16 elements per activation row in the window
    __nv_bfloat16* xs = reinterpret_cast<__nv_bfloat16*>(sm.reg_a);
    float* red = sm.red;
    float* psum = sm.psum;

    const float* xf = p.x;
    const __nv_bfloat16* xb = (type == kStOproj) ? p.a : p.t;
    constexpr bool kLLCap = LL;
    constexpr bool ll = LL;                                       // activations come and go through the tagged buffers
    const uint32_t tag_x = p.pass_tag + (uint32_t)st.src_stage;   // tag of the hidden state this stage reads
    const uint32_t tag_in = p.pass_tag + (uint32_t)(stage - 1);   // tag of the attention / SwiGLU output (previous stage)
    const uint32_t tag_out = p.pass_tag + (uint32_t)stage;        // tag of what this stage writes
    const bool direct = kFewRows<M> && norm && p.embed_direct && st.src_stage == 0;  // the hidden state is still the rows' embeddings
    unsigned ll_spins = 0;
    long long ll_t0 = 0;
    // Fewer groups than warps (the d x d matrices leave ~28 rows to a CTA): several warps share a group, warp set ks
    // taking the segments congruent to ks modulo S and summing into its own copy of the partial sums; the copies are
    // added in the epilogue in the order ks = 0, 1, ... (a fixed order that depends on the matrix shape only).
    const int S = sm.split[type * 4 + 3];
    const int copy_stride = np * 2 * M;
    // A warp's first item of the stage stores its sums, later items add: the partial sums need no zeroing (there are no more warp sets than segments)
    constexpr bool kKeepX = (M == 1);
    constexpr int kOpBlocks = M > 8 ? 2 : 4;  // column blocks of an item whose operands are in registers at a time
    // tagged handoff: no barrier stands between the cosine sums of a stage and the next RMSNorm, whose sums therefore lie elsewhere
    constexpr int kRedNorm = LL ? 3 : 0;
    const int chunks = n_in > kPassConsumers * 8 ? 3 : n_in > kPassConsumers * 4 ? 2 : 1;  // of 4 elements of a thread; short rows skip the code of the others
    const bool keep = kKeepX && norm && (LL || n_in <= kPassConsumers * 12);
    uint2 gpre[3] = {make_uint2(0u, 0u), make_uint2(0u, 0u), make_uint2(0u, 0u)};  // this thread's RMSNorm gains
    const bool short_rows = norm && n_in <= kPassConsumers * 12;  // a thread owns at most three 4-element chunks of a row
    if (short_rows) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const int i = (tid + c * kPassConsumers) * 4;
            if (i < n_in) gpre[c] = *reinterpret_cast<const uint2*>(st.gain + i);
        }
    }
    // One or two rows: what the epilogue will need from global memory is requested ahead of the weight stream
    // (the rotary factors of this thread's pair before the barrier, the old hidden state of its row after it),
    // so the epilogue does not wait for a memory round trip.
    constexpr bool kSpreadEpi = (M >= 3);  // measured: spreading the epilogue's items over the threads pays from three rows on (two rows: no difference)
    constexpr bool kPre = (M <= 2);
    float pre[kPre ? 2 * M : 1];
    float pre0 = 0.f, pre1 = 0.f;  // spread epilogue: what the first item of this thread / warp needs (see the epi_*_rows functions)
    if (kSpreadEpi && type == kStQkv && tid < np * M) {
        const int m = tid / np;
        int ra, rb;
        stage_pair_rows(type, p, pair0 + (tid - m * np), ra, rb);
        if (ra < p.d_model + p.kv_dim) {
            const int half = p.head_dim >> 1, jr = p.hd_shift ? (ra & (p.head_dim - 1)) : ra % p.head_dim;
            pre0 = p.rope_cos[(size_t)(p.pos0 + m) * half + jr];
            pre1 = p.rope_sin[(size_t)(p.pos0 + m) * half + jr];
        }
    }
    if (kPre && type == kStQkv && tid < np) {
        int ra, rb;
        stage_pair_rows(type, p, pair0 + tid, ra, rb);
        if (ra < p.d_model + p.kv_dim) {
            const int half = p.head_dim >> 1, jr = p.hd_shift ? (ra & (p.head_dim - 1)) : ra % p.head_dim;
#pragma unroll
            for (int m = 0; m < (kPre ? M : 0); ++m) {
                pre[m] = p.rope_cos[(size_t)(p.pos0 + m) * half + jr];
                pre[M + m] = p.rope_sin[(size_t)(p.pos0 + m) * half + jr];
            }
        }
    }
    if (ll || direct || type == kStLmHead) trace_mark(p, stage, 1);  // no barrier: the loads below wait for exactly the words they need,
    else stage_begin(p, stage);  // the embeddings are there, and in front of the LM head the finish stage has waited
    if (kSpreadEpi && (type == kStOproj || type == kStDown)) {
        const int W = (np * 2 + 31) >> 5;
        if (warp < M * W) {
            const int m = warp / W, e = (warp - m * W) * 32 + lane;
            if (e < np * 2 && 2 * pair0 + e < n_rows) pre0 = __ldcg(p.x + (size_t)m * n_rows + 2 * pair0 + e);
        }
    }
    if (kPre && (type == kStOproj || type == kStDown) && tid < np * 2 && 2 * pair0 + tid < n_rows) {
        if (ll) {
            unsigned long long raw[kPre ? M : 1] = {};
            bool ok;
            do {
                ok = true;
#pragma unroll
                for (int m = 0; m < (kPre ? M : 0); ++m) raw[m] = ll_load1(p.xl + (size_t)m * n_rows + 2 * pair0 + tid);
#pragma unroll
                for (int m = 0; m < (kPre ? M : 0); ++m) ok = ok && ll_ready(raw[m], tag_x);
            } while (!ok && ll_keep_waiting(p, ll_spins, ll_t0, stage));
#pragma unroll
            for (int m = 0; m < (kPre ? M : 0); ++m) pre[m] = __uint_as_float((uint32_t)raw[m]);
        } else {
#pragma unroll
            for (int m = 0; m < (kPre ? M : 0); ++m) pre[m] = __ldcg(p.x + (size_t)m * n_rows + 2 * pair0 + tid);
        }
    }

    // ---- RMSNorm statistics (same arithmetic for every row count). With one row the hidden state read here stays in
    //      registers for the window fill below (one L2 round trip less per stage); two and more rows whose window
    //      holds them whole take norm_rows_into_window() instead.
    float4 xr[kKeepX ? M : 1][3];
    float inv[M];
    constexpr bool kFusedNorm = (M >= 2);
    const bool fused = kFusedNorm && short_rows && n_seg <= wseg;  // whole rows in one window: statistics and fill in one go below
    if (norm && !fused) {
        float ssq[M];  // this thread's share of every row's sum of squares; per row the additions run in index order
#pragma unroll
        for (int m = 0; m < M; ++m) ssq[m] = 0.f;
        if (keep) {
            if (ll) {
                // all of this thread's words of all rows in flight together; then only the 16-byte halves whose tags are
                // still stale are loaded again, with a growing pause in between (a CTA that is early would otherwise
                // re-read 32 KB per row and round and crowd the other CTAs' weight streams out of L2's ports)
                unsigned long long raw[kKeepX ? M : 1][3][4] = {};
                unsigned stale = 0u;  // bit (m * 3 + c) * 2 + h
#pragma unroll
                for (int m = 0; m < (kKeepX ? M : 0); ++m)
#pragma unroll
                    for (int c = 0; c < 3; ++c)
                        if (!direct && (tid + c * kPassConsumers) * 4 < n_in) stale |= 3u << ((m * 3 + c) * 2);
                for (;;) {
#pragma unroll
                    for (int m = 0; m < (kKeepX ? M : 0); ++m)
#pragma unroll
                        for (int c = 0; c < 3; ++c) {
                            if (c >= chunks) break;
#pragma unroll
                            for (int h = 0; h < 2; ++h)
                                if (stale & (1u << ((m * 3 + c) * 2 + h)))
                                    ll_load2(p.xl + (size_t)m * n_in + (tid + c * kPassConsumers) * 4 + 2 * h, raw[m][c][2 * h], raw[m][c][2 * h + 1]);
                        }
#pragma unroll
                    for (int m = 0; m < (kKeepX ? M : 0); ++m)
#pragma unroll
                        for (int c = 0; c < 3; ++c) {
                            if (c >= chunks) break;
#pragma unroll
                            for (int h = 0; h < 2; ++h)
                                if ((stale & (1u << ((m * 3 + c) * 2 + h))) && ll_ready(raw[m][c][2 * h], tag_x) && ll_ready(raw[m][c][2 * h + 1], tag_x))
                                    stale &= ~(1u << ((m * 3 + c) * 2 + h));
                        }
                    if (stale == 0u || !ll_keep_waiting(p, ll_spins, ll_t0, stage)) break;
                    __nanosleep(ll_spins < 4 ? 100u : 300u);
                }
#pragma unroll
                for (int m = 0; m < (kKeepX ? M : 0); ++m)
#pragma unroll
                    for (int c = 0; c < 3; ++c)
                        xr[m][c] = make_float4(__uint_as_float((uint32_t)raw[m][c][0]), __uint_as_float((uint32_t)raw[m][c][1]),
                                               __uint_as_float((uint32_t)raw[m][c][2]), __uint_as_float((uint32_t)raw[m][c][3]));
            }
#pragma unroll
            for (int m = 0; m < M; ++m) {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    if (c >= chunks) break;
                    const int i = (tid + c * kPassConsumers) * 4;
                    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (ll && !direct) v = xr[kKeepX ? m : 0][c];
                    else if (ll) v = i < n_in ? load_row4(xf, p.embed, sm.tok, m, n_in, i) : v;
                    else if (i < n_in) v = __ldcg(reinterpret_cast<const float4*>(xf + (size_t)m * n_in + i));
                    xr[kKeepX ? m : 0][c] = v;
                    if (i < n_in) {
                        float s = ssq[m];
                        s = fmaf(v.x, v.x, s);
                        s = fmaf(v.y, v.y, s);
                        s = fmaf(v.z, v.z, s);
                        s = fmaf(v.w, v.w, s);
                        ssq[m] = s;
                    }
                }
            }
        } else {
            // long rows: the loads of up to four rows are in flight together (one memory round trip per four rows and stride)
            for (int i = tid * 4; i < n_in; i += kPassConsumers * 4) {
#pragma unroll
                for (int m0 = 0; m0 < M; m0 += 4) {
                    float4 v[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (m0 + u < M) v[u] = __ldcg(reinterpret_cast<const float4*>(xf + (size_t)(m0 + u) * n_in + i));
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (m0 + u < M) {
                            float s = ssq[m0 + u];
                            s = fmaf(v[u].x, v[u].x, s);
                            s = fmaf(v[u].y, v[u].y, s);
                            s = fmaf(v[u].z, v[u].z, s);
                            s = fmaf(v[u].w, v[u].w, s);
                            ssq[m0 + u] = s;
                        }
                }
            }
        }
#pragma unroll
        for (int m = 0; m < M; ++m) {
            const float s = warp_sum(ssq[m]);
            if (lane == 0) red[warp * (kPassMaxRows * 4) + m + kRedNorm] = s;
        }
        consumers_sync();
#pragma unroll
        for (int m = 0; m < M; ++m) {
            float s = 0.f;
#pragma unroll
            for (int w = 0; w < kPassConsumerWarps; ++w) s += red[w * (kPassMaxRows * 4) + m + kRedNorm];
            inv[m] = __frsqrt_rn(fmaf(s, p.inv_d, p.eps));
        }
    }
    trace_mark(p, stage, 6);

    long long cyc_wait = 0, cyc_work = 0;  // when tracing: cycles this warp spent waiting for slots / working on them
    // ---- stream the slab window by window
    const int g8 = lane >> 2, q4 = lane & 3;  // tensor-core fragment coordinates of this lane
    for (int w0 = 0; w0 < n_seg; w0 += wseg) {
        const int ws = min(wseg, n_seg - w0);
        const int k0 = w0 * kSegK;
        const int wlen = ws * kSegK;  // inputs in this window, including the zero padding past n_in
        // previous window fully consumed (the first one: the stage before has ended with a barrier behind its products; with 16 rows the warps that
        // drift apart without it cost more than it does, 7B width 684 -> 696 us)
        if (w0 > 0 || M > kMaxRows) consumers_sync();
        if (fused) {
            norm_rows_into_window<M>(xf, direct ? p.embed : nullptr, sm.tok, st.gain, n_in, wlen, xstride, p.inv_d, p.eps, xs, red);
        } else if (keep) {  // a single window (n_in <= 5760): normalise the rows held in registers
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                if (c >= chunks && c * kPassConsumers * 4 >= wlen) break;
                const int i = (tid + c * kPassConsumers) * 4;
                if (i < wlen) {
                    const bool in = i < n_in;
                    const uint2 gv = gpre[c];
                    const float g0 = bf_lo(gv.x), g1 = bf_hi(gv.x), g2 = bf_lo(gv.y), g3 = bf_hi(gv.y);
#pragma unroll
                    for (int m = 0; m < M; ++m) {
                        uint2 o = make_uint2(0u, 0u);
                        if (in) {
                            const float4 v = xr[kKeepX ? m : 0][c];
                            __nv_bfloat162 lo = __floats2bfloat162_rn(v.x * inv[m] * g0, v.y * inv[m] * g1);
                            __nv_bfloat162 hi = __floats2bfloat162_rn(v.z * inv[m] * g2, v.w * inv[m] * g3);
                            o.x = *reinterpret_cast<uint32_t*>(&lo);
                            o.y = *reinterpret_cast<uint32_t*>(&hi);
                        }
                        *reinterpret_cast<uint2*>(xs + (size_t)m * xstride + i) = o;
                    }
                }
            }
            for (int i = kPassConsumers * 12 + tid * 4; i < wlen; i += kPassConsumers * 4)  // zero padding past 5760
                for (int m = 0; m < M; ++m) *reinterpret_cast<uint2*>(xs + (size_t)m * xstride + i) = make_uint2(0u, 0u);
        } else if (norm) {
            for (int i = tid * 4; i < wlen; i += kPassConsumers * 4) {
                const bool in = k0 + i < n_in;
                uint2 gv = make_uint2(0u, 0u);
                if (in) gv = *reinterpret_cast<const uint2*>(st.gain + k0 + i);
                const float g0 = bf_lo(gv.x), g1 = bf_hi(gv.x), g2 = bf_lo(gv.y), g3 = bf_hi(gv.y);
#pragma unroll
                for (int m0 = 0; m0 < M; m0 += 4) {
                    float4 v[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (m0 + u < M && in) v[u] = __ldcg(reinterpret_cast<const float4*>(xf + (size_t)(m0 + u) * n_in + k0 + i));
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (m0 + u < M) {
                            const int m = m0 + u;
                            uint2 o = make_uint2(0u, 0u);
                            if (in) {
                                __nv_bfloat162 lo = __floats2bfloat162_rn(v[u].x * inv[m] * g0, v[u].y * inv[m] * g1);
                                __nv_bfloat162 hi = __floats2bfloat162_rn(v[u].z * inv[m] * g2, v[u].w * inv[m] * g3);
                                o.x = *reinterpret_cast<uint32_t*>(&lo);
                                o.y = *reinterpret_cast<uint32_t*>(&hi);
                            }
                            *reinterpret_cast<uint2*>(xs + (size_t)m * xstride + i) = o;
                        }
                }
            }
        } else if (ll) {
            // bf16 inputs as tagged words (two bf16 each): the window holds whole rows; two 8-element chunks per row and
            // thread in flight together, repeated until every tag is the expected one
            const uint2* src = (type == kStOproj) ? p.al : p.tl;
            for (int i0 = tid * 8; i0 < wlen; i0 += 2 * kPassConsumers * 8) {
                unsigned long long raw[kLLCap ? M : 1][2][4] = {};
                unsigned stale = 0u;  // bit (m * 2 + u) * 2 + h
#pragma unroll
                for (int m = 0; m < (kLLCap ? M : 0); ++m)
#pragma unroll
                    for (int u = 0; u < 2; ++u)
                        if (i0 + u * kPassConsumers * 8 < n_in) stale |= 3u << ((m * 2 + u) * 2);
                for (;;) {
#pragma unroll
                    for (int m = 0; m < (kLLCap ? M : 0); ++m)
#pragma unroll
                        for (int u = 0; u < 2; ++u)
#pragma unroll
                            for (int h = 0; h < 2; ++h)
                                if (stale & (1u << ((m * 2 + u) * 2 + h)))
                                    ll_load2(src + (((size_t)m * n_in + i0 + u * kPassConsumers * 8) >> 1) + 2 * h, raw[m][u][2 * h], raw[m][u][2 * h + 1]);
#pragma unroll
                    for (int m = 0; m < (kLLCap ? M : 0); ++m)
#pragma unroll
                        for (int u = 0; u < 2; ++u)
#pragma unroll
                            for (int h = 0; h < 2; ++h)
                                if ((stale & (1u << ((m * 2 + u) * 2 + h))) && ll_ready(raw[m][u][2 * h], tag_in) && ll_ready(raw[m][u][2 * h + 1], tag_in))
                                    stale &= ~(1u << ((m * 2 + u) * 2 + h));
                    if (stale == 0u || !ll_keep_waiting(p, ll_spins, ll_t0, stage)) break;
                    __nanosleep(ll_spins < 4 ? 100u : 300u);
                }
#pragma unroll
                for (int m = 0; m < (kLLCap ? M : 0); ++m)
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const int i = i0 + u * kPassConsumers * 8;
                        if (i < wlen) {
                            uint4 v = make_uint4(0u, 0u, 0u, 0u);
                            if (i < n_in) v = make_uint4((uint32_t)raw[m][u][0], (uint32_t)raw[m][u][1], (uint32_t)raw[m][u][2], (uint32_t)raw[m][u][3]);
                            *reinterpret_cast<uint4*>(xs + (size_t)m * xstride + i) = v;
                        }
                    }
            }
        } else {
            for (int i = tid * 8; i < wlen; i += kPassConsumers * 8) {
                const bool in = k0 + i < n_in;
#pragma unroll
                for (int m = 0; m < M; ++m) {
                    uint4 v = make_uint4(0u, 0u, 0u, 0u);
                    if (in) v = __ldcg(reinterpret_cast<const uint4*>(xb + (size_t)m * n_in + k0 + i));
                    *reinterpret_cast<uint4*>(xs + (size_t)m * xstride + i) = v;
                }
            }
        }
        consumers_sync();

        if (w0 == 0) trace_mark(p, stage, 7);
        // Ring order is segment-major: consecutive items are different groups, i.e. different warps. One item is up to
        // 16 weight rows x 256 inputs, stored as column blocks of 32 inputs ([block][row][64 bytes]); lane (g8, q4)
        // owns inputs 32*block + 8*q4 .. +7 of rows g8 and g8 + 8. Two m16n8k16 steps per block: the weights are the
        // 16-row A operand, the activation rows the 8 columns of the B operand (columns >= M are zero), so every
        // step covers 16 weight rows and nothing of the tile is wasted on padding rows.
        const __nv_bfloat16* xa = xs + (size_t)min(g8, M - 1) * xstride + q4 * 8;
        const __nv_bfloat16* xb2 = xs + (size_t)min(g8 + 8, M - 1) * xstride + q4 * 8;
        const int set = sm.warp_set[type * 16 + warp];
        const int ks = set & 0xFF, o_first = set >> 8;             // which copy of the partial sums this warp adds into, and its first group
        const int o_step = (S > 1) ? n_oct : kPassConsumerWarps;  // S > 1: exactly one group per warp
        float* psum_w = psum + (size_t)ks * copy_stride;
        // this warp set's segments of the window: ks, ks + S, ... (one remainder per window instead of one per segment)
        int seg_first = w0;
        if (S > 1) seg_first += ks;
        if (S > 1 && w0 > 0) {
            const int r = w0 % S;
            seg_first = w0 + (ks >= r ? ks - r : ks + S - r);
        }
        for (int seg = seg_first; seg < w0 + ws; seg += S) {
            const int sg = seg - w0;
            for (int o = o_first; o < n_oct; o += o_step) {
                const uint32_t g = gi + (uint32_t)(seg * n_oct + o);
                const int rows = 2 * min(kGrpPairs, np - kGrpPairs * o);
                const long long tw0 = p.trace ? clock64() : 0;
                int slot;
                uint32_t gen;
                ring_locate(p, g, slot, gen);
                ring_wait_full(p, sm, g, slot, gen, stage, M * 1000 + seg);
                const long long tw1 = p.trace ? clock64() : 0;
                const unsigned char* sl = sm.ring + (size_t)slot * kSlotBytes + g8 * 64 + q4 * 16;
                const int blk = rows * 64;
                const int nblk = min(kSegBlocks, ((n_in + 31) >> 5) - seg * kSegBlocks);
                // Four independent accumulators (column block parity x half of the block), added in a fixed order;
                // acc2 holds activation rows 8..15 (row passes of a prompt with more than 8 rows).
                float acc[4][4], acc2[M > 8 ? 4 : 1][4];
#pragma unroll
                for (int a = 0; a < 4; ++a) acc[a][0] = acc[a][1] = acc[a][2] = acc[a][3] = 0.f;
#pragma unroll
                for (int a = 0; a < (M > 8 ? 4 : 1); ++a) acc2[a][0] = acc2[a][1] = acc2[a][2] = acc2[a][3] = 0.f;
                // Operands of four column blocks in registers, two with more than eight rows (16 rows, 2048 wide: 213 -> 195 us, they spilled), then two steps for each block. Lanes whose weight row lies
                // beyond the item's rows, or whose activation row beyond M, read whatever follows in the slot / the last
                // activation row: every output element depends on its own weight row and activation row only, and the
                // outputs of such rows are never stored. Only column blocks past the end of a ragged last segment must
                // contribute nothing and are replaced by zeros.
                if (nblk == kSegBlocks) {
#pragma unroll (M > 8 ? 1 : kSegBlocks / kOpBlocks)
                    for (int h = 0; h < kSegBlocks / kOpBlocks; ++h) {
                        uint4 wlo[kOpBlocks], whi[kOpBlocks], xv[kOpBlocks], xv2[M > 8 ? kOpBlocks : 1];
#pragma unroll
                        for (int j = 0; j < kOpBlocks; ++j) {
                            wlo[j] = *reinterpret_cast<const uint4*>(sl + (h * kOpBlocks + j) * blk);
                            whi[j] = *reinterpret_cast<const uint4*>(sl + (h * kOpBlocks + j) * blk + 8 * 64);
                            xv[j] = *reinterpret_cast<const uint4*>(xa + sg * kSegK + (h * kOpBlocks + j) * 32);
                            if (M > 8) xv2[j] = *reinterpret_cast<const uint4*>(xb2 + sg * kSegK + (h * kOpBlocks + j) * 32);
                        }
#pragma unroll
                        for (int j = 0; j < kOpBlocks; ++j) {
                            mma_bf16_16816(acc[(j & 1) * 2 + 0], wlo[j].x, whi[j].x, wlo[j].y, whi[j].y, xv[j].x, xv[j].y);
                            mma_bf16_16816(acc[(j & 1) * 2 + 1], wlo[j].z, whi[j].z, wlo[j].w, whi[j].w, xv[j].z, xv[j].w);
                            if (M > 8) {
                                mma_bf16_16816(acc2[(j & 1) * 2 + 0], wlo[j].x, whi[j].x, wlo[j].y, whi[j].y, xv2[j].x, xv2[j].y);
                                mma_bf16_16816(acc2[(j & 1) * 2 + 1], wlo[j].z, whi[j].z, wlo[j].w, whi[j].w, xv2[j].z, xv2[j].w);
                            }
                        }
                    }
                } else {
#pragma unroll 1
                    for (int h = 0; h * kOpBlocks < nblk; ++h) {
                        uint4 wlo[kOpBlocks], whi[kOpBlocks], xv[kOpBlocks], xv2[M > 8 ? kOpBlocks : 1];
#pragma unroll
                        for (int j = 0; j < kOpBlocks; ++j) {
                            const bool inb = h * kOpBlocks + j < nblk;
                            wlo[j] = inb ? *reinterpret_cast<const uint4*>(sl + (h * kOpBlocks + j) * blk) : make_uint4(0u, 0u, 0u, 0u);
                            whi[j] = inb ? *reinterpret_cast<const uint4*>(sl + (h * kOpBlocks + j) * blk + 8 * 64) : make_uint4(0u, 0u, 0u, 0u);
                            xv[j] = *reinterpret_cast<const uint4*>(xa + sg * kSegK + (h * kOpBlocks + j) * 32);
                            if (M > 8) xv2[j] = *reinterpret_cast<const uint4*>(xb2 + sg * kSegK + (h * kOpBlocks + j) * 32);
                        }
#pragma unroll
                        for (int j = 0; j < kOpBlocks; ++j) {
                            mma_bf16_16816(acc[(j & 1) * 2 + 0], wlo[j].x, whi[j].x, wlo[j].y, whi[j].y, xv[j].x, xv[j].y);
                            mma_bf16_16816(acc[(j & 1) * 2 + 1], wlo[j].z, whi[j].z, wlo[j].w, whi[j].w, xv[j].z, xv[j].w);
                            if (M > 8) {
                                mma_bf16_16816(acc2[(j & 1) * 2 + 0], wlo[j].x, whi[j].x, wlo[j].y, whi[j].y, xv2[j].x, xv2[j].y);
                                mma_bf16_16816(acc2[(j & 1) * 2 + 1], wlo[j].z, whi[j].z, wlo[j].w, whi[j].w, xv2[j].z, xv2[j].w);
                            }
                        }
                    }
                }
                __syncwarp();
                if (lane == 0) ring_release(sm, slot, gen);
                // c[0], c[1]: weight row g8 of the group, activation rows 2*q4 and 2*q4 + 1; c[2], c[3]: weight row g8 + 8.
                // Local weight row 16*o + r is row (r & 1) of local pair 8*o + r/2. Segments are added in ascending
                // order, always by this lane.
#pragma unroll
                for (int hr = 0; hr < 2; ++hr) {
                    const int wr = g8 + 8 * hr;
                    if (wr < rows) {
                        float* dst = psum_w + (size_t)(kGrpRows * o + wr) * M;
                        const bool first = seg == ((S > 1) ? ks : 0);
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const int mm = 2 * q4 + e;
                            if (mm < M) {
                                const float v = (acc[0][2 * hr + e] + acc[2][2 * hr + e]) + (acc[1][2 * hr + e] + acc[3][2 * hr + e]);
                                dst[mm] = first ? v : dst[mm] + v;
                            }
                            if (M > 8 && mm + 8 < M) {
                                const float v = (acc2[0][2 * hr + e] + acc2[2][2 * hr + e]) + (acc2[1][2 * hr + e] + acc2[3][2 * hr + e]);
                                dst[mm + 8] = first ? v : dst[mm + 8] + v;
                            }
                        }
                    }
                }
                if (p.trace) {
                    cyc_wait += tw1 - tw0;
                    cyc_work += clock64() - tw1;
                }
            }
        }
    }
    gi += (uint32_t)(n_oct * n_seg);
    consumers_sync();
    trace_mark(p, stage, 2);
    if (p.trace && tid == 0) {
        p.trace[((size_t)stage * kTraceEntries + 4) * gridDim.x + blockIdx.x] = cyc_wait;
        p.trace[((size_t)stage * kTraceEntries + 5) * gridDim.x + blockIdx.x] = cyc_work;
    }

    if constexpr (!kSpreadEpi) {
    // ---- epilogue of a pass of one or two rows: thread t owns pairs t, t+480, ... of this CTA and all M rows of them
    float s_loc[M][3];
    float best_v[M], sec_v[M];
    int best_i[M];
#pragma unroll
    for (int m = 0; m < M; ++m) {
        s_loc[m][0] = s_loc[m][1] = s_loc[m][2] = 0.f;
        best_v[m] = sec_v[m] = -INFINITY;
        best_i[m] = INT_MAX;
    }
    const bool resid = (type == kStOproj || type == kStDown);
    if (resid) {
        // residual add: one thread per weight row, the M loads of the old hidden state issued together
        float* out = p.x;
        for (int e = tid; e < np * 2; e += kPassConsumers) {
            const int row = 2 * pair0 + e;
            if (row >= n_rows) continue;
            float xv[M];
#pragma unroll
            for (int m = 0; m < M; ++m) {
                if (kPre && e == tid) {
                    xv[m] = pre[kPre ? m : 0];
                } else if (ll) {  // (a CTA with more rows than threads: not on the benchmark shapes)
                    unsigned long long raw;
                    do raw = ll_load1(p.xl + (size_t)m * n_rows + row);
                    while (!ll_ready(raw, tag_x) && ll_keep_waiting(p, ll_spins, ll_t0, stage));
                    xv[m] = __uint_as_float((uint32_t)raw);
                } else {
                    xv[m] = __ldcg(out + (size_t)m * n_rows + row);
                }
            }
#pragma unroll
            for (int m = 0; m < M; ++m) {
                const float y = xv[m] + psum_total(psum, e * M + m, S, copy_stride);
                if (ll) ll_store(p.xl + (size_t)m * n_rows + row, __float_as_uint(y), tag_out);
                else out[(size_t)m * n_rows + row] = y;
                s_loc[m][0] = fmaf(xv[m], y, s_loc[m][0]);
                s_loc[m][1] = fmaf(xv[m], xv[m], s_loc[m][1]);
                s_loc[m][2] = fmaf(y, y, s_loc[m][2]);
            }
        }
    }
    if (ll && type == kStGateUp) {
        // pair0 and np are even: outputs pair0 + 2j and pair0 + 2j + 1 form one tagged word
        for (int pj = tid; 2 * pj < np; pj += kPassConsumers) {
#pragma unroll
            for (int m = 0; m < M; ++m) {
                uint32_t word = 0u;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int pl = 2 * pj + h;
                    const float va = psum_total(psum, (pl * 2 + 0) * M + m, S, copy_stride), vb = psum_total(psum, (pl * 2 + 1) * M + m, S, copy_stride);
                    const float t = va / (1.0f + expf(-va)) * vb;
                    word |= (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(t)) << (16 * h);
                }
                ll_store(p.tl + (((size_t)m * (n_rows >> 1) + pair0) >> 1) + pj, word, tag_out);
            }
        }
    }
    for (int pl = (resid || (ll && type == kStGateUp)) ? np : tid; pl < np; pl += kPassConsumers) {
        int ra, rb;
        stage_pair_rows(type, p, pair0 + pl, ra, rb);
        const bool has_b = rb < n_rows;
        // rotary factors of all rows first: the stores below may alias them as far as the compiler knows, and one
        // memory round trip per row would add up
        float rc[M], rs[M];
        if (type == kStQkv && ra < p.d_model + p.kv_dim) {
            const int half = p.head_dim >> 1, jr = p.hd_shift ? (ra & (p.head_dim - 1)) : ra % p.head_dim;
#pragma unroll
            for (int m = 0; m < M; ++m) {
                rc[m] = (kPre && pl == tid) ? pre[kPre ? m : 0] : p.rope_cos[(size_t)(p.pos0 + m) * half + jr];
                rs[m] = (kPre && pl == tid) ? pre[kPre ? M + m : 0] : p.rope_sin[(size_t)(p.pos0 + m) * half + jr];
            }
        }
#pragma unroll
        for (int m = 0; m < M; ++m) {
            float va = psum_total(psum, (pl * 2 + 0) * M + m, S, copy_stride), vb = psum_total(psum, (pl * 2 + 1) * M + m, S, copy_stride);
            if (type == kStGateUp) {
                const float t = va / (1.0f + expf(-va)) * vb;
                p.t[(size_t)m * (n_rows >> 1) + (pair0 + pl)] = __float2bfloat16_rn(t);
            } else if (type == kStQkv) {
                const int pos = p.pos0 + m;
                if (ra < p.d_model + p.kv_dim) {  // q or k: rotate the pair (j, j + head_dim/2) by pos * theta_j
                    // explicit roundings: the same arithmetic whatever the row count the kernel was compiled for
                    const float c = rc[m], s = rs[m];
                    const float r0 = __fmaf_rn(va, c, -__fmul_rn(vb, s));
                    const float r1 = __fmaf_rn(vb, c, __fmul_rn(va, s));
                    va = r0;
                    vb = r1;
                }
                const __nv_bfloat16 ha = __float2bfloat16_rn(va), hb = __float2bfloat16_rn(vb);
                if (ll) {  // the attention stage of this pass takes q, k, v from tagged words (k, v also go to the cache)
                    uint2* dst = ra < p.d_model ? p.ql : (ra < p.d_model + p.kv_dim ? p.kl : p.vl);
                    const int off = ra < p.d_model ? 0 : (ra < p.d_model + p.kv_dim ? p.d_model : p.d_model + p.kv_dim);
                    ll_store(dst + (ra - off), (uint32_t)__bfloat16_as_ushort(ha), tag_out);
                    ll_store(dst + (rb - off), (uint32_t)__bfloat16_as_ushort(hb), tag_out);
                }
                if (ra < p.d_model) {
                    if (!ll) {
                        p.q[(size_t)m * p.d_model + ra] = ha;
                        p.q[(size_t)m * p.d_model + rb] = hb;
                    }
                } else if (ra < p.d_model + p.kv_dim) {
                    st.k_cache[(size_t)pos * p.kv_dim + (ra - p.d_model)] = ha;
                    st.k_cache[(size_t)pos * p.kv_dim + (rb - p.d_model)] = hb;
                } else {
                    st.v_cache[(size_t)pos * p.kv_dim + (ra - p.d_model - p.kv_dim)] = ha;
                    st.v_cache[(size_t)pos * p.kv_dim + (rb - p.d_model - p.kv_dim)] = hb;
                }
            } else {  // LM head
                if (p.logits_out) {
                    p.logits_out[(size_t)m * n_rows + ra] = va;
                    if (has_b) p.logits_out[(size_t)m * n_rows + rb] = vb;
                }
                if (va > best_v[m]) {  // rows come in ascending order: an equal logit keeps the lower index
                    sec_v[m] = best_v[m];
                    best_v[m] = va;
                    best_i[m] = ra;
                } else {
                    sec_v[m] = fmaxf(sec_v[m], va);
                }
                if (has_b) {
                    if (vb > best_v[m]) {
                        sec_v[m] = best_v[m];
                        best_v[m] = vb;
                        best_i[m] = rb;
                    } else {
                        sec_v[m] = fmaxf(sec_v[m], vb);
                    }
                }
            }
        }
    }

    if (type == kStOproj || type == kStDown) {
        // cosine similarity of the hidden state before and after this sublayer: warp-shuffle partial dot and
        // norm products, one block-level finish; the per-CTA partials are combined by the finish stage of the pass
#pragma unroll
        for (int m = 0; m < M; ++m)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const float v = warp_sum(s_loc[m][j]);
                if (lane == 0) red[warp * (kPassMaxRows * 4) + m * 4 + j] = v;
            }
        consumers_sync();
        if (tid < M * 3) {
            const int m = tid / 3, j = tid - m * 3;
            float tot = 0.f;
#pragma unroll
            for (int w = 0; w < kPassConsumerWarps; ++w) tot += red[w * (kPassMaxRows * 4) + m * 4 + j];
            p.partials[(((size_t)st.resid_slot * gridDim.x + blockIdx.x) * kPassMaxRows + m) * 4 + j] = tot;
        }
    } else if (type == kStLmHead) {
#pragma unroll
        for (int m = 0; m < M; ++m) {
            float v = best_v[m], sc = sec_v[m];
            int i = best_i[m];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const float ov = __shfl_xor_sync(0xffffffffu, v, o);
                const int oi = __shfl_xor_sync(0xffffffffu, i, o);
                const float os = __shfl_xor_sync(0xffffffffu, sc, o);
                top2_merge(v, i, sc, ov, oi, os);
            }
            if (lane == 0) {
                red[warp * (kPassMaxRows * 4) + m * 4 + 0] = v;
                red[warp * (kPassMaxRows * 4) + m * 4 + 1] = __int_as_float(i);
                red[warp * (kPassMaxRows * 4) + m * 4 + 2] = sc;
            }
        }
        consumers_sync();
        if (tid < M) {
            float v = -INFINITY, sc = -INFINITY;
            int i = INT_MAX;
            for (int w = 0; w < kPassConsumerWarps; ++w)
                top2_merge(v, i, sc, red[w * (kPassMaxRows * 4) + tid * 4 + 0], __float_as_int(red[w * (kPassMaxRows * 4) + tid * 4 + 1]),
                           red[w * (kPassMaxRows * 4) + tid * 4 + 2]);
            float* lmp = p.partials + (size_t)p.n_resid * gridDim.x * kPassMaxRows * 4;
            lmp[((size_t)blockIdx.x * kPassMaxRows + tid) * 4 + 0] = v;
            lmp[((size_t)blockIdx.x * kPassMaxRows + tid) * 4 + 1] = __int_as_float(i);
            lmp[((size_t)blockIdx.x * kPassMaxRows + tid) * 4 + 2] = sc;
        }
    }
    } else {
        if (type == kStOproj || type == kStDown)
            epi_resid_rows<M>(p.x, psum, red, p.partials + ((size_t)st.resid_slot * gridDim.x + blockIdx.x) * kPassMaxRows * 4, n_rows, pair0, np, S,
                              pre0);
        else if (type == kStQkv)
            epi_qkv_rows<M>(psum, pair0, np, S, p.pos0, p.d_model, p.kv_dim, p.head_dim, p.rope_cos, p.rope_sin, p.q, st.k_cache, st.v_cache, pre0,
                            pre1);
        else if (type == kStGateUp)
            epi_gateup_rows<M>(psum, pair0, np, S, p.t, n_rows >> 1);
        else
            epi_lmhead_rows<M>(psum, red, pair0, np, S, n_rows, p.logits_out,
                               p.partials + ((size_t)p.n_resid * gridDim.x + blockIdx.x) * kPassMaxRows * 4);
    }
    if (type == kStLmHead) {
        if (kFewRows<M> && blockIdx.x < (unsigned)p.n_resid) bar_sync(kFinishBar, kPassThreads);  // this CTA's share of the cosines is done as well
        const bool last_cta = last_cta_consumers(p.fin_counter, sm.flag);
        if (p.logits_host) {  // (behind the ticket, whose release would wait for the way over PCIe)
            const int n = min(2 * np, n_rows - 2 * pair0);
            for (int i = tid; i < M * n; i += kPassConsumers) {
                const int m = i / n, e = i - m * n;
                p.logits_host[(size_t)m * n_rows + 2 * pair0 + e] = psum_total(psum, e * M + m, S, copy_stride);
            }
        }
        if (last_cta) {
            int* g = reinterpret_cast<int*>(red);
            for (int m = warp; m < M; m += kPassConsumerWarps) {  // a warp per row: lanes scan the per-CTA partials, then a butterfly; ties -> lowest index
                float v = -INFINITY, sc = -INFINITY;
                int i = INT_MAX;
                const float* lmp = p.partials + (size_t)p.n_resid * gridDim.x * kPassMaxRows * 4;
                for (unsigned b = lane; b < gridDim.x; b += 32) {
                    const float4 o4 = __ldcg(reinterpret_cast<const float4*>(lmp + ((size_t)b * kPassMaxRows + m) * 4));
                    top2_merge(v, i, sc, o4.x, __float_as_int(o4.y), o4.z);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const float ov = __shfl_xor_sync(0xffffffffu, v, o);
                    const int oi = __shfl_xor_sync(0xffffffffu, i, o);
                    const float os = __shfl_xor_sync(0xffffffffu, sc, o);
                    top2_merge(v, i, sc, ov, oi, os);
                }
                if (lane == 0) {
                    if (i == INT_MAX) i = 0;
                    p.argmax_out[m] = i;
                    if (p.margin_out) p.margin_out[m] = v - sc;
                    g[m] = i;
                    if (p.host_out && m == M - 1) reinterpret_cast<float*>(p.host_out)[kHostMargin] = v - sc;
                }
            }
            consumers_sync();
            if (tid == 0) {
                int* h = p.host_out;
                if (p.accept_out) {
                    // greedy verification (Section 1): drafted token j+1 is accepted while it equals M's argmax of row j
                    int a = 0;
                    while (a < M - 1 && pass_token(p, a + 1) == g[a]) ++a;
                    for (int j = 0; j <= a + 1; ++j) {
                        const int v = j == 0 ? a : (j <= a ? pass_token(p, j) : g[a]);
                        p.accept_out[j] = v;
                        if (h) h[j] = v;
                    }
                } else if (h) {
                    h[0] = g[M - 1];
                }
                if (h) {  // every CTA has arrived here, so whoever gave up waiting has said so
                    for (int j = 0; j < 8; ++j) h[kHostErr + j] = *(static_cast<volatile int*>(p.err) + j);
                    h[kHostStamp] = p.host_stamp;
                }
                *p.fin_counter = 0u;
            }
        }
    }
}

// ============================================================================================ finish stage
// Cosine similarities of all residual stages of the pass (summand of C_l, Section 3.2). Residual stage r is finished by the
// producer warp of CTA r mod gridDim.x when its last copy is on its way, beside the LM head's products: the per-CTA partials b = lane, lane +
// 32, ... are added in order, then by an xor butterfly, all in double precision (fixed order, independent of the row count). As a
// stage of the consumer warps it stood between the last sublayer and the LM head (figures: pass_kernel, embedding stage).
// Passes of more rows finish them by their consumer warps, a warp per row.
template <int M>
__device__ void finish_stage(const PassParams& p, const PassSmem& sm) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int r = blockIdx.x; r < p.n_resid; r += gridDim.x) {
        const float* part = p.partials + (size_t)r * gridDim.x * kPassMaxRows * 4;
        const ResidOut out = p.resid[r];
        for (int m = warp; m < M; m += kPassConsumerWarps) {
            double sxy = 0, sxx = 0, syy = 0;
            for (unsigned b = lane; b < gridDim.x; b += 32) {
                const float4 v = __ldcg(reinterpret_cast<const float4*>(part + ((size_t)b * kPassMaxRows + m) * 4));
                sxy += (double)v.x, sxx += (double)v.y, syy += (double)v.z;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                sxy += __shfl_xor_sync(0xffffffffu, sxy, o);
                sxx += __shfl_xor_sync(0xffffffffu, sxx, o);
                syy += __shfl_xor_sync(0xffffffffu, syy, o);
            }
            if (lane == 0) out.cos_out[m] = sm.red[m] = (float)(sxy / fmax(sqrt(sxx) * sqrt(syy), 1e-30));
        }
        consumers_sync();
        if (tid == 0 && p.acc_sim && out.sumcos) {  // rows are added in order: chunked prefill equals one-shot prefill
            double acc = *out.sumcos;
            for (int m = 0; m < M; ++m) acc += (double)sm.red[m];
            *out.sumcos = acc;
            p.sim_host[out.sumcos - p.sim_base] = acc;
        }
        consumers_sync();
    }
}
template <int M>
__device__ __forceinline__ void finish_rows(const PassParams& p) {
    static_assert(kFewRows<M>, "the partials of all rows are requested together");
    const int lane = threadIdx.x & 31;
    if (blockIdx.x >= (unsigned)p.n_resid) return;
    if (lane == 0) {
        grid_poll(p, p.grid_bar, p.bar_base + (unsigned)p.finish_stage * gridDim.x + p.bar_extra_last);  // (test hook: extra arrivals that never come)
    }
    __syncwarp();
    for (int r = blockIdx.x; r < p.n_resid; r += gridDim.x) {
        const float4* part = reinterpret_cast<const float4*>(p.partials + (size_t)r * gridDim.x * kPassMaxRows * 4);
        const ResidOut out = p.resid[r];
        const bool sum = lane == 0 && p.acc_sim && out.sumcos;
        double acc = sum ? *out.sumcos : 0.0;  // rows are added in order: chunked prefill equals one-shot prefill
        double s[M][3] = {};
        for (unsigned b0 = 0; b0 < gridDim.x; b0 += 160) {
            float4 v[M][5];
#pragma unroll
            for (int m = 0; m < M; ++m)
#pragma unroll
                for (int i = 0; i < 5; ++i) {
                    const unsigned b = b0 + i * 32 + lane;
                    v[m][i] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (b < gridDim.x) v[m][i] = __ldcg(part + (size_t)b * kPassMaxRows + m);
                }
#pragma unroll
            for (int m = 0; m < M; ++m)
#pragma unroll
                for (int i = 0; i < 5; ++i) s[m][0] += (double)v[m][i].x, s[m][1] += (double)v[m][i].y, s[m][2] += (double)v[m][i].z;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int m = 0; m < M; ++m)
#pragma unroll
                for (int j = 0; j < 3; ++j) s[m][j] += __shfl_xor_sync(0xffffffffu, s[m][j], o);
        if (lane == 0) {
#pragma unroll
            for (int m = 0; m < M; ++m) {
                const float c = (float)(s[m][0] / fmax(sqrt(s[m][1]) * sqrt(s[m][2]), 1e-30));
                out.cos_out[m] = c;
                acc += (double)c;
            }
        }
        if (sum) {
            *out.sumcos = acc;
            p.sim_host[out.sumcos - p.sim_base] = acc;
        }
    }
    __syncwarp();
    if (p.finish_stage + 1 < p.n_stages) bar_arrive(kFinishBar, kPassThreads);  // the LM head stage's last word comes after this
}

// ============================================================================================ attention stage
// Byte offset of (key row r of the 128-key tile, 16-byte chunk c of the head) inside the tile's ring slots.
struct TileAddr {
    int nhb, row_bytes, swz;
    __device__ __forceinline__ void locate(int r, int c, int& slot_in_tile, int& off) const {
        const int rg = r / kBoxKeys, rr = r % kBoxKeys;
        const int hb = (nhb > 1) ? (c >> 3) : 0;
        const int cc = (nhb > 1) ? (c & 7) : c;
        slot_in_tile = rg * nhb + hb;
        off = rr * row_bytes + ((swz ? (cc ^ (rr & 7)) : cc) << 4);
    }
};

// Four 8x8 matrices of bf16 from shared memory, a row address per lane; the second form hands out their transposes.
__device__ __forceinline__ void ldmatrix4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldmatrix4_trans(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
// A * B alone: the sum of 16 products starts from zero
__device__ __forceinline__ void mma_bf16_zero(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
                 : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}

// Work items (kv head, 128-key chunk) of this CTA on the tensor cores (mma.sync m16n8k16), a group of four warps to an item. The COLUMNS of the
// products are the (row, query head) pairs that share the item's keys, eight at a time; what a column gets does not depend on its
// neighbours, so neither does a row's result on the row count.
//   S^T = K Q^T: 16 keys are the rows of a step (a warp has 32 keys), both operands read with ldmatrix; every 16 products start from zero, and the sums
//   of a score are added on the CUDA cores, from heads of 128 on as a tree.
//   softmax statistics of the chunk in fp32, the scale behind the difference from the maximum, the probabilities as the exact sum of three bf16 terms (cut off at 8 bits each) to shared memory.
//   O^T = V^T P: 16 dimensions are the rows (a warp has head_dim / 4 of them), V read transposed; every 16 products of a term start from zero as
//   above. (One or two columns have room for their three terms in one product: a third of the steps.)
// The order of the keys inside a block of 16 is free. Row r of a step is key r (r < 8) or 8 + ((r - 8) ^ 4): a lane then holds two keys that become
// neighbours in P, and the eight rows of every matrix, of K as of V, have different swizzles: no bank conflicts.
// Error: the tensor core cuts off what lies below the last bits of its sum (on average 0.2 2^-24 of a score), and every addition behind it rounds. The
// tree, and the scale behind the subtraction, keep a score within what four chains of FMAs gave: two keys with equal scores, errors in 2^-24 of the
// score, heads of 128 and 256: FMAs 0.56 and 0.55, sums added one after the other 0.79 and 0.98, this 0.47 and 0.52. Attention of one to nine
// rows on up to 8000 positions, heads of 64 and 128 (error of the fp32 output, 2^-24): 2.06, 2.07, 1.74; heads of 128 of a 40-head decoder 3.57,
// 4.31, 3.31. Heads of up to 64 have four sums at most, in a chain. The tree costs 0-1.5 % with heads of 128 (16 rows of the 7B width, four layers,
// 590 -> 598 us, five rows 404.5 -> 405.2), 0-3 % with 256.
// What bounds it: at 8000 positions of the 7B width the K/V stream (20 us a layer), the barrier and the merge behind it (10 us); at few positions the chain of an item
// (three barriers, about 3 us). Against fp32 FMAs fed from shared memory, heads one after the other and rows unrolled, kernel times in us (four layers of the 7B
// width; two layers 2048 wide with 32 heads of 64 on 8): five rows on 8000 keys 595 -> 546, nine 876 -> 720, 16 rows of a prompt 683 -> 636; grouped
// queries: one row on 8000 keys 111 -> 89, five 185 -> 140, nine 295 -> 188, 16 rows of a prompt 244 -> 211. (As the whole pass is now: 530, 699, 598; 87, 140,
// 182, 174.)
// HD: the head size when the code is compiled for it, 0: p.head_dim, 16 or 32 (a box of K or V is narrower than 128 bytes then, and not swizzled).
template <int M, bool LL, int HD>
__device__ void attn_items(const PassParams& p, const StageDesc& st, const PassSmem& sm, uint32_t gi0, int stage, int n_chunks, int first, int n_local) {
    const int tid = threadIdx.x, warp = tid >> 5;
    const int hd = HD ? HD : p.head_dim;
    constexpr int nhb = HD > 64 ? HD / 64 : 1;
    constexpr int tile_slots = (kAttnChunk / kBoxKeys) * nhb;
    const uint32_t tag_in = p.pass_tag + (uint32_t)(stage - 1), tag_out = p.pass_tag + (uint32_t)stage;  // W_qkv's stage precedes this one
    unsigned ll_spins = 0;
    long long ll_t0 = 0;
    const int grp = warp >> 2;
    const int gt = tid & 127, glane = gt & 31, gwarp = gt >> 5;
    const int g8 = glane >> 2, q4 = glane & 3;  // fragment coordinates: row g8 (and g8 + 8), columns 2 q4 and 2 q4 + 1
    const int bar_id = 2 + grp;
    const int group = p.n_heads / p.n_kv_heads;
    const int n_cols = M * group;  // column c: row c % M of query head c / M of the group
    const int vec_per_row = hd / 8;
    const TileAddr ta{nhb, HD ? 128 : hd * 2, HD ? 1 : 0};

    const int q_row = 2 * hd + 16, ct_max = attn_cols(M, group);
    unsigned char* qs = sm.reg_a + (size_t)grp * attn_scratch_bytes(M, group, hd);
    unsigned char* ps = qs + ct_max * q_row;
    float* red = reinterpret_cast<float*>(ps + 3 * ct_max * kAttnPRow);  // [4][8] maxima, then [4][8] sums
    const uint32_t ring_addr = smem_u32(sm.ring);

    // matrix rows that this lane addresses: of K (matrix bit 0: rows 8-15, bit 1: second half of 16 dimensions), of V (bit 0: second
    // half of 16 dimensions, bit 1: keys 8-15 of P's order), of Q and P (a column; the matrices follow one another along the row)
    const int mi = glane & 7, mat = glane >> 3;
    const int k_key = (mat & 1) ? 8 + (mi ^ 4) : mi;
    const int v_pos = (mat >> 1) * 8 + mi, v_key = (v_pos & 1) ? 8 + ((v_pos >> 1) ^ 4) : v_pos >> 1;
    const int k_swz = ta.swz ? (k_key & 7) : 0, v_swz = ta.swz ? (v_key & 7) : 0;

    int q_kvh = -1;  // kv head whose queries are in qs
    for (int j = grp; j < n_local; j += p.attn_groups) {
        const int idx = first + j;
        const int kvh = idx / n_chunks, chunk = idx - kvh * n_chunks;
        const int key0 = chunk * kAttnChunk;
        const int last_pos = p.pos0 + M - 1;
        const int n_valid = min(kAttnChunk, last_pos + 1 - key0);
        const uint32_t gk = gi0 + (uint32_t)(j * 2 * tile_slots), gv = gk + tile_slots;
        auto slot_off = [&](uint32_t g) -> uint32_t {
            int slot;
            uint32_t gen;
            ring_locate(p, g, slot, gen);
            return (uint32_t)slot * kSlotBytes;
        };
        // the boxes of a tile: every warp waits for all of them, a lane each
        auto wait_tile = [&](uint32_t g0, int tag) {
            if (glane < tile_slots) {
                int slot;
                uint32_t gen;
                ring_locate(p, g0 + (uint32_t)glane, slot, gen);
                ring_wait_full(p, sm, g0 + (uint32_t)glane, slot, gen, stage, tag);
            }
            __syncwarp();
        };
        auto release_tile = [&](uint32_t g0) {  // behind a barrier of the group
            if (gt < tile_slots) {
                fence_proxy_async_smem();
                int slot;
                uint32_t gen;
                ring_locate(p, g0 + (uint32_t)gt, slot, gen);
                ring_release(sm, slot, gen);
            }
        };
        // The rows that this pass has just written: the producer may have copied the tile before the QKV stage of this pass stored them. They are
        // requested before the waits, so patching the tiles costs no round trip.
        const int fresh0 = max(p.pos0, key0), fresh1 = min(last_pos, key0 + kAttnChunk - 1);
        const int n_fresh = fresh1 - fresh0 + 1;
        constexpr int kFreshPer = LL ? 1 : (M * (HD ? HD : 32) / 8 + 127) / 128;
        uint4 kpre[kFreshPer], vpre[kFreshPer];
        constexpr int kLLPer = LL && HD == 256 ? 2 : 1;  // tagged handoff: one word per element
        unsigned long long kraw[kLLPer] = {}, vraw[kLLPer] = {};
        const bool has_fresh = n_fresh > 0;
        if (LL) {
#pragma unroll
            for (int u = 0; u < kLLPer; ++u) {
                const int e = gt + u * 128;
                if (has_fresh && e < hd) kraw[u] = ll_load1(p.kl + (size_t)kvh * hd + e), vraw[u] = ll_load1(p.vl + (size_t)kvh * hd + e);
            }
        } else {
#pragma unroll
            for (int u = 0; u < kFreshPer; ++u) {
                const int i = gt + u * 128;
                kpre[u] = vpre[u] = make_uint4(0u, 0u, 0u, 0u);
                if (i < n_fresh * vec_per_row) {
                    const int fr = i / vec_per_row, c = i - fr * vec_per_row;
                    const size_t at = (size_t)(fresh0 + fr) * p.kv_dim + (size_t)kvh * hd + c * 8;
                    kpre[u] = __ldcg(reinterpret_cast<const uint4*>(st.k_cache + at));
                    vpre[u] = __ldcg(reinterpret_cast<const uint4*>(st.v_cache + at));
                }
            }
        }
        auto patch = [&](uint32_t g0, const uint4 (&rows)[kFreshPer], const uint2* src, unsigned long long (&raw)[kLLPer]) {
            if (LL) {
#pragma unroll
                for (int u = 0; u < kLLPer; ++u) {
                    const int e = gt + u * 128;
                    if (e < hd) {
                        while (!ll_ready(raw[u], tag_in) && ll_keep_waiting(p, ll_spins, ll_t0, stage)) raw[u] = ll_load1(src + (size_t)kvh * hd + e);
                        int sit, off;
                        ta.locate(p.pos0 - key0, e >> 3, sit, off);
                        *reinterpret_cast<unsigned short*>(sm.ring + slot_off(g0 + sit) + off + (e & 7) * 2) = (unsigned short)raw[u];
                    }
                }
            } else {
#pragma unroll
                for (int u = 0; u < kFreshPer; ++u) {
                    const int i = gt + u * 128;
                    if (i < n_fresh * vec_per_row) {
                        const int fr = i / vec_per_row, c = i - fr * vec_per_row;
                        int sit, off;
                        ta.locate(fresh0 + fr - key0, c, sit, off);
                        *reinterpret_cast<uint4*>(sm.ring + slot_off(g0 + sit) + off) = rows[u];
                    }
                }
            }
        };

        for (int c0 = 0; c0 < n_cols; c0 += kAttnCols) {  // eight columns at a time
            const int ct = min(kAttnCols, n_cols - c0);
            if (q_kvh != kvh || n_cols > kAttnCols) {
                // queries of these columns (nobody reads the ones before any more: the group has met at a barrier behind their scores)
                if (LL) {
                    for (int i0 = gt; i0 < ct * hd; i0 += 2 * 128) {
                        unsigned long long raw[2] = {};
                        const uint2* src = p.ql + (size_t)(kvh * group + c0) * hd;
#pragma unroll
                        for (int u = 0; u < 2; ++u)
                            if (i0 + u * 128 < ct * hd) raw[u] = ll_load1(src + i0 + u * 128);
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const int i = i0 + u * 128;
                            if (i < ct * hd) {
                                while (!ll_ready(raw[u], tag_in) && ll_keep_waiting(p, ll_spins, ll_t0, stage)) raw[u] = ll_load1(src + i);
                                const int c = i / hd;
                                *reinterpret_cast<unsigned short*>(qs + c * q_row + (i - c * hd) * 2) = (unsigned short)raw[u];
                            }
                        }
                    }
                } else {
                    for (int i = gt; i < ct * vec_per_row; i += 128) {
                        const int c = i / vec_per_row, v = i - c * vec_per_row;
                        const int g = (c0 + c) / M, m = (c0 + c) - g * M;
                        *reinterpret_cast<uint4*>(qs + c * q_row + v * 16) =
                            __ldcg(reinterpret_cast<const uint4*>(p.q + (size_t)m * p.d_model + (size_t)(kvh * group + g) * hd) + v);
                    }
                }
            }
            if (c0 == 0) {
                wait_tile(gk, M * 1000 + j);
                if (has_fresh) patch(gk, kpre, p.kl, kraw);
            }
            bar_sync(bar_id, 128);  // queries and patched keys are there
            if (j == 0 && c0 == 0) trace_mark(p, stage, 2);  // attention timeline: 2 = inputs staged, 4 = softmax done, 5 = P V done, 6 = value tile released, 7 = merged

            // ---- scores: keys 32 gwarp + 16 t + {g8, 8 + (g8 ^ 4)} of columns 2 q4, 2 q4 + 1 to a lane
            float s[2][4] = {};
            {
                float s_odd[2][4] = {};  // (heads of 256: boxes 1 and 3, or 0 and 2 where s has those)
                const uint32_t q_addr = smem_u32(qs) + min(mi, ct - 1) * q_row + mat * 16;
                const uint32_t k_row = (uint32_t)(((gwarp & 1) * 32 + k_key) * ta.row_bytes);
                const uint32_t tile0 = gk + (uint32_t)((gwarp >> 1) * nhb);
#pragma unroll 1  // (unrolled, here and in P V: five rows on 8000 keys 546 -> 559 us, the instruction caches)
                for (int hb = 0; hb < nhb; ++hb) {
                    const uint32_t k_addr = ring_addr + slot_off(tile0 + hb) + k_row;
                    float box[2][4];
#pragma unroll
                    for (int ks = 0; ks < 4; ks += 2) {  // two steps of 16 dimensions
                        if (!HD && ks * 16 >= hd) break;
                        uint32_t q[4];
                        ldmatrix4(q, q_addr + (uint32_t)((hb * 4 + ks) * 32));
#pragma unroll
                        for (int t = 0; t < 2; ++t) {
                            uint32_t a[4];
                            float d[4];
                            ldmatrix4(a, k_addr + (uint32_t)(t * 16 * ta.row_bytes) + (uint32_t)(((ks * 2 + (mat >> 1)) ^ k_swz) << 4));
                            mma_bf16_zero(d, a, q[0], q[1]);
                            if (HD <= 64) {
#pragma unroll
                                for (int e = 0; e < 4; ++e) s[t][e] += d[e];
                            }
                            if (HD || (ks + 1) * 16 < hd) {
                                float d2[4];
                                ldmatrix4(a, k_addr + (uint32_t)(t * 16 * ta.row_bytes) + (uint32_t)(((ks * 2 + 2 + (mat >> 1)) ^ k_swz) << 4));
                                mma_bf16_zero(d2, a, q[2], q[3]);
#pragma unroll
                                for (int e = 0; e < 4; ++e) {
                                    if (HD <= 64) {
                                        s[t][e] += d2[e];
                                    } else if (ks == 0) {
                                        box[t][e] = d[e] + d2[e];
                                    } else {
                                        const float sum = s[t][e] + (box[t][e] + (d[e] + d2[e]));
                                        if (HD == 256) s[t][e] = s_odd[t][e], s_odd[t][e] = sum;
                                        else s[t][e] = sum;
                                    }
                                }
                            }
                        }
                    }
                }
                if (HD == 256) {
#pragma unroll
                    for (int t = 0; t < 2; ++t)
#pragma unroll
                        for (int e = 0; e < 4; ++e) s[t][e] += s_odd[t][e];
                }
            }
            // ---- softmax statistics of the chunk; the row at position pos0 + m sees keys <= pos0 + m
            const int my_key = key0 + gwarp * 32 + g8, other = 8 + (g8 ^ 4) - g8;
            float mx[2] = {-INFINITY, -INFINITY}, sum[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int pos = p.pos0 + (c0 + 2 * q4 + e) % M;
#pragma unroll
                for (int t = 0; t < 2; ++t)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        float& v = s[t][e + 2 * h];
                        v = my_key + t * 16 + h * other <= pos ? v : -INFINITY;
                        mx[e] = fmaxf(mx[e], v);
                    }
#pragma unroll
                for (int o = 4; o < 32; o *= 2) mx[e] = fmaxf(mx[e], __shfl_xor_sync(0xffffffffu, mx[e], o));
            }
            if (glane < 4) *reinterpret_cast<float2*>(red + gwarp * kAttnCols + 2 * q4) = make_float2(mx[0], mx[1]);
            bar_sync(bar_id, 128);
            if (c0 + kAttnCols >= n_cols) release_tile(gk);  // K tile no longer needed: hand its slots back to the producer
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                const float2 r = *reinterpret_cast<const float2*>(red + w * kAttnCols + 2 * q4);
                mx[0] = fmaxf(mx[0], r.x), mx[1] = fmaxf(mx[1], r.y);
            }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                sum[e] = 0.f;
                if (e >= ct) break;  // a single column
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float& v = s[i >> 1][e + 2 * (i & 1)];
                    v = v == -INFINITY ? 0.f : expf((v - mx[e]) * p.attn_scale);
                }
                sum[e] = (s[0][e] + s[0][e + 2]) + (s[1][e] + s[1][e + 2]);
                if (2 * q4 + e < ct) {
                    unsigned char* dst = ps + (2 * q4 + e) * kAttnPRow + (gwarp * 32 + 2 * g8) * 2;
#pragma unroll
                    for (int t = 0; t < 2; ++t) {
                        float a = s[t][e], b = s[t][e + 2];
#pragma unroll
                        for (int term = 0; term < 3; ++term) {
                            const uint32_t w = __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);  // the upper halves
                            *reinterpret_cast<uint32_t*>(dst + term * ct_max * kAttnPRow + t * 32) = w;
                            a -= bf_lo(w), b -= bf_hi(w);  // exact
                        }
                    }
                }
#pragma unroll
                for (int o = 4; o < 32; o *= 2) sum[e] += __shfl_xor_sync(0xffffffffu, sum[e], o);
            }
            if (glane < 4) *reinterpret_cast<float2*>(red + 4 * kAttnCols + gwarp * kAttnCols + 2 * q4) = make_float2(sum[0], sum[1]);
            const int n_steps = (n_valid + 15) >> 4;  // blocks of 16 keys
            if (c0 == 0) {  // V tile: wait and patch once per item
                wait_tile(gv, M * 1000 + 500 + j);
                if (has_fresh) patch(gv, vpre, p.vl, vraw);
                // the probabilities behind the last key are zero, and so are the values that they meet
                for (int i = gt; i < (n_steps * 16 - n_valid) * vec_per_row; i += 128) {
                    const int fr = i / vec_per_row, c = i - fr * vec_per_row;
                    int sit, off;
                    ta.locate(n_valid + fr, c, sit, off);
                    *reinterpret_cast<uint4*>(sm.ring + slot_off(gv + sit) + off) = make_uint4(0u, 0u, 0u, 0u);
                }
            }
            bar_sync(bar_id, 128);
            if (gt < ct) {
                const float m = fmaxf(fmaxf(red[gt], red[kAttnCols + gt]), fmaxf(red[2 * kAttnCols + gt], red[3 * kAttnCols + gt]));
                const float* r = red + 4 * kAttnCols + gt;
                const float l = ((r[0] + r[kAttnCols]) + r[2 * kAttnCols]) + r[3 * kAttnCols];
                const int g = (c0 + gt) / M, row = (c0 + gt) - g * M;
                const size_t at = (size_t)(kvh * group + g) * p.chunk_stride + chunk;
                if (LL) ll_store(p.pl_ml + at * 2, __float_as_uint(m), tag_out), ll_store(p.pl_ml + at * 2 + 1, __float_as_uint(l), tag_out);
                else *reinterpret_cast<float2*>(p.part_ml + (at * kPassMaxRows + row) * 2) = make_float2(m, l);
            }
            if (j == 0 && c0 == 0) trace_mark(p, stage, 4);
            // ---- P V: dimensions 16 mt + {g8, g8 + 8} of columns 2 q4, 2 q4 + 1 to a lane, two such blocks side by side from 128 dimensions on.
            //      One or two columns: the terms are columns of one product. Either way the sums of a term over the blocks of 16 keys are added
            //      in order, then hi + (mid + lo).
            constexpr int kBlocks = HD >= 64 ? HD / 64 : 1;  // of a warp
            auto products = [&](auto packed) {
                constexpr bool kPacked = decltype(packed)::value;
                constexpr int kTiles = kBlocks == 1 || M <= 2 ? 1 : 2;  // (one and two rows: their registers)
                constexpr int kTerms = kPacked ? 1 : 3;
                const uint32_t p_addr = smem_u32(ps) + min(mi, (kPacked ? 3 : 1) * ct - 1) * kAttnPRow + mat * 16;
#pragma unroll 1
                for (int mt0 = gwarp * kBlocks; mt0 < (gwarp + 1) * kBlocks && mt0 * 16 < hd; mt0 += kTiles) {
                    uint32_t v_addr[kTiles];
#pragma unroll
                    for (int w = 0; w < kTiles; ++w) {
                        const int c = (mt0 + w) * 2 + (mat & 1);  // 16-byte chunk of the head
                        v_addr[w] = ring_addr + (uint32_t)(v_key * ta.row_bytes) + (uint32_t)(((nhb > 1 ? c & 7 : c) ^ v_swz) << 4);
                    }
                    const int hb = nhb > 1 ? mt0 >> 2 : 0;  // (both blocks lie in one box)
                    float acc[kTiles][kTerms][4] = {};
#pragma unroll 1
                    for (int kk = 0; kk < kAttnChunk / 16; kk += 2) {
                        if (kk >= n_steps) break;
                        uint32_t b[kTerms][4];
#pragma unroll
                        for (int term = 0; term < kTerms; ++term) ldmatrix4(b[term], p_addr + (uint32_t)(term * ct_max * kAttnPRow + kk * 32));
                        const uint32_t box = slot_off(gv + (uint32_t)((kk >> 2) * nhb + hb)) + (uint32_t)((kk & 3) * 16 * ta.row_bytes);
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            if (kk + u >= n_steps) break;
#pragma unroll
                            for (int w = 0; w < kTiles; ++w) {
                                uint32_t a[4];
                                ldmatrix4_trans(a, v_addr[w] + box + (uint32_t)(u * 16 * ta.row_bytes));
#pragma unroll
                                for (int term = 0; term < kTerms; ++term) {
                                    float d[4];
                                    mma_bf16_zero(d, a, b[term][2 * u], b[term][2 * u + 1]);
#pragma unroll
                                    for (int e = 0; e < 4; ++e) acc[w][term][e] += d[e];
                                }
                            }
                        }
                    }
#pragma unroll
                    for (int w = 0; w < kTiles; ++w)
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int col = 2 * q4 + (e & 1), dim = (mt0 + w) * 16 + g8 + (e >> 1) * 8;
                            float o;
                            if constexpr (kPacked) {  // the terms of a column are 1 or 2 columns apart
                                const float next = __shfl_down_sync(0xffffffffu, acc[w][0][e], 1), after = __shfl_down_sync(0xffffffffu, acc[w][0][e], 2);
                                o = ct == 1 ? acc[w][0][e] + (acc[w][0][e | 1] + next) : acc[w][0][e] + (next + after);
                            } else {
                                o = acc[w][0][e] + (acc[w][1][e] + acc[w][2][e]);
                            }
                            if (col < ct) {
                                const int g = (c0 + col) / M, m = (c0 + col) - g * M;
                                const size_t at = (size_t)(kvh * group + g) * p.chunk_stride + chunk;
                                if (LL) ll_store(p.pl_acc + at * hd + dim, __float_as_uint(o), tag_out);
                                else p.part_acc[(at * kPassMaxRows + m) * hd + dim] = o;
                            }
                        }
                }
            };
            if (M <= 2 && n_cols <= 2) products(std::true_type{});
            else products(std::false_type{});
        }
        q_kvh = kvh;
        if (j == 0) trace_mark(p, stage, 5);
        // the first warp hands the value tile back when all four have read it
        if (gwarp == 0) {
            bar_sync(kAttnDoneBar + grp, 128);
            release_tile(gv);
        } else {
            bar_arrive(kAttnDoneBar + grp, 128);
        }
        if (j == 0) trace_mark(p, stage, 6);
    }
}

// Merging the chunks of a head, 32 output dimensions and one row at a time: `unit` of n_heads * rows * parts. A lane has four dimensions of every
// fourth chunk (with one dimension of every chunk the chain of additions and shuffles was four times as long).
struct MergeUnit {
    int head, m, e, sub;
    bool act;
    __device__ __forceinline__ MergeUnit(int unit, int rows, int hd) {
        const int parts = (hd + 31) >> 5, lane = threadIdx.x & 31;
        const int hm = unit / parts;
        head = hm / rows, m = hm - head * rows, e = (unit - hm * parts) * 32 + (lane & 7) * 4, sub = lane >> 3;
        act = e < hd;
    }
};
// The running maximum, sum of weights and sums of a merge. 32 chunks come in at a time: lane i works out the weight exp(m_i - maximum) of
// chunk i, every lane adds the partial results of its chunks in ascending order, and the four lanes of a dimension are added in the end. The
// same arithmetic in every instantiation.
struct Merge {
    float mx = -INFINITY, l = 0.f, w;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    // ml: (maximum before scaling, sum of weights) of this lane's chunk, -inf past the last one
    __device__ __forceinline__ void begin(float2 ml, float scale) {
        const float m = fmaxf(mx, warp_max(ml.x)), s = expf((mx - m) * scale);
        mx = m, w = expf((ml.x - m) * scale);
        l = __fmaf_rn(l, s, warp_sum(__fmul_rn(w, ml.y)));
        acc = make_float4(__fmul_rn(acc.x, s), __fmul_rn(acc.y, s), __fmul_rn(acc.z, s), __fmul_rn(acc.w, s));
    }
    __device__ __forceinline__ void add(int i, const float4& v) {  // chunk i of the 32 (another one for every lane >> 3)
        const float f = __shfl_sync(0xffffffffu, w, i);
        acc = make_float4(__fmaf_rn(f, v.x, acc.x), __fmaf_rn(f, v.y, acc.y), __fmaf_rn(f, v.z, acc.z), __fmaf_rn(f, v.w, acc.w));
    }
    // the four dimensions as two words of two bf16, in every lane
    __device__ __forceinline__ uint2 result() const {
        auto of = [&](float v) {
            v += __shfl_xor_sync(0xffffffffu, v, 8);
            v += __shfl_xor_sync(0xffffffffu, v, 16);
            return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(__fdiv_rn(v, l)));
        };
        const uint32_t a = of(acc.x), b = of(acc.y), c = of(acc.z), d = of(acc.w);
        return make_uint2(a | (b << 16), c | (d << 16));
    }
};

// Tagged handoff: the warps without attention items merge. They ask for the chunks' (maximum, sum of weights) until the tags are
// this stage's, then for the sums of 16 chunks at a time. Nobody who produces a partial result ever waits for a merge, so the
// wait ends. The chunks before the last one are merged while that one is still being worked on: at 512 positions of the 7B shape the
// stage is 4.9 us, 1.0 of it behind the last item. (A group that merged the heads whose last chunk it had took 2-3 us there, and 11 at 65 chunks.)
__device__ __forceinline__ void merge_tagged(const PassParams& p, int stage, int n_chunks, int warp0, int n_warps) {
    const int lane = threadIdx.x & 31, hd = p.head_dim, warp = (threadIdx.x >> 5) - warp0;
    const uint32_t tag_out = p.pass_tag + (uint32_t)stage;
    const int units = p.n_heads * ((hd + 31) >> 5);
    unsigned spins = 0;
    long long t0 = 0;
    for (int u = blockIdx.x + warp * gridDim.x; u < units; u += n_warps * gridDim.x) {
        const MergeUnit mu(u, 1, hd);
        const size_t chunk0 = (size_t)mu.head * p.chunk_stride;
        Merge mg;
#pragma unroll 1
        for (int c0 = 0; c0 < n_chunks; c0 += 32) {
            unsigned long long rm = 0, rl = 0;
            bool stale_ml = c0 + lane < n_chunks;
            for (;;) {
                if (stale_ml) {
                    ll_load2(p.pl_ml + (chunk0 + c0 + lane) * 2, rm, rl);
                    stale_ml = !(ll_ready(rm, tag_out) && ll_ready(rl, tag_out));
                }
                if (!__any_sync(0xffffffffu, stale_ml)) break;
                if (!__all_sync(0xffffffffu, ll_keep_waiting(p, spins, t0, stage))) break;
                __nanosleep(100u);
            }
            mg.begin(c0 + lane < n_chunks ? make_float2(__uint_as_float((uint32_t)rm), __uint_as_float((uint32_t)rl)) : make_float2(-INFINITY, 0.f), p.attn_scale);
#pragma unroll 1
            for (int c1 = 0; c1 < 32 && c0 + c1 < n_chunks; c1 += 16) {
                unsigned long long ra[4][4] = {};
                unsigned stale = 0u;
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (mu.act && c0 + c1 + 4 * i + mu.sub < n_chunks) stale |= 1u << i;
                for (;;) {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (stale & (1u << i)) {
                            const uint2* src = p.pl_acc + (chunk0 + c0 + c1 + 4 * i + mu.sub) * hd + mu.e;
                            ll_load2(src, ra[i][0], ra[i][1]);
                            ll_load2(src + 2, ra[i][2], ra[i][3]);
                        }
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if ((stale & (1u << i)) && ll_ready(ra[i][0], tag_out) && ll_ready(ra[i][1], tag_out) && ll_ready(ra[i][2], tag_out) && ll_ready(ra[i][3], tag_out))
                            stale &= ~(1u << i);
                    if (!__any_sync(0xffffffffu, stale != 0u)) break;
                    if (!__all_sync(0xffffffffu, ll_keep_waiting(p, spins, t0, stage))) break;
                    __nanosleep(100u);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)  // (chunks past the last one weigh nothing)
                    mg.add(c1 + 4 * i + mu.sub, make_float4(__uint_as_float((uint32_t)ra[i][0]), __uint_as_float((uint32_t)ra[i][1]), __uint_as_float((uint32_t)ra[i][2]),
                                                            __uint_as_float((uint32_t)ra[i][3])));
            }
        }
        const uint2 out = mg.result();
        if (mu.act && mu.sub < 2) ll_store(p.al + (((size_t)mu.head * hd + mu.e) >> 1) + mu.sub, mu.sub ? out.y : out.x, tag_out);
    }
}

// Without tags: behind a grid barrier of its own the heads and rows are dealt to all warps of the grid: 3.3 us behind the last item at 512
// positions of the 7B shape, barriers included, of a stage of 9.2 with five rows. (Merged by the group whose report completes a head, on 32 of
// the 148 CTAs with a chain of 18 trips to L2 in each, five rows took 4 us at five chunks and 29 at 65.)
template <int M>
__device__ __forceinline__ void merge_all(const PassParams& p) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, hd = p.head_dim;
    const int units = p.n_heads * M * ((hd + 31) >> 5);
#pragma unroll 1
    for (int u = blockIdx.x + warp * gridDim.x; u < units; u += kPassConsumerWarps * gridDim.x) {
        const MergeUnit mu(u, M, hd);
        const int nc = (p.pos0 + mu.m) / kAttnChunk + 1;
        const size_t row0 = (size_t)mu.head * p.chunk_stride * kPassMaxRows + mu.m;
        const float* src = p.part_acc + (row0 + (size_t)mu.sub * kPassMaxRows) * hd + (mu.act ? mu.e : 0);
        Merge mg;
#pragma unroll 1
        for (int c0 = 0; c0 < nc; c0 += 32) {
            const float2 ml = c0 + lane < nc ? __ldcg(reinterpret_cast<const float2*>(p.part_ml + (row0 + (size_t)(c0 + lane) * kPassMaxRows) * 2))
                                             : make_float2(-INFINITY, 0.f);
            float4 pa[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                pa[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (c0 + 4 * i + mu.sub < nc) pa[i] = __ldcg(reinterpret_cast<const float4*>(src + (size_t)(c0 + 4 * i) * kPassMaxRows * hd));
            }
            mg.begin(ml, p.attn_scale);
#pragma unroll
            for (int i = 0; i < 8; ++i) mg.add(4 * i + mu.sub, pa[i]);  // (chunks past the last one weigh nothing)
        }
        const uint2 out = mg.result();
        if (mu.act && mu.sub == 0) *reinterpret_cast<uint2*>(p.a + (size_t)mu.m * p.d_model + (size_t)mu.head * hd + mu.e) = out;
    }
}

template <int M, bool LL, int HD>
__device__ void attn_stage(const PassParams& p, const StageDesc& st, const PassSmem& sm, uint32_t& gi, unsigned& merge_target, int stage) {
    const int warp = threadIdx.x >> 5;
    int n_chunks, first;
    const int n_local = attn_local_items(p, M, n_chunks, first);
    const uint32_t gi0 = gi;
    gi += (uint32_t)(n_local * 2 * (kAttnChunk / kBoxKeys) * (p.head_dim > 64 ? p.head_dim / 64 : 1));
    if (LL) trace_mark(p, stage, 1);  // tagged handoff: every item waits for exactly the words it needs
    else stage_begin(p, stage);      // all consumer warps, also those without attention work
    const int item_warps = 4 * p.attn_groups;
    if (warp < item_warps) {
        attn_items<M, LL, HD>(p, st, sm, gi0, stage, n_chunks, first, n_local);
    } else if (LL) {
        merge_tagged(p, stage, n_chunks, item_warps, kPassConsumerWarps - item_warps);
    }
    if (LL) consumers_sync();  // the next stage's window takes the place of the items' scratch
    if (!LL) {
        grid_arrive(p.merge_bar);
        merge_target += gridDim.x;
        grid_wait(p, p.merge_bar, merge_target);
        merge_all<M>(p);
        trace_mark(p, stage, 7);
    }
}

// ============================================================================================ the kernel
// HD: the head size that attention is compiled for, 0: any. (A kernel each: the code of a pass is larger than the instruction caches, and code in
// between that does not run costs as well.)
template <int M, bool LL, int HD>
__global__ void __launch_bounds__(kPassThreads, 1) pass_kernel(const __grid_constant__ PassParams p) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* base = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    PassSmem sm;
    sm.ring = base;
    sm.full = reinterpret_cast<uint64_t*>(base + p.off_bars);
    sm.empty = sm.full + p.ns;
    sm.red = reinterpret_cast<float*>(base + p.off_misc);
    sm.flag = reinterpret_cast<int*>(sm.red + 16 * kPassMaxRows * 4);
    sm.consumed = reinterpret_cast<volatile unsigned*>(sm.flag + 8);
    int* split = reinterpret_cast<int*>(const_cast<unsigned*>(sm.consumed) + kMaxSlots);
    sm.split = split;
    int* tok = split + 8 * 4;
    sm.tok = tok;
    unsigned short* warp_set = reinterpret_cast<unsigned short*>(tok + kPassMaxRows);
    sm.warp_set = warp_set;
    sm.psum = reinterpret_cast<float*>(base + p.off_psum);
    sm.reg_a = base + p.off_reg_a;

    if (threadIdx.x == 0) {
        for (int i = 0; i < p.ns; ++i) {
            mbar_init(&sm.full[i], 1);
            mbar_init(&sm.empty[i], 1);
            sm.consumed[i] = 0u;
        }
        mbar_fence_init();
    }
    if (threadIdx.x >= 32 && threadIdx.x < 40) {  // split table: rows of the matrix of every stage type
        const int type = threadIdx.x - 32;
        const int n_rows = type == kStQkv ? p.d_model + 2 * p.kv_dim
                         : (type == kStOproj || type == kStDown) ? p.d_model
                         : type == kStGateUp ? 2 * p.d_ffn
                         : type == kStLmHead ? p.vocab : 0;
        int pair0 = 0, np = 0;
        if (n_rows > 0) cta_pairs(n_rows, type, pair0, np);
        const int n_oct = (np + kGrpPairs - 1) / kGrpPairs;
        // fewer groups than warps: several warp sets share a group, no more of them than a row has segments (see gemv_stage; copies of the partial
        // sums that nobody wrote were zeroed and added all the same: one row of the tiny decoder 100 -> 92 us, five rows 138 -> 129)
        const int n_seg = ((type == kStDown ? p.d_ffn : p.d_model) + kSegK - 1) / kSegK;
        split[type * 4 + 0] = pair0, split[type * 4 + 1] = np, split[type * 4 + 2] = n_oct;
        split[type * 4 + 3] = (n_oct > 0 && n_oct < 8) ? max(1, min(kPassConsumerWarps / n_oct, n_seg)) : 1;
        const int S = split[type * 4 + 3];
        for (int w = 0; w < kPassConsumerWarps; ++w) {  // S > 1: exactly one group per warp
            const int ks = S > 1 ? w / n_oct : 0;
            warp_set[type * 16 + w] = (unsigned short)(ks | (S > 1 ? (ks < S ? w - ks * n_oct : n_oct) : w) << 8);
        }
    }
    if (threadIdx.x >= 64 && threadIdx.x < 64 + M && p.stages[0].type == kStEmbed) {
        const int m = threadIdx.x - 64;
        tok[m] = min(max(pass_token(p, m), 0), p.vocab - 1);
    }
    __syncthreads();

    if (threadIdx.x >= kPassConsumers) {
        pass_producer<M>(p, sm);
        if constexpr (kFewRows<M>) finish_rows<M>(p);
        return;
    }

    uint32_t gi = 0;
    unsigned merge_target = p.merge_base;
    if (p.trace && threadIdx.x == 0) {  // which SM runs this CTA (entry 4 of the embedding stage, which streams nothing)
        unsigned smid;
        asm volatile("mov.u32 %0, %smid;" : "=r"(smid));
        p.trace[((size_t)0 * kTraceEntries + 4) * gridDim.x + blockIdx.x] = smid;
    }
    for (int s = 0; s < p.n_stages; ++s) {
        trace_mark(p, s, 0);
        const StageDesc st = p.stages[s];  // static: read before waiting for the previous stage
        // the next descriptor is requested now so that reading it at the next stage boundary hits L1
        if (threadIdx.x < 2 && s + 1 < p.n_stages)
            asm volatile("prefetch.global.L1 [%0];" ::"l"(reinterpret_cast<const char*>(p.stages + s + 1) + threadIdx.x * 64));
        if (p.trace && threadIdx.x == 0) p.trace[((size_t)s * kTraceEntries + 11) * gridDim.x + blockIdx.x] = st.type >= 0 ? global_ns() : 0;  // descriptor read
        if (st.type == kStEmbed) {
            trace_mark(p, s, 1);  // (nothing to wait for)
            const int d = p.d_model;
            if (kFewRows<M> && p.embed_direct) {
                // The first RMSNorm reads the embeddings itself; what the residual stages will want of them, the CTA's own rows, it leaves here
                // for itself, and nobody waits for anybody. (A stage that spread the embeddings over the CTAs cost a hand-off; without it and with
                // the cosines beside the LM head one row of the 7B width, four layers, took 329.8 us for 332.7, two rows of the tiny decoder 121 for 124.)
                const int row0 = 2 * split[kStOproj * 4 + 0], n = min(2 * split[kStOproj * 4 + 1], d - row0);
                for (int i = threadIdx.x; i < M * n; i += kPassConsumers) {
                    const int m = i / n, e = row0 + i - m * n;
                    const float v = __bfloat162float(p.embed[(size_t)tok[m] * d + e]);
                    if (LL) ll_store(p.xl + (size_t)m * d + e, __float_as_uint(v), p.pass_tag);
                    else p.x[(size_t)m * d + e] = v;
                }
            } else {
                for (int i = blockIdx.x * kPassConsumers + threadIdx.x; i < M * d; i += gridDim.x * kPassConsumers) {
                    const int m = i / d, e = i - m * d;
                    p.x[i] = __bfloat162float(p.embed[(size_t)tok[m] * d + e]);
                }
            }
        } else if (st.type == kStFinish) {
            // The LM head wants the hidden state of all CTAs. The cosines of one and two rows are the producer warp's work (finish_rows), those of
            // more rows the consumer warps'. (The test hook's wait is this one: the arrivals behind it would end the producer's.)
            if (!LL) stage_begin(p, s, p.bar_extra_last);
            else trace_mark(p, s, 1);
            if constexpr (!kFewRows<M>) finish_stage<M>(p, sm);
        } else if (st.type == kStAttn) {
            attn_stage<M, LL, HD>(p, st, sm, gi, merge_target, s);
        } else {
            gemv_stage<M, LL>(p, st, sm, gi, s);
        }
        trace_mark(p, s, 3);
        if (!LL) {
            grid_arrive(p.grid_bar);
        } else if (s + 1 == p.finish_stage) {
            // Tagged handoff: only the finish stage waits at the grid barrier, so the CTA arrives once for all stages in front of it. (Nothing
            // else ends a stage with a barrier: what the next one writes first, the window and the sums of squares, nobody reads any more.)
            grid_arrive(p.grid_bar, (unsigned)(s + 1));
        }
    }
}

}  // namespace asd
