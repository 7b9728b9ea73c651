// The fused sublayer product as a launch of its own (gemv.cu).
#pragma once
#include "common.cuh"

namespace asd {

constexpr int kGemvWarps = 8;  // multiplying warps of a CTA

enum Epilogue : int { kEpiPlain = 0, kEpiSwiglu = 1, kEpiResidual = 2 };

struct GemvParams {
    const __nv_bfloat16* W;  // [n_rows, n_in]
    int M, n_rows, n_in;
    const void* x;              // gain ? float [M, n_in] : bf16 [M, n_in]
    const __nv_bfloat16* gain;  // [n_in] or null
    float eps;
    void* out;          // plain / swiglu / residual
    float* cos_out;     // residual: [M]
    float* partials;    // [gridDim.x][kMaxRows][4] cross-CTA partial results
    unsigned* counter;  // zero before launch; reset by the last CTA
    int* err;           // 8 words: the first is set while warps whose bounded wait has run out leave, the others say where
    // the plan, filled in by launch_gemv
    int cta_pairs, cta_more;          // pairs of rows: pairs / CTAs and the remainder
    unsigned div_grid, div_groups;    // for divisions by the numbers of CTAs and of groups
    int n_blk;               // blocks of rows of a CTA
    int groups, group_rows;  // groups of rows per block, and the most rows of one
    int seg, tail;           // inputs of a piece, and how many more the last one of a row may have
    int whole;               // a piece is whole rows, copied as one
    int by_warp;             // a group of rows is one warp's alone
    int win;                 // inputs whose activations are in shared memory at a time
    int xs_ld;               // bf16 per activation row there
    int pitch, stage_bytes, n_stages, off_xs, off_ring;  // the ring of weight pieces
};

cudaError_t launch_gemv(GemvParams p, int epi, bool norm, int max_smem, int sms, cudaStream_t s);
cudaError_t configure_gemv(int max_smem);

}  // namespace asd
