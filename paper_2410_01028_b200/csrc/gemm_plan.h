// How a dense product of the prompt path is cut into tiles and dealt to the SMs: plain C++, shared by the kernel's launcher
// and the host code that picks tensor maps and buffers.
#pragma once
#include <algorithm>

namespace asd {

constexpr int kGemmBM = 128;  // rows of the activation tile of one CTA (the M of tcgen05.mma)
constexpr int kGemmBK = 64;   // reduction elements per pipeline stage: 128 bytes, one swizzle span

// How a product runs: tiles of 128 * cg rows x bn columns on units of cg SMs, the reduction dimension in `parts` parts. The first `wide`
// tiles of a row of tiles are bn columns, the others `narrow` (at most bn); `items` tiles in all (`tiles` if all were bn columns).
struct GemmPlan {
    int bn, cg, m_tiles, tiles, parts;
    int wide, narrow, items;
    int w_box() const { return bn / cg; }  // rows of a box of W's tensor map
};
// the heights that w_box() can have; a weight matrix has one tensor map for each
constexpr int kWBoxRows[] = {32, 64, 96, 112, 128, 160, 256};
constexpr int kWBoxes = sizeof(kWBoxRows) / sizeof(kWBoxRows[0]);

// The plan of C[M, N] = A[M, K] * W[N, K]^T on `sms` SMs. With max_parts > 1 the reduction dimension may be cut into up to that
// many parts, products of their own.
//
// The rule: the tile and the number of parts with the least time over their rounds: rounds x k-blocks of a part x the time
// of a k-block (64 elements of the reduction), plus writing and reading the further parts (8 bytes per element at about 4
// TB/s). The times of a k-block in the table are the slopes of one round of tiles; with every SM busy and several rounds all
// of them grow by about a quarter. Over 48 products of 64 to 2048 rows and 3072 to 22016 columns, each timed with all
// tiles, the rule's choice was within 0.2 % of the best on average and 5 % at worst. Pairs of SMs win where the tiles fill
// the chip for rounds, 128 columns on single SMs where one round is enough (511 x 4096 x 11008: 45.5 us against 63.7 with
// 256-column pair tiles), narrow tiles for short prompts (64 x 4096 x 11008: 33 us against 60). (A 192-column tile on
// single SMs, 316 ns, was the choice for none of 80000 products.)
inline GemmPlan plan_gemm(int M, int N, int K, int max_parts, int sms) {
    const int num_kb = (K + kGemmBK - 1) / kGemmBK;
    long long best_ns = -1;
    GemmPlan best{};
    auto consider = [&](int bn, int cg, int ns_kb) {
        GemmPlan p{};
        p.bn = bn, p.cg = cg;
        p.m_tiles = (M + kGemmBM * cg - 1) / (kGemmBM * cg);
        p.tiles = p.m_tiles * ((N + bn - 1) / bn);
        const int units = sms / cg;
        for (p.parts = 1; p.parts == 1 || (p.parts <= max_parts && num_kb / p.parts >= 8); ++p.parts) {
            const long long rounds = ((long long)p.tiles * p.parts + units - 1) / units;
            const long long ns = rounds * ((num_kb + p.parts - 1) / p.parts) * ns_kb + (long long)(p.parts - 1) * M * N / 500;
            if (best_ns < 0 || ns < best_ns) best_ns = ns, best = p;
        }
    };
    consider(256, 2, 315);
    consider(224, 2, 281);
    consider(192, 2, 247);
    consider(256, 1, 354);
    consider(160, 1, 244);
    consider(128, 1, 209);
    consider(96, 1, 195);
    consider(64, 1, 145);
    consider(32, 1, 138);
    // Pair tiles over several rounds: the units of the last rounds have columns to spare, so tiles there are narrower, as narrow as
    // still cover the product in these rounds. A tile of bn - 32 columns takes 34 ns less for each 64 elements of the reduction, but no tile less than
    // its operands' way from L2, and the copies fetch bn columns of W either way: bn - 64 at least.
    // Only where rows of A and W are whole multiples of 64 bytes and rows of C of 32: otherwise the copies (a memory sector more for every 128 bytes
    // and tile) or the stores (word by word) are what bounds a round, and more tiles or a shorter one behind a longer epilogue do not pay. With narrow
    // tiles against without, in turn, 192 products of 33 to 2048 rows and 1024 to 22016 columns for each kind, K from 1024 on: K % 32 == 0 and N % 8
    // == 0 2.8-2.9 % faster on average and none slower; K an odd multiple of 8 0.4 % slower (one in four more than 1 %, 6 % at worst), of 16 1.8 %
    // faster (1.4 % slower at worst); N odd 1.2 % faster (one in nine more than 1 % slower, 3.3 % at worst). (A product against itself: 0.5 %.)
    best.wide = best.tiles / best.m_tiles, best.narrow = best.bn, best.items = best.tiles;
    if (best.cg == 2 && best.parts == 1 && K % 32 == 0 && N % 8 == 0) {
        const int units = sms / 2, rounds = (best.tiles + units - 1) / units;
        const int cols = (int)((long long)rounds * units / best.m_tiles);  // tiles of a row of tiles that these rounds hold
        int saved = 0;
        for (int last = 1; last <= rounds; ++last) {  // narrow tiles in the last ones
            const int wide = (int)((long long)(rounds - last) * units / best.m_tiles), left = N - wide * best.bn;
            if (left <= 0 || cols <= wide) continue;
            const int narrow = std::max(((left + cols - wide - 1) / (cols - wide) + 31) / 32 * 32, best.bn - 64);
            if (narrow < best.bn && last * (best.bn - narrow) > saved) {
                saved = last * (best.bn - narrow);
                best.wide = wide, best.narrow = narrow, best.items = (wide + (left + narrow - 1) / narrow) * best.m_tiles;
            }
        }
    }
    return best;
}

}  // namespace asd
