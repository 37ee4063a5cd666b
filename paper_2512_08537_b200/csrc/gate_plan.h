// How the block-prefix gate deals its draft blocks to CTAs: host arithmetic alone, so that it can be checked without a GPU.
#pragma once
#include <stdint.h>

namespace ardiff {

constexpr int64_t kMaxRowsPerCta = 24576;     // row entropies of a CTA in shared memory: 96 KB

struct DraftPlan {
    int64_t blocks_per_cta;
    int64_t grid;                             // 0: the shape does not fit one pass
};

// n_blocks draft blocks of rows_per_block rows; the warps of a CTA take rows_per_round rows at a time; `want` CTAs fill the
// GPU (the waves that the input's size asks for); max_blocks CTAs is what the count scratch holds.
inline DraftPlan plan_draft_blocks(int64_t n_blocks, int64_t rows_per_block, int64_t rows_per_round, int64_t want,
                                   int64_t max_blocks) {
    if (rows_per_block > kMaxRowsPerCta) return DraftPlan{0, 0};
    if (want > max_blocks) want = max_blocks;
    // One wave of CTAs; but where a CTA would have two draft blocks, one each if that gives its warps two rounds of rows or
    // more: then SMs that are done early take the next draft block. With less work a CTA's start is what it costs.
    // 1024 channels (16 rows a round), one each / two each, us: 128 rows 450 draft blocks 33.6 / 34.5, 600 40.5 / 46.7, 886
    // 47.0 / 47.5; 32 rows 600 15.1 / 16.1, 886 17.1 / 16.3; 16 rows 600 11.9 / 11.3, 886 13.1 / 11.5; 8 rows 600 10.5 / 8.5,
    // 886 11.2 / 8.7. (256 channels, 64 rows a round: 32 rows 600 10.5 / 8.6, 886 11.1 / 8.9.)
    const bool alone = n_blocks <= 2 * want && n_blocks <= max_blocks && rows_per_block >= 2 * rows_per_round;
    int64_t bpc = alone ? 1 : (n_blocks + want - 1) / want;
    if (bpc * rows_per_block > kMaxRowsPerCta) bpc = kMaxRowsPerCta / rows_per_block;
    const int64_t grid = (n_blocks + bpc - 1) / bpc;
    return DraftPlan{bpc, grid <= max_blocks ? grid : 0};
}

}  // namespace ardiff
