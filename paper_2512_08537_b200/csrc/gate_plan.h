// How the block-prefix gate deals its draft blocks to CTAs: host arithmetic alone, so that it can be checked without a GPU.
#pragma once
#include <stdint.h>

namespace ardiff {

constexpr int64_t kMaxRowsPerCta = 24576;     // row entropies of a CTA in shared memory: 96 KB

struct DraftPlan {
    int64_t blocks_per_cta;
    int64_t grid;                             // 0: the shape does not fit one pass
};

// n_blocks draft blocks of rows_per_block rows; `want` CTAs fill the GPU (the waves that the input's size asks for);
// max_blocks CTAs is what the count scratch holds.
inline DraftPlan plan_draft_blocks(int64_t n_blocks, int64_t rows_per_block, int64_t want, int64_t max_blocks) {
    if (rows_per_block > kMaxRowsPerCta) return DraftPlan{0, 0};
    if (want > max_blocks) want = max_blocks;
    // one wave of CTAs, but where a CTA would have only two or three draft blocks, one each: 512 draft blocks of
    // 128 rows as 256 CTAs left half of the warps idle (21 % occupancy)
    int64_t bpc = n_blocks <= 2 * want && n_blocks <= max_blocks ? 1 : (n_blocks + want - 1) / want;
    if (bpc * rows_per_block > kMaxRowsPerCta) bpc = kMaxRowsPerCta / rows_per_block;
    const int64_t grid = (n_blocks + bpc - 1) / bpc;
    return DraftPlan{bpc, grid <= max_blocks ? grid : 0};
}

}  // namespace ardiff
