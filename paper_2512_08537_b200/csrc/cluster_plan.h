// How the cluster schedule (cluster.cuh) lays a head out: arithmetic alone, also for the host.
#pragma once
#include <math.h>
#include <stddef.h>
#include <stdint.h>

#ifndef ARDIFF_HD
#ifdef __CUDACC__
#define ARDIFF_HD __host__ __device__
#else
#define ARDIFF_HD
#endif
#endif

constexpr int CL_MAX_CTAS = 16;                // CTAs of a cluster
constexpr int CL_UNIT = 16;                    // tokens: the fewest that one product takes
constexpr int CL_MAX_UNITS = 4;                // units of 16 tokens in a cluster's group
constexpr int CL_MAX_STAGES = 6;               // of weights in the ring
constexpr int CL_MIN_STAGES = 2;
constexpr int CL_SMEM = 226 * 1024;            // dynamic shared memory, 1 KB of it to align the ring
constexpr int CL_THREADS = 32 * 11;            // weights, products, eight epilogue warps, activations
constexpr int CL_KS = 64;                      // K slice: one swizzle row of weights
// K slices of a stage: 32 KB of weights or a little more (36 at 96 rows), the columns of 4, 2 or 1 CTAs.
ARDIFF_HD constexpr int cl_slices(int rows) { return rows == 64 ? 4 : rows == 96 ? 3 : 2; }

// Shared memory of one CTA: the weight ring, activations (u and a share a buffer where two do not fit), x as bf16 (operand of
// the in-projection) and as fp32, LayerNorm partials of all CTAs, those of this CTA's warps.
struct ClusterLayout {
    int bufs, stages;
    uint32_t stage, act, u, a, xb, x, stats, part, total;
    ARDIFF_HD ClusterLayout(int W, int C, int rows, int units) {
        const uint32_t N = (uint32_t)units * CL_UNIT, ctas = (uint32_t)(W / rows);
        stage = (uint32_t)rows * CL_KS * 2 * cl_slices(rows);
        act = N * (uint32_t)W * 2;
        const uint32_t rest = N * 128 + N * (uint32_t)C * 4 + N * ctas * 8 + N * 32, room = CL_SMEM - 1024;
        bufs = 2 * act + rest + 3 * stage <= room ? 2 : 1;
        const uint32_t used = (uint32_t)bufs * act + rest;
        int fit = used < room ? (int)((room - used) / stage) : 0;
        stages = fit < CL_MAX_STAGES ? fit : CL_MAX_STAGES;
        u = (uint32_t)stages * stage;
        a = u + (uint32_t)(bufs - 1) * act;
        xb = a + act;
        x = xb + N * 128;
        stats = x + N * (uint32_t)C * 4;
        part = stats + N * ctas * 8;
        total = part + N * 32;
    }
};

// Heads created for at most so many tokens split a layer over as many CTAs as a cluster may have. us, 64 or 96 columns a CTA /
// 128: W = 256, 32 tokens 74 / 76, 1024 101 / 95; W = 1024, 64 tokens 168 / 174, 128 207 / 177.
constexpr int CL_FEW_TOKENS = 64;
// u (or a) of a cluster's tokens, bytes up to which the CTAs copy it to one another. us, copied / through L2: 8 KB (W = 256, 16
// tokens) 74 / 97, 32 KB (1024, 16) 168 / 190, 48 KB (1536, 16) 745 / 773, 64 KB (2048, 16) 332 / 330, 96 KB (1024, 48) 359 / 318.
constexpr uint32_t CL_DIRECT_BYTES = 48 * 1024;
// Bytes of u and of a on their way between the CTAs of the clusters, through L2.
inline size_t cluster_xch_bytes(int W, int units, int clusters) {
    return (size_t)clusters * 2 * units * CL_UNIT * W * 2;
}

// Output columns that one CTA of a cluster owns of every W-wide layer; 0: no cluster schedule for this width. Heads for few
// tokens take as many CTAs as there may be in a cluster (each streams fewer weights), others have room for more clusters.
inline int cluster_rows(int W, int64_t max_tokens) {
    const int choices[] = {64, 96, 128};
    for (int rows : choices)
        if (W % rows == 0 && W / rows <= CL_MAX_CTAS && (rows == 128 || max_tokens <= CL_FEW_TOKENS || W > 8 * 128))
            return rows;
    return 0;
}
// Most units of 16 tokens that a cluster takes at once: as many as fit, where a split can need them (64 columns a CTA are for heads
// of at most CL_FEW_TOKENS = 64 tokens, and on any device with 4 such clusters one unit each is all of them; 96 are for W = 1536).
ARDIFF_HD constexpr int cl_most_units(int rows) { return rows == 64 ? 1 : rows == 96 ? 2 : CL_MAX_UNITS; }
inline int cluster_units(int W, int C, int rows) {
    int units = cl_most_units(rows);
    while (units > 0 && ClusterLayout(W, C, rows, units).stages < CL_MIN_STAGES) --units;
    return units;
}

// Survivors up to which the clusters serve a call of K steps: one round of groups. A second round takes as long again, and
// the tile schedule hardly longer for twice the tokens (W = 1024, 3 blocks, K = 4, 700 / 1434 tokens: clusters 321 / 565 us,
// tiles 426 / 475). With few layers in all, what the modulations cost (written and read back in fp32) shows in the largest
// groups, and the round ends earlier. us, clusters / tiles, K = 1: W = 256, 3 blocks, 3848 tokens 89 / 89, 4736 106 / 94, 5
// blocks 4440 129 / 126, 4736 131 / 127; 512, 3, 1716 97 / 104, 2112 113 / 106, 4, 1716 125 / 123, 2112 134 / 125; 768, 3,
// 1408 131 / 121; 1024, 3, 691 120 / 122, 748 132 / 122, 960 143 / 130, 4, 748 159 / 155 (medians over nine heads; groups of
// 64 tokens leave the ring two stages there); K = 2: 256, 2, 3848 118 / 119, 4440 129 / 120; 512, 1, 1980 101 / 104, 2112
// 108 / 103, 2, 1848 137 / 147, 2112 149 / 144. With one or two layers both take as long (256, 2, 4736 76 / 76), with more
// layers or steps all of it gains (256, 12, 4736 210 / 233; 512, 3, K = 2, 2112 181 / 186; 512, 1, K = 4, 2112 174 / 179),
// and so do groups of up to 48 tokens (1280, 4, 528 174 / 193; 1536, 1, 224 66 / 84).
inline int64_t cluster_survivors(int W, int clusters, int units, int K, int L) {
    int sixteenths = 16;
    if (units == 4 && K == 1 && L >= 3 && L <= 6) sixteenths = L > 4 ? 15 : W == 1024 ? 12 : 13;
    if (units == 4 && K == 2 && L <= 2) sixteenths = W == 256 ? 14 : 15;
    return (int64_t)clusters * units * CL_UNIT * sixteenths / 16;
}

// Survivors up to which the chain (chain.cuh, at most 32 beside the clusters) stays the faster one: it spreads the weights
// of a layer over W / 16 SMs, a cluster over 16, and has no second launch, but loses time in every step (x goes between the
// SMs too) and with every token. The more steps and the fewer blocks in each, the fewer: a doubling of K costs 18 tokens
// with one block, 3 with 12. (Constants for the least loss over widths of 768 to 2048, 1, 3 and 12 blocks, 1 to 8 steps, 1
// to 32 tokens: none above 4 %, but 6 % at W = 1792 with one block and K = 4.) us, chain / clusters: W = 768, K = 1, 3
// blocks, 6 59 / 59, 14 60 / 59, 6 blocks, 6 82 / 82, 14 86 / 81, 12 blocks, 6 124 / 130, 10 127 / 131, 14 135 / 131
// (medians over nine heads, between which the chain's times differ by up to 10 %), K = 2, 8 212 / 206; W = 1024, 3 blocks, K
// = 1, 24 72 / 72, K = 2, 8 98 / 102, 17 101 / 103, K = 4, 1 152 / 166, 8 166 / 166, K = 8, 4 293 / 299, 8 303 / 299; 12
// blocks, K = 4, 16 485 / 490, 24 515 / 490, K = 8, 12 901 / 922; 1 block, K = 2, 4 64 / 65, 8 66 / 65; W = 1280, 3 blocks,
// K = 2, 24 124 / 124, K = 4, 12 206 / 205, 12 blocks, K = 4, 24 609 / 621; W = 1536, 3 blocks, K = 8, 16 443 / 450, 24 462
// / 450, 12 blocks, K = 8, 28 1371 / 1407; W = 2048, 1 block, K = 8, 16 276 / 317, 32 325 / 318, all else up to 32. At 512
// and below never (1 token, 12 blocks, K = 1: 112 / 97). Clusters of 64 columns a CTA are faster: W = 768, 12 blocks, K = 1,
// 4 125 / 125, 8 136 / 124; W = 1024, 3 blocks, K = 2, 8 94 / 100, 17 108 / 101, 12 blocks, K = 2, 8 246 / 260, 16 285 /
// 262, K = 8, 4 837 / 878, 12 922 / 879.
inline int chain_beside_clusters(int W, int rows, int K, int L) {
    if (W < 768 || K < 1) return 0;
    if (W < 1024) return K > 1 ? 0 : L > 6 && rows == 64 ? 4 : L < 4 ? 2 * L + 2 : 10;
    const int most = W >= 1792 ? 76 : W >= 1536 ? 38 : W >= 1280 ? 30 : rows == 64 ? 18 : 23;
    const double per_doubling = rows == 64 ? 6.0 + 10.0 / L : 2.0 + 16.0 / L;
    const int tokens = (int)(most - per_doubling * log2((double)K)), least = L > 1 ? 4 : 1;
    return tokens > 32 ? 32 : tokens < least ? least : tokens;
}

constexpr size_t CL_MODS_LIMIT = (size_t)256 << 20;      // bytes of the modulation buffer
// Survivors up to which a modulation buffer of this size serves a call of K steps.
inline int64_t mods_survivors(size_t bytes, int K, int L, int W) {
    return (int64_t)(bytes / ((size_t)K * (3 * L + 2) * W * sizeof(float))) / 8 * 8;
}
inline size_t mods_bytes(int K_max, int64_t max_tokens, int L, int W) {
    const size_t per_token = (size_t)K_max * (3 * L + 2) * W * sizeof(float);
    const size_t tokens = (size_t)(max_tokens + 7) / 8 * 8;
    return tokens < CL_MODS_LIMIT / per_token ? tokens * per_token : CL_MODS_LIMIT;
}

// Modulation values of one layer and step: tiles of 32 channels x 8 tokens as the epilogue's lanes hold them (cluster.cuh),
// 1 KB each, the tokens of 32 channels side by side. Tokens rounded up to whole tiles:
ARDIFF_HD inline int mods_stride(int S) { return (S + 7) / 8 * 8; }
