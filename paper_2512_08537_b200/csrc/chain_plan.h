// Where the chain (chain.cuh) keeps things, and how many survivors its buffers serve: arithmetic alone, also for the host.
#pragma once
#include <stddef.h>
#include <stdint.h>

#ifdef __CUDACC__
#define ARDIFF_HD __host__ __device__
#else
#define ARDIFF_HD
#endif

constexpr int CHAIN_MAX_TOKENS = 64;
constexpr int CHAIN_COLS = 16;                 // columns of a layer that one CTA owns
constexpr int CHAIN_WARPS = 8;                 // consumer warps; one more feeds the weight ring
constexpr int CHAIN_HINT_LINE = 128;           // one hint per line and K eighth
constexpr int CHAIN_HINT_BYTES = CHAIN_WARPS * CHAIN_HINT_LINE;
constexpr size_t CHAIN_BUFFER_LIMIT = (size_t)128 << 20;   // of the modulations, and of the exchange buffer

// Where things are in the exchange buffer of a call with S tokens: u, LayerNorm partials and (mean, 1 / std) per (step,
// block or final layer), a per (step, block), x per step.
// u and a are stored as the B fragments their readers load: [K chunk of 32][token tile of 8][lane][16 bytes].
// The hints come first, zeroed; everything else starts as CHAIN_EMPTY.
struct ChainLayout {
    size_t act;                                // bytes of one u or a
    size_t hints, u, a, st, fin, xb, total;    // byte offsets
    ARDIFF_HD ChainLayout(int S, int K, int L, int W, int C) {
        const size_t S8 = (size_t)(S + 7) / 8 * 8, layers = (size_t)K * (L + 1);
        act = S8 * W * 2;
        hints = 0;
        u = 2 * layers * CHAIN_HINT_BYTES;
        a = u + layers * act;
        st = a + (size_t)K * L * act;
        fin = st + layers * S8 * (W / 2);
        xb = fin + layers * S8 * 16;
        total = xb + (size_t)K * S8 * C * 2;
    }
};
// fp32 modulation values of one token and one step
inline size_t mods_floats_per_token_step(int L, int W) { return (size_t)(3 * L + 2) * W; }

// Bytes of the two buffers for calls of up to K_max steps and max_tokens survivors: what the largest such call needs, within
// the limit.
inline size_t chain_mods_bytes(int K_max, int64_t max_tokens, int L, int W) {
    const size_t tokens = (size_t)(max_tokens < CHAIN_MAX_TOKENS ? max_tokens : CHAIN_MAX_TOKENS);
    const size_t need = (size_t)K_max * tokens * mods_floats_per_token_step(L, W) * sizeof(float);
    return need < CHAIN_BUFFER_LIMIT ? need : CHAIN_BUFFER_LIMIT;
}
inline size_t chain_xch_bytes(int K_max, int64_t max_tokens, int L, int W, int C) {
    const int tokens = (int)(max_tokens < CHAIN_MAX_TOKENS ? max_tokens : CHAIN_MAX_TOKENS);
    const size_t need = ChainLayout(tokens, K_max, L, W, C).total;
    return need < CHAIN_BUFFER_LIMIT ? need : CHAIN_BUFFER_LIMIT;
}
// Survivors up to which buffers of these sizes serve a call of K steps.
inline int chain_survivors(size_t mods_bytes, size_t xch_bytes, int K, int L, int W, int C) {
    if (K < 1) return 0;
    const ChainLayout eight(8, K, L, W, C);    // 8 tokens: the hints, then a part that every further 8 tokens repeat
    const size_t per_eight = eight.total - eight.u;
    const size_t by_mods = mods_bytes / ((size_t)K * mods_floats_per_token_step(L, W) * sizeof(float));
    const size_t by_xch = xch_bytes > eight.u ? (xch_bytes - eight.u) / per_eight * 8 : 0;
    const size_t fit = by_mods < by_xch ? by_mods : by_xch;
    return (int)(fit < CHAIN_MAX_TOKENS ? fit : CHAIN_MAX_TOKENS);
}
