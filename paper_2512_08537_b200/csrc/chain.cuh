// The head's chain of dependent layers for calls of few tokens: at most 32 beside the clusters of cluster.cuh, of heads 768 and
// more wide, where it is the faster one (chain_beside_clusters); up to CHAIN_MAX_TOKENS at any width, in two passes, on a device
// that takes no clusters of this size. (Without the second pass, which a whole B200 never runs, the compiler's code for the
// first is slower: W = 1536, 12 blocks, 28 tokens 728 -> 773 us, W = 1024, one token 153 -> 165.)
//
// With few tokens the head is K * (3 L + 3) exchanges between SMs in a row, and a call takes as long as they do: the tile
// schedule spends 5 to 12 us on each (TMA round trip, K loop, epilogue, store completion, release, poll). There it
// therefore only makes what does not depend on the residual stream (conditioning, s_k, all modulations of all steps,
// read from the weights once); after a grid barrier this code runs the chain with as little as possible in each exchange:
//   - CTA i owns 16 columns of every W-wide layer for the whole call; its piece of h never leaves registers.
//   - The 16 x W weight tiles of the coming layers stream into a shared-memory ring (they depend on nothing).
//   - A value is its own flag: exchange buffers start as all ones (no bf16 pair or fp32 number that is stored can be
//     that, NaN results are canonical) and are written once; readers check the words themselves, with relaxed loads, so
//     no exchange needs a fence. Counters (hints, not ordered with the data) say when looking is worthwhile: all CTAs
//     spinning on the data itself made their reads queue before the writes they waited for.
//   - Products are mma.sync m16n8k16: 16 weight rows x 8 tokens, the 8 warps split K, partials meet in shared memory.
//     (tcgen05 would add a TMA and a tensor-memory round trip to every exchange; the arithmetic is not what bounds.)
// It is a part of head_kernel, not a launch of its own: a cooperative kernel that only finds out that it has nothing to do
// cost every larger call 13 us.
// What bounds it: latency. An exchange takes 2 K cycles at W = 256 (16 CTAs) and 5 K at W = 1536 (96 CTAs), of which the
// reads of all S x W activations by every CTA are 2 K at 32 tokens; a second pass of 32 tokens costs another 3 us there.
// Whole calls with the tile schedule and with the chain, us, K = 4: W = 256, L = 2, 33 tokens 164 / 127; W = 1024, L = 3,
// 32 tokens 345 / 179, 64 tokens 346 / 244, 128 tokens 346 / 419; W = 1536, L = 12, 8 / 29 / 64 tokens 1658 / 594, 1702 /
// 681, 1702 / 958, 128 tokens about even: hence the limit of 64. Not kept: CTAs that start their reads at different
// pieces (spills; 681 -> 800), two or one token tiles of 8 loaded at once instead of four (712, 803), LayerNorm partials
// read by every CTA instead of one warp per token (10 K cycles an exchange instead of 5 K).
#pragma once

constexpr int CHAIN_MAX_NC = 8;                // W / 256
constexpr int CHAIN_GROUPS = CHAIN_MAX_TOKENS / 32;
__host__ __device__ constexpr int chain_token_tiles(int nc) { return nc <= 2 ? 8 : 4; }   // of 8, in a pass
__host__ __device__ constexpr int chain_red_bytes(int nc) {
    return CHAIN_WARPS * CHAIN_COLS * (8 * chain_token_tiles(nc) + 1) * 4;
}
constexpr int CHAIN_MAX_SLOTS = 8;
constexpr uint32_t CHAIN_EMPTY = 0xffffffffu;

struct ChainParams {
    int C, W, L, K, n_slots;
    size_t out_row0;                           // Wout in the packed weights
    const int* idx;
    const bf16 *Wcat, *Win;
    const float *bias_cat, *bin, *noise, *step_noise, *mods;
    long long step_stride;
    float* out;
    uint8_t* xch;
    int *status, *abort_flag;
    unsigned long long wait_limit_ns;
    float ax[KMAX], av[KMAX], an[KMAX];
};

// modulation values of step k: [block][shift, scale, gate][token][W], then the final layer's [shift, scale][token][W]
__host__ __device__ __forceinline__ size_t mods_index(int S, int L, int W, int k, int block, int which) {
    return ((size_t)k * (3 * L + 2) + 3 * block + which) * (size_t)S * W;
}

__device__ __forceinline__ uint4 ld_relaxed_u4(const void* p) {
    uint4 v;
    asm volatile("ld.relaxed.gpu.global.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void publish_u32(void* p, uint32_t v) {
    if (v == CHAIN_EMPTY) v = 0x7fffffffu;
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void publish_f2(void* p, float2 f) {
    uint32_t a = __float_as_uint(f.x), b = __float_as_uint(f.y);
    if (a == CHAIN_EMPTY) a = 0x7fffffffu;
    if (b == CHAIN_EMPTY) b = 0x7fffffffu;
    asm volatile("st.relaxed.gpu.global.v2.u32 [%0], {%1,%2};" ::"l"(p), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ bool chain_missing(const uint4& v) {
    return max(max(v.x, v.y), max(v.z, v.w)) == CHAIN_EMPTY;
}
__device__ __forceinline__ void mma_bf16_16x8x16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                                 uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// A bound on every wait of a thread: after an abort all further waits return at once, the kernel runs to its end on
// whatever it has and the call is reported as timed out.
struct ChainWait {
    const ChainParams& P;
    volatile int* s_abort;
    uint64_t t0 = 0;
    uint32_t it = 0;
    __device__ __forceinline__ ChainWait(const ChainParams& p, volatile int* f) : P(p), s_abort(f) {}
    __device__ __forceinline__ bool give_up() {
        if ((++it & 31u) != 0) return false;
        if (*s_abort) return true;
        const uint64_t now = ptx::globaltimer_ns();
        if (t0 == 0) t0 = now;
        bool stop = ptx::ld_relaxed_gpu(P.abort_flag) != 0;
        if (!stop && now - t0 > P.wait_limit_ns) {
            atomicExch(P.abort_flag, 1);
            atomicCAS(P.status, 0, ARDIFF_ERR_TIMEOUT);
            stop = true;
        }
        if (stop) *s_abort = 1;
        return stop;
    }
    __device__ __forceinline__ void begin() { t0 = 0; it = 0; }
    __device__ __forceinline__ void mbar(uint32_t bar, uint32_t parity) {
        begin();
        while (!ptx::mbar_try_wait(bar, parity))
            if (give_up()) return;
    }
};

// One piece of 16 (8) bytes that another CTA publishes.
__device__ __forceinline__ uint4 chain_poll(const void* p, ChainWait& w) {
    uint4 v = ld_relaxed_u4(p);
    w.begin();
    while (chain_missing(v)) {
        if (w.give_up()) break;
        v = ld_relaxed_u4(p);
    }
    return v;
}
__device__ __forceinline__ float2 chain_poll_f2(const void* p, ChainWait& w) {
    uint32_t a, b;
    w.begin();
    for (;;) {
        asm volatile("ld.relaxed.gpu.global.v2.u32 {%0,%1}, [%2];" : "=r"(a), "=r"(b) : "l"(p) : "memory");
        if (max(a, b) != CHAIN_EMPTY || w.give_up()) break;
    }
    return make_float2(__uint_as_float(a), __uint_as_float(b));
}

__device__ __forceinline__ void chain_sync() { asm volatile("bar.sync 1, %0;" ::"n"(32 * CHAIN_WARPS) : "memory"); }

// NC = W / 256: 32-wide K chunks of a warp's eighth of a row.
// Fragment layout: K positions inside a chunk are assigned so that a lane's four A (and B) values of two consecutive
// products are eight neighbouring elements: lane q = lane % 4 takes elements 8 q .. 8 q + 7 of the chunk.
template <int NC>
struct Chain {
    static constexpr int W = 256 * NC;
    static constexpr int GT = chain_token_tiles(NC);               // token tiles of 8 that one pass takes
    static constexpr int NT = NC <= 6 ? GT : 2;                    // of them loaded at once (registers)
    static constexpr int TOKENS = 8 * GT;                          // of a pass
    static constexpr int PER = GT / 4;                             // tokens of a pass that a consumer thread owns
    static constexpr int RED_LD = TOKENS + 1;
    static constexpr uint32_t ROW_BYTES = W * 2 + 64;  // rows of a weight tile start 64 bytes apart modulo the banks
    static constexpr uint32_t TILE_BYTES = CHAIN_COLS * ROW_BYTES;

    // Sums of 16 weight rows x the TOKENS tokens of pass g; every consumer thread gets those of its own column pair
    // (tid % 8) and tokens (tid / 8 + 32 i)
    __device__ static __forceinline__ void product(const uint8_t* act, const uint8_t* hint, uint32_t signals, int S, int g,
                                                   uint32_t tile, float* red, int warp, int lane, ChainWait& wait,
                                                   float2 (&out)[PER]) {
        const int q = lane & 3, r = lane >> 2;
        const int left = S - TOKENS * g;
        float acc[GT][4];
#pragma unroll
        for (int t = 0; t < GT; ++t)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[t][i] = 0.f;
        const uint32_t a_base = tile + (uint32_t)r * ROW_BYTES + (uint32_t)(warp * NC) * 64 + (uint32_t)q * 16;
        const uint32_t tiles = (uint32_t)(S + 7) >> 3;
        const uint8_t* base = act + ((size_t)(warp * NC) * tiles + GT * g) * 512 + lane * 16;
        const uint32_t chunk = tiles * 512;
        if (g == 0) {
            // the CTAs that own this warp's eighth of K have published (see the header)
            if (lane == 0) {
                wait.begin();
                while ((uint32_t)ptx::ld_relaxed_gpu(reinterpret_cast<const int*>(hint + warp * CHAIN_HINT_LINE)) < signals)
                    if (wait.give_up()) break;
            }
            __syncwarp();
        }
#pragma unroll
        for (int t0 = 0; t0 < GT; t0 += NT) {
            if (8 * t0 >= left) break;
            uint4 b[NT][NC];
#pragma unroll
            for (int t = 0; t < NT; ++t)
#pragma unroll
                for (int c = 0; c < NC; ++c)
                    b[t][c] = 8 * (t0 + t) + r < left ? ld_relaxed_u4(base + c * chunk + (t0 + t) * 512)
                                                      : make_uint4(0, 0, 0, 0);
            wait.begin();
            for (;;) {
                bool miss = false;
#pragma unroll
                for (int t = 0; t < NT; ++t)
#pragma unroll
                    for (int c = 0; c < NC; ++c)
                        if (chain_missing(b[t][c])) {
                            miss = true;
                            b[t][c] = ld_relaxed_u4(base + c * chunk + (t0 + t) * 512);
                        }
                if (!miss || wait.give_up()) break;
            }
            __syncwarp();
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                uint4 lo, hi;
                asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                             : "=r"(lo.x), "=r"(lo.y), "=r"(lo.z), "=r"(lo.w) : "r"(a_base + c * 64));
                asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                             : "=r"(hi.x), "=r"(hi.y), "=r"(hi.z), "=r"(hi.w) : "r"(a_base + 8 * ROW_BYTES + c * 64));
#pragma unroll
                for (int t = 0; t < NT; ++t) {
                    if (GT > 4 && 8 * (t0 + t) >= left) break;
                    mma_bf16_16x8x16(acc[t0 + t], lo.x, hi.x, lo.y, hi.y, b[t][c].x, b[t][c].y);
                    mma_bf16_16x8x16(acc[t0 + t], lo.z, hi.z, lo.w, hi.w, b[t][c].z, b[t][c].w);
                }
            }
        }
        float* mine = red + warp * (CHAIN_COLS * RED_LD);
#pragma unroll
        for (int t = 0; t < GT; ++t) {
            if (GT > 4 && 8 * t >= left) break;
            const int tok = 8 * t + 2 * q;
            mine[r * RED_LD + tok] = acc[t][0];
            mine[r * RED_LD + tok + 1] = acc[t][1];
            mine[(r + 8) * RED_LD + tok] = acc[t][2];
            mine[(r + 8) * RED_LD + tok + 1] = acc[t][3];
        }
        chain_sync();
        const int tid = warp * 32 + lane, cp = tid & 7;
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int tok = 32 * i + (tid >> 3);
            out[i] = make_float2(0.f, 0.f);
            if (tok >= left) continue;
#pragma unroll
            for (int w = 0; w < CHAIN_WARPS; ++w) {
                out[i].x += red[(w * CHAIN_COLS + 2 * cp) * RED_LD + tok];
                out[i].y += red[(w * CHAIN_COLS + 2 * cp + 1) * RED_LD + tok];
            }
        }
    }

    // (mean, M2) of the 16 columns that eight neighbouring threads hold as pairs
    __device__ static __forceinline__ float2 own_stats(float2 h) {
        float s = h.x + h.y;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        const float mean = s * (1.0f / 16.0f);
        const float dx = h.x - mean, dy = h.y - mean;
        float m2 = fmaf(dx, dx, dy * dy);
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) m2 += __shfl_xor_sync(0xffffffffu, m2, o);
        return make_float2(mean, m2);
    }
    // Mean and 1 / std of a token from its W / 16 partials, by one warp of the CTA that serves the token; published for
    // all. (Every CTA reading all partials moves S W^2 / 32 bytes per exchange; this way each partial is read once.)
    __device__ static __forceinline__ void serve_stats(const uint8_t* st_row, uint8_t* fin, int lane, ChainWait& wait) {
        constexpr int PIECES = 8 * NC;                  // of two partials
        constexpr int PER = (PIECES + 31) / 32;
        float m[2 * PER], m2 = 0.f, sd = 0.f;
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const bool have = lane + 32 * i < PIECES;
            uint4 v = make_uint4(0, 0, 0, 0);
            if (have) v = chain_poll(st_row + (size_t)(lane + 32 * i) * 16, wait);
            m[2 * i] = __uint_as_float(v.x);
            m[2 * i + 1] = __uint_as_float(v.z);
            m2 += __uint_as_float(v.y) + __uint_as_float(v.w);
        }
        __syncwarp();
        const float p = __shfl_sync(0xffffffffu, m[0], 0);          // pivot: nothing cancels
#pragma unroll
        for (int i = 0; i < PER; ++i)
            if (lane + 32 * i < PIECES) sd += (m[2 * i] - p) + (m[2 * i + 1] - p);
        const float dm = warp_add(sd) * (1.0f / (2 * PIECES));
#pragma unroll
        for (int i = 0; i < PER; ++i)
            if (lane + 32 * i < PIECES) {
                const float d0 = (m[2 * i] - p) - dm, d1 = (m[2 * i + 1] - p) - dm;
                m2 = fmaf(16.0f * d0, d0, m2);
                m2 = fmaf(16.0f * d1, d1, m2);
            }
        m2 = warp_add(m2);
        if (lane == 0) publish_f2(fin, make_float2(p + dm, rsqrtf(m2 * (1.0f / W) + 1e-6f)));
    }
    __device__ static __forceinline__ float warp_add(float v) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    }

    __device__ static __forceinline__ void feed(const ChainParams& P, int cta, uint32_t ring, uint32_t bars, ChainWait& wait) {
        // one thread: the weight tiles in the order they are used
        int slot = 0;
        uint32_t ph = 0, issued = 0, parity = 0;     // slots ever filled, phase of each one's last filling
        auto tile = [&](size_t row0) {
            wait.mbar(bars + 8u * (CHAIN_MAX_SLOTS + slot), ph ^ 1u);
            if (*wait.s_abort) return;
            const uint32_t full = bars + 8u * slot, dst = ring + slot * TILE_BYTES;
            ptx::mbar_arrive_expect_tx(full, CHAIN_COLS * W * 2);
            const bf16* src = P.Wcat + row0 * W;
            for (int r = 0; r < CHAIN_COLS; ++r) ptx::bulk_load(dst + r * ROW_BYTES, src + (size_t)r * W, W * 2, full);
            issued |= 1u << slot;
            parity = (parity & ~(1u << slot)) | (ph << slot);
            if (++slot == P.n_slots) { slot = 0; ph ^= 1u; }
        };
        for (int k = 0; k < P.K && !*wait.s_abort; ++k) {
            for (int b = 0; b < P.L; ++b) {
                tile((size_t)b * 5 * W + 3 * W + cta * CHAIN_COLS);
                tile((size_t)b * 5 * W + 4 * W + cta * CHAIN_COLS);
            }
            if (cta < P.C / CHAIN_COLS) tile(P.out_row0 + cta * CHAIN_COLS);
        }
        // Copies in flight land before the CTA may leave, also where the call is aborted after the last tile was sent for
        // (the consumers then return without waiting for it). Bounded by time; after a normal run all have landed.
        for (int s = 0; s < P.n_slots; ++s)
            if (issued & (1u << s)) drain_mbar(bars + 8u * s, (parity >> s) & 1u);
    }

    __device__ static __forceinline__ void run(const ChainParams& P, int S, int cta, uint32_t ring, uint32_t bars, float* red,
                                               const bf16* win, int warp, int lane, ChainWait& wait) {
        const int tid = warp * 32 + lane, cp = tid & 7, tok0 = tid >> 3;
        const int L = P.L, C = P.C, K = P.K;
        const int n0 = cta * CHAIN_COLS, col = n0 + 2 * cp;
        const int ng = (S + 31) / 32;
        const bool owns_out = cta < C / CHAIN_COLS;
        const ChainLayout lay(S, K, L, W, C);
        const size_t act = lay.act;
        // a warp signals once per exchange if it has tokens; 2 NC CTAs own an eighth of K
        const uint32_t signals = (uint32_t)min(CHAIN_WARPS, (S + 3) / 4) * 2 * NC;
        // this thread's column pair inside an activation tile, and the hint of the K eighth that this CTA writes
        const uint32_t put = (uint32_t)((col % 32) / 8) * 16 + (col % 8) * 2;
        const size_t put_chunk = (size_t)(col / 32) * ((S + 7) / 8) * 512;
        const uint32_t my_hint = (uint32_t)(cta / (2 * NC)) * CHAIN_HINT_LINE;
        auto place = [&](int tok) { return put_chunk + (size_t)(tok >> 3) * 512 + (tok & 7) * 64 + put; };
        auto signal = [&](uint8_t* hint) {
            __syncwarp();
            if (lane == 0 && 4 * warp < S) atomicAdd(reinterpret_cast<unsigned int*>(hint + my_hint), 1u);
        };
        auto hint_u = [&](int q) { return P.xch + (size_t)q * CHAIN_HINT_BYTES; };
        auto hint_a = [&](int q) { return P.xch + (size_t)(K * (L + 1) + q) * CHAIN_HINT_BYTES; };
        int slot = 0, rb = 0;
        uint32_t ph = 0;
        float2 h[CHAIN_GROUPS], x[CHAIN_GROUPS];
        int row[CHAIN_GROUPS];                  // token ids of this thread's tokens
#pragma unroll
        for (int g = 0; g < CHAIN_GROUPS; ++g) row[g] = 32 * g + tok0 < S ? __ldg(P.idx + 32 * g + tok0) : 0;
        const float2 b_in = *reinterpret_cast<const float2*>(P.bin + col);
        if (owns_out) {
#pragma unroll
            for (int g = 0; g < CHAIN_GROUPS; ++g) {
                const int tok = 32 * g + tok0;
                x[g] = tok < S ? *reinterpret_cast<const float2*>(P.noise + (size_t)row[g] * C + col)
                               : make_float2(0.f, 0.f);
            }
        }
        auto take_tile = [&]() { wait.mbar(bars + 8u * slot, ph); return ring + slot * TILE_BYTES; };
        auto free_tile = [&]() {
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bars + 8u * (CHAIN_MAX_SLOTS + slot));
            if (++slot == P.n_slots) { slot = 0; ph ^= 1u; }
        };
        auto product_of = [&](const uint8_t* a, const uint8_t* hint, int p, uint32_t tile, float2 (&out)[PER]) {
            rb ^= 1;
            product(a, hint, signals, S, p, tile, red + rb * (chain_red_bytes(NC) / 4), warp, lane, wait, out);
        };
        // LayerNorm and modulation of h, published as u of (step, layer) index q
        auto publish_u = [&](int k, int block, int q) {
            uint8_t* st = P.xch + lay.st + (size_t)q * ((size_t)(S + 7) / 8 * 8 * (W / 2));
            uint8_t* u = P.xch + lay.u + (size_t)q * act;
            uint8_t* fin = P.xch + lay.fin + (size_t)q * ((size_t)(S + 7) / 8 * 8 * 16);
            const float* sh = P.mods + mods_index(S, L, W, k, block, 0);
            const float* sc = P.mods + mods_index(S, L, W, k, block, 1);
            float2 shv[CHAIN_GROUPS], scv[CHAIN_GROUPS];
#pragma unroll
            for (int g = 0; g < CHAIN_GROUPS; ++g) {
                if (g >= ng) break;
                const int tok = 32 * g + tok0;
                const float2 s = own_stats(h[g]);
                if (cp == 0 && tok < S) publish_f2(st + ((size_t)tok * (W / CHAIN_COLS) + cta) * 8, s);
                const size_t at = (size_t)min(tok, S - 1) * W + col;
                shv[g] = *reinterpret_cast<const float2*>(sh + at);
                scv[g] = *reinterpret_cast<const float2*>(sc + at);
            }
            // token t is served by warp t / CTAs of CTA t % CTAs: at most 4 tokens a CTA (16 CTAs, 64 tokens)
            {
                const int tok = warp * (W / CHAIN_COLS) + cta;
                if (tok < S)
                    serve_stats(st + (size_t)tok * (W / CHAIN_COLS) * 8, fin + (size_t)tok * 16, lane, wait);
            }
#pragma unroll
            for (int g = 0; g < CHAIN_GROUPS; ++g) {
                if (g >= ng) break;
                const int tok = 32 * g + tok0;
                if (tok < S) {
                    const float2 mr = chain_poll_f2(fin + (size_t)tok * 16, wait);
                    const float ux = fmaf((h[g].x - mr.x) * mr.y, 1.0f + scv[g].x, shv[g].x);
                    const float uy = fmaf((h[g].y - mr.x) * mr.y, 1.0f + scv[g].y, shv[g].y);
                    publish_u32(u + place(tok), pack_bf16x2(ux, uy));
                }
            }
            signal(hint_u(q));
        };
        for (int k = 0; k < K; ++k) {
            // h = Win x + bin: the step's x as bf16, from the noise rows or from the CTAs that own x
#pragma unroll
            for (int g = 0; g < CHAIN_GROUPS; ++g) {
                if (g >= ng) break;
                const int tok = 32 * g + tok0;
                h[g] = make_float2(0.f, 0.f);
                // the eight threads of a token fetch 8 of its C <= 64 values each and hand them round
                uint4 v = make_uint4(0, 0, 0, 0);
                if (tok < S && 8 * cp < C) {
                    if (k == 0) {
                        const float* nrow = P.noise + (size_t)row[g] * C + 8 * cp;
                        const float4 a = *reinterpret_cast<const float4*>(nrow);
                        const float4 b = *reinterpret_cast<const float4*>(nrow + 4);
                        v = make_uint4(pack_bf16x2(a.x, a.y), pack_bf16x2(a.z, a.w), pack_bf16x2(b.x, b.y),
                                          pack_bf16x2(b.z, b.w));
                    } else {
                        v = chain_poll(P.xch + lay.xb + (((size_t)(k - 1) * S + tok) * C + 8 * cp) * 2, wait);
                    }
                }
                __syncwarp();
                for (int c = 0; c < C; c += 8) {
                    const uint4 w0 = *reinterpret_cast<const uint4*>(win + (2 * cp) * XB_COLS + c);
                    const uint4 w1 = *reinterpret_cast<const uint4*>(win + (2 * cp + 1) * XB_COLS + c);
                    const uint32_t wa[4] = {w0.x, w0.y, w0.z, w0.w}, wb[4] = {w1.x, w1.y, w1.z, w1.w};
                    const uint32_t mine[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const uint32_t xv = __shfl_sync(0xffffffffu, mine[i], c / 8, 8);
                        h[g].x = fmaf(bf16lo(wa[i]), bf16lo(xv), h[g].x);
                        h[g].x = fmaf(bf16hi(wa[i]), bf16hi(xv), h[g].x);
                        h[g].y = fmaf(bf16lo(wb[i]), bf16lo(xv), h[g].y);
                        h[g].y = fmaf(bf16hi(wb[i]), bf16hi(xv), h[g].y);
                    }
                }
                h[g].x += b_in.x;
                h[g].y += b_in.y;
            }
            for (int b = 0; b < L; ++b) {
                const int q = k * (L + 1) + b;
                publish_u(k, b, q);
                const float2 b1 = *reinterpret_cast<const float2*>(P.bias_cat + (size_t)b * 5 * W + 3 * W + col);
                const float2 b2 = *reinterpret_cast<const float2*>(P.bias_cat + (size_t)b * 5 * W + 4 * W + col);
                const uint8_t* u = P.xch + lay.u + (size_t)q * act;
                uint8_t* a = P.xch + lay.a + (size_t)(k * L + b) * act;
                uint32_t tile = take_tile();
                float2 s[PER];
#pragma unroll
                for (int p = 0; p < CHAIN_GROUPS / PER; ++p) {
                    if (TOKENS * p >= S) break;
                    product_of(u, hint_u(q), p, tile, s);
#pragma unroll
                    for (int i = 0; i < PER; ++i) {
                        const int tok = TOKENS * p + 32 * i + tok0;
                        if (tok < S)
                            publish_u32(a + place(tok), pack_bf16x2(silu_f(s[i].x + b1.x), silu_f(s[i].y + b1.y)));
                    }
                }
                signal(hint_a(q));
                free_tile();
                tile = take_tile();
                const float* gt = P.mods + mods_index(S, L, W, k, b, 2);
#pragma unroll
                for (int p = 0; p < CHAIN_GROUPS / PER; ++p) {
                    if (TOKENS * p >= S) break;
                    float2 gate[PER];
#pragma unroll
                    for (int i = 0; i < PER; ++i)
                        gate[i] = *reinterpret_cast<const float2*>(
                            gt + (size_t)min(TOKENS * p + 32 * i + tok0, S - 1) * W + col);
                    product_of(a, hint_a(q), p, tile, s);
#pragma unroll
                    for (int i = 0; i < PER; ++i) {
                        float2& hh = h[p * PER + i];
                        hh.x = fmaf(gate[i].x, s[i].x + b2.x, hh.x);
                        hh.y = fmaf(gate[i].y, s[i].y + b2.y, hh.y);
                    }
                }
                free_tile();
            }
            publish_u(k, L, k * (L + 1) + L);
            if (owns_out) {
                const uint32_t tile = take_tile();
                const float2 bo = *reinterpret_cast<const float2*>(P.bias_cat + P.out_row0 + col);
                const uint8_t* u = P.xch + lay.u + (size_t)(k * (L + 1) + L) * act;
                float2 s[PER];
#pragma unroll
                for (int p = 0; p < CHAIN_GROUPS / PER; ++p) {
                    if (TOKENS * p >= S) break;
                    product_of(u, hint_u(k * (L + 1) + L), p, tile, s);
#pragma unroll
                    for (int i = 0; i < PER; ++i) {
                        const int g = p * PER + i, tok = 32 * g + tok0;
                        if (tok >= S) continue;
                        float2 base = make_float2(P.ax[k] * x[g].x, P.ax[k] * x[g].y);      // ax = 1: exactly x
                        const size_t at = (size_t)row[g] * C + col;
                        if (P.step_noise) {
                            const float2 z = *reinterpret_cast<const float2*>(P.step_noise + (size_t)k * P.step_stride + at);
                            base.x = fmaf(P.an[k], z.x, base.x);
                            base.y = fmaf(P.an[k], z.y, base.y);
                        }
                        x[g].x = fmaf(P.av[k], s[i].x + bo.x, base.x);
                        x[g].y = fmaf(P.av[k], s[i].y + bo.y, base.y);
                        if (k == K - 1) *reinterpret_cast<float2*>(P.out + at) = x[g];
                        else
                            publish_u32(P.xch + lay.xb + (((size_t)k * S + tok) * C + col) * 2, pack_bf16x2(x[g].x, x[g].y));
                    }
                }
                free_tile();
            }
        }
    }
};

// One CTA's part, called by all its threads: warp 0 feeds, warps 2 .. 9 compute (a call keeps the registers and the code of
// the tile schedule free of it). `bars`: 2 CHAIN_MAX_SLOTS barriers, initialised; smem: 128-byte aligned.
template <int NC>
__device__ __noinline__ void chain_cta(const ChainParams& P, int S, uint8_t* smem, uint32_t bars, volatile int* s_abort) {
    float* red = reinterpret_cast<float*>(smem);
    bf16* win = reinterpret_cast<bf16*>(smem + 2 * chain_red_bytes(NC));
    const uint32_t ring = ptx::smem_u32(smem) + 2 * chain_red_bytes(NC) + CHAIN_COLS * XB_COLS * 2;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, cta = blockIdx.x;
    ChainWait wait(P, s_abort);
    if (warp == 0) {
        if (ptx::elect_one()) Chain<NC>::feed(P, cta, ring, bars, wait);
        __syncwarp();
    } else if (warp >= 2) {
        for (int i = threadIdx.x - 64; i < CHAIN_COLS * XB_COLS / 8; i += 32 * CHAIN_WARPS)
            reinterpret_cast<uint4*>(win)[i] =
                __ldg(reinterpret_cast<const uint4*>(P.Win + (size_t)cta * CHAIN_COLS * XB_COLS) + i);
        chain_sync();
        Chain<NC>::run(P, S, cta, ring, bars, red, win, warp - 2, lane, wait);
    }
}
