// The head's chain of dependent layers for calls of few tokens: one cluster of CTAs takes a group of 16 to 64 tokens through
// all steps, and no cluster waits for another. (The head kernel has made s_k and all modulations before: OP_MOD.)
//   - CTA r of the cluster owns ROWS columns of every layer (W / ROWS CTAs, at most 16). Its weights stream through a ring
//     in shared memory as the A operand of tcgen05.mma (M = 128, of which ROWS rows count), the tokens' activations are
//     the B operand (N = tokens), so an epilogue thread holds four channels of its tokens in fp32 registers: h never leaves
//     them, and biases are one value per thread.
//   - u and a, as bf16, go from every CTA to all others: directly, by bulk copies into their shared memory, where they are
//     small, else through L2, where each fetches them (CL_DIRECT_BYTES). LayerNorm partials go by st.async.
//   - The out-projection is made by every CTA for itself, so x and the in-projection need no exchange.
//   - Five roles: weights (warp 0), products (warp 1), epilogue (warps 2 .. 9), fetching u and a (warp 10).
// What bounds it: the exchanges. Of a block's 22 K cycles at W = 1024 and 48 tokens in each of 15 clusters of 8, the products
// take 6 K (16 slices of 64 at 182 cycles, twice), the rest is publishing u and a (2 K each: the release waits for L2),
// fetching 86 KB of them (5 K each) and the LayerNorm's partials and arithmetic (4 K). With no weights loaded and a quarter of
// the products the same block took 85 % of its time. Direct copies move 11 bytes per cycle and SM (8 K cycles for these 86
// KB, 2.6 K for the 30 KB of 16 tokens), L2 gives more but takes 2.5 K to start.
// Kernel times of a call (K = 4, modulations included), us, tile schedule or chain.cuh / clusters: W = 256, 2 blocks, 32
// tokens 125 / 72, 256 177 / 76, 4096 212 / 180; W = 512, 3 blocks, 64 232 / 115, 2048 346 / 289; W = 1024, 3 blocks, 28
// 197 / 168, 128 358 / 178, 700 426 / 321, but two rounds of groups, 1434 475 / 565: hence one round at most. W = 1280 16
// 201 / 210, 64 336 / 216; W = 1536, 12 blocks, 28 728 / 749, 64 1094 / 745, 224 1675 / 912; W = 2048, 28 303 / 330, 64 434 /
// 331, 200 604 / 460: hence chain.cuh for the fewest tokens of wide heads.
#pragma once

struct ClusterParams {
    int C, W, L, K, n_ctas, max_tokens;
    int above, limit;                          // calls of more than `above` and up to `limit` survivors
    uint32_t direct_bytes;                     // up to this size u and a go from CTA to CTA directly (see cluster_kernel)
    int map_cat, map_in, map_out;              // weight boxes: ROWS x 64 of the packed weights and of Win, C x 64 of Wout
    size_t out_row0;                           // Wout in the packed weights
    const CUtensorMap* maps;
    const int *idx, *count;
    const float *bias_cat, *bin, *noise, *step_noise, *mods;
    long long step_stride;
    float* out;
    uint8_t* xch;                              // u and a of every cluster
    int *status, *abort_flag;
    unsigned long long wait_limit_ns;
    int stall_cluster;                         // self-test: this cluster's last CTA gets no weights after the first block's W1 (-1: none)
    float ax[KMAX], av[KMAX], an[KMAX];
};

struct ClusterBars {
    uint64_t full[CL_MAX_STAGES], empty[CL_MAX_STAGES];
    uint64_t src_u[CL_MAX_CTAS], src_a[CL_MAX_CTAS];     // the part of u (a) that this CTA of the cluster owns is there
    uint64_t sig[2];                                     // u (a) of all other CTAs is in L2
    uint64_t x, acc[2], stat[2], drain;
};

// Modulation values of step k: [block][shift, scale, gate], then the final layer's [shift, scale]; of each, tiles
// [32 channels][8 tokens][16 channels][lane][4]: lane l has channels l / 4 and l / 4 + 8, tokens 2 (l % 4) and + 1.
__host__ __device__ __forceinline__ size_t mods_at(int L, int W, int ld, int k, int block, int which, int ch32, int tok8) {
    return (((size_t)k * (3 * L + 2) + 3 * block + which) * (W / 32) + ch32) * (ld / 8) * 256 + (size_t)tok8 * 256;
}

// A bound on every wait of a thread: after an abort all further waits return at once, the kernel runs to its end on
// whatever it has and the call is reported as timed out.
struct ClusterWait {
    const ClusterParams& P;
    volatile int* s_abort;
    __device__ __forceinline__ ClusterWait(const ClusterParams& p, volatile int* f) : P(p), s_abort(f) {}
    __device__ __forceinline__ bool aborted() const { return *s_abort != 0; }
    template <bool CLUSTER = false>
    __device__ __forceinline__ bool mbar(uint32_t bar, uint32_t parity) {      // false: gave up
        auto there = [&] { return CLUSTER ? ptx::mbar_try_wait_cluster(bar, parity) : ptx::mbar_try_wait(bar, parity); };
        if (there()) return true;
        uint64_t t0 = 0;
        for (uint32_t it = 1;; ++it) {
            if (there()) return true;
            if (*s_abort) return false;
            if ((it & 1023u) != 0) continue;             // (the two reads below take 1000 cycles)
            const uint64_t now = ptx::globaltimer_ns();
            if (t0 == 0) t0 = now;
            bool stop = ptx::ld_relaxed_gpu(P.abort_flag) != 0;
            if (!stop && now - t0 > P.wait_limit_ns) {
                atomicExch(P.abort_flag, 1);
                atomicCAS(P.status, 0, ARDIFF_ERR_TIMEOUT);
                stop = true;
            }
            if (stop) { *s_abort = 1; return false; }
        }
    }
};

template <int ROWS, int G>
struct ClusterEpilogue {
    static constexpr int N = G * CL_UNIT;
    static constexpr int NQ = ROWS / 32;                 // TMEM lane quarters in use
    static constexpr int THREADS = 2 * NQ * 32;          // epilogue threads in use
    using Tile = float[G][2][4];    // [8 tokens][16 channels][channel l / 4 (+ 8), tokens 2 (l % 4), + 1]

    __device__ static __forceinline__ void load_acc(uint32_t tacc, Tile& v) {
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
            for (int i = 0; i < 2; ++i) ptx::tmem_ld_16x256b(tacc + ((uint32_t)(16 * i) << 16) + 8 * g, v[g][i]);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) asm volatile("" : "+f"(v[g][i][e]));
        ptx::tc_fence_before();
    }
    __device__ static __forceinline__ float add8(float v) {      // over the eight lanes that hold a token's channels
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    }

    __device__ static __forceinline__ void run(const ClusterParams& P, int S, int cluster, int rank, uint32_t smem, uint32_t tmem,
                                               ClusterBars& B, int warp, int lane, ClusterWait& wait) {
        const int quarter = (warp + 2) & 3, half = warp >> 2;    // (warp: 0 .. 7 of the epilogue; quarter = hardware warp % 4)
        if (quarter >= NQ) return;
        const int W = P.W, C = P.C, L = P.L, K = P.K, n_ctas = P.n_ctas;
        const ClusterLayout lay(W, C, ROWS, G);
        const int me = half * NQ + quarter;              // this warp among the active ones
        const int r8 = lane >> 2, c4 = lane & 3;
        const int ch0 = rank * ROWS + quarter * 32 + r8; // channel of [.][0][0 .. 1]; the others 8, 16 and 24 further
        const int ld = mods_stride(S);
        const uint32_t tacc0 = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(half * 8 * G);
        const uint32_t bar_x = ptx::smem_u32(&B.x), bar_acc = ptx::smem_u32(B.acc), bar_stat = ptx::smem_u32(&B.stat[half]);
        uint8_t* const xch = P.xch + (size_t)cluster * 2 * lay.act;      // u, then a
        const bool direct = lay.act <= P.direct_bytes;
        const uint32_t part = smem + lay.part + (uint32_t)half * (4 * G * NQ * 16);
        const uint32_t stats = smem + lay.stats + (uint32_t)half * (4 * G * n_ctas * 16);
        // where this lane's row of a stored 8 x 8 block goes: block lane / 8 (channels), token lane % 8
        const uint32_t put = ((uint32_t)(quarter * 4 + (lane >> 3)) * N + (uint32_t)(half * 8 * G + (lane & 7))) * 16;
        const uint32_t own = (uint32_t)rank * (ROWS * 2 * N);
        const float inv_ctas = 1.0f / (float)n_ctas, inv_w = 1.0f / (float)W;
        uint32_t n_acc = 0, ph_stat = 0;

        auto next_acc = [&](Tile& v) {
            wait.mbar(bar_acc + 8 * (n_acc & 1), (n_acc >> 1) & 1);
            __syncwarp();
            ptx::tc_fence_after();
            load_acc(tacc0 + (n_acc & 1) * 64, v);
            ++n_acc;
        };
        auto store_blocks = [&](uint32_t base, const Tile& v) {
#pragma unroll
            for (int g = 0; g < G; ++g)
                ptx::stmatrix_x4_trans(base + g * 128, pack_bf16x2(v[g][0][0], v[g][0][1]), pack_bf16x2(v[g][0][2], v[g][0][3]),
                                       pack_bf16x2(v[g][1][0], v[g][1][1]), pack_bf16x2(v[g][1][2], v[g][1][3]));
        };
        // this CTA's channels of u or a to every CTA of the cluster
        auto publish = [&](uint32_t act, uint64_t* src, uint64_t* sig, uint8_t* global, const Tile& v) {
            store_blocks(smem + act + own + put, v);
            if (direct) {
                ptx::fence_proxy_async_smem();
                ptx::bar_sync(1, THREADS);
                if (ptx::elect_one() && !wait.aborted()) {
                    const uint32_t from = smem + act + own, bar = ptx::smem_u32(&src[rank]);
                    for (int p = me; p < n_ctas; p += 2 * NQ) {
                        if (p != rank) ptx::bulk_copy_cluster(ptx::map_peer(from, p), from, ROWS * 2 * N, ptx::map_peer(bar, p));
                    }
                }
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&src[rank]));
            } else {
                __syncwarp();
                // the warp's 4 x 8 G pieces of 16 bytes to L2, then word to the CTAs that will fetch them
#pragma unroll
                for (int t = lane; t < 32 * G; t += 32) {
                    const uint32_t at = own + ((uint32_t)(quarter * 4 + t / (8 * G)) * N + (uint32_t)(half * 8 * G + t % (8 * G))) * 16;
                    ptx::st_u4(global + at, ptx::lds_u4(smem + act + at));
                }
                ptx::fence_proxy_async_smem();            // (this CTA's products read the part where it lies)
                __syncwarp();
                if (lane < n_ctas) {
                    if (lane == rank) ptx::mbar_arrive(ptx::smem_u32(&src[rank]));
                    else if (!wait.aborted()) ptx::mbar_arrive_cluster(ptx::map_peer(ptx::smem_u32(sig), lane));
                }
                __syncwarp();
            }
        };

        const int tok0 = cluster * N + half * 8 * G + 2 * c4;
        // modulations of this thread's channels and tokens (no read-only loads: the kernel before, which writes them, may
        // still run when this one starts)
        auto mods = [&](int k, int block, int which, Tile& v) {
            const float* m = P.mods + mods_at(L, W, ld, k, block, which, rank * NQ + quarter, 0) + lane * 4;
#pragma unroll
            for (int g = 0; g < G; ++g)
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int tok8 = min(cluster * (N / 8) + half * G + g, ld / 8 - 1);
                    const float4 w = ptx::ldcg_f4(m + (size_t)tok8 * 256 + i * 128);
                    v[g][i][0] = w.x; v[g][i][1] = w.y; v[g][i][2] = w.z; v[g][i][3] = w.w;
                }
        };
        // those of the CTA into L2, for later: many tokens' lie in HBM
        auto fetch = [&](int k, int block, int which) {
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                ptx::bulk_prefetch_l2(P.mods + mods_at(L, W, ld, k, block, which, rank * NQ + q, cluster * (N / 8)),
                                      (uint32_t)min(N / 8, ld / 8 - cluster * (N / 8)) * 1024);
        };
        auto bias = [&](const float* b, float (&v)[2][2]) {
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j) v[i][j] = __ldg(b + 16 * i + 8 * j);
        };
        Tile h;
        // x of this thread's output channels (the warps of the first 64 channels; the same in every CTA): few steps
        // change it, so it lies in shared memory
        const bool has_x = quarter < 2;
        const int cx = quarter * 32 + r8;
        auto row_of = [&](int g, int e) {                  // token id, or -1
            const int tok = tok0 + 8 * g + e;
            return tok < S ? __ldg(P.idx + tok) : -1;
        };
        auto rows_of = [&](const float* base, Tile& v) {
#pragma unroll
            for (int g = 0; g < G; ++g)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int rw = row_of(g, e);
#pragma unroll
                    for (int i = 0; i < 2; ++i)
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            const int c = cx + 16 * i + 8 * j;
                            v[g][i][2 * j + e] = c < C && rw >= 0 ? __ldg(base + (size_t)rw * C + c) : 0.f;
                        }
                }
        };
        const uint32_t x_at = smem + lay.x + (uint32_t)(cx * N + half * 8 * G + 2 * c4) * 4;
        auto store_x = [&](const Tile& x) {
#pragma unroll
            for (int g = 0; g < G; ++g)
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int j = 0; j < 2; ++j)
                        if (cx + 16 * i + 8 * j < C)
                            ptx::sts_f2(x_at + (uint32_t)((16 * i + 8 * j) * N + 8 * g) * 4, x[g][i][2 * j], x[g][i][2 * j + 1]);
            // as bf16, and where the slice of 64 has room for it what the rounding took off in the C columns behind (Win
            // is there twice): the in-projection then sees x to 16 bits, for nothing
            if (C <= 32) {
                Tile lo;
#pragma unroll
                for (int g = 0; g < G; ++g)
#pragma unroll
                    for (int i = 0; i < 2; ++i)
#pragma unroll
                        for (int e = 0; e < 4; ++e) lo[g][i][e] = x[g][i][e] - __bfloat162float(__float2bfloat16_rn(x[g][i][e]));
                if (C == 16) {
#pragma unroll
                    for (int g = 0; g < G; ++g)
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float v = lo[g][0][e];
                            lo[g][0][e] = x[g][0][e];
                            lo[g][1][e] = quarter == 0 ? v : 0.f;
                        }
                    store_blocks(smem + lay.xb + put, lo);
                } else if (quarter == 0) {
                    store_blocks(smem + lay.xb + put, x);
                    store_blocks(smem + lay.xb + put + 4 * N * 16, lo);
                }
            } else {
                store_blocks(smem + lay.xb + put, x);
            }
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar_x);
        };
        if (has_x) {
            Tile x;
            rows_of(P.noise, x);
            store_x(x);
        }
        for (int k = 0; k < K; ++k) {
            {   // h = Win x + bin
                float b[2][2];
                bias(P.bin + ch0, b);
                next_acc(h);
#pragma unroll
                for (int g = 0; g < G; ++g)
#pragma unroll
                    for (int i = 0; i < 2; ++i)
#pragma unroll
                        for (int e = 0; e < 4; ++e) h[g][i][e] += b[i][e >> 1];
            }
            for (int b = 0;; ++b) {
                // u = LN(h) (1 + scale) + shift
                {
#pragma unroll
                    for (int g = 0; g < G; ++g) {
                        float mean[2], m2[2];
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const float s = add8((h[g][0][e] + h[g][0][2 + e]) + (h[g][1][e] + h[g][1][2 + e]));
                            mean[e] = s * (1.0f / 32.0f);
                            float q = 0.f;
#pragma unroll
                            for (int i = 0; i < 2; ++i)
#pragma unroll
                                for (int j = 0; j < 2; ++j) {
                                    const float d = h[g][i][2 * j + e] - mean[e];
                                    q = fmaf(d, d, q);
                                }
                            m2[e] = add8(q);
                        }
                        if (r8 == 0) ptx::sts_f4(part + (uint32_t)((4 * g + c4) * NQ + quarter) * 16, mean[0], m2[0], mean[1], m2[1]);
                    }
                    ptx::bar_sync(2 + half, 32 * NQ);
                    // the CTA's partials of 4 G pairs of tokens, to every CTA of the cluster
                    for (int t = quarter * 32 + lane; t < 4 * G * n_ctas; t += 32 * NQ) {
                        const int pair = t % (4 * G), peer = t / (4 * G);
                        float4 v[NQ];
#pragma unroll
                        for (int q = 0; q < NQ; ++q) v[q] = ptx::lds_f4(part + (uint32_t)(pair * NQ + q) * 16);
                        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                        for (int q = 0; q < NQ; ++q) { o.x += v[q].x; o.z += v[q].z; o.y += v[q].y; o.w += v[q].w; }
                        o.x *= 1.0f / NQ;
                        o.z *= 1.0f / NQ;
#pragma unroll
                        for (int q = 0; q < NQ; ++q) {
                            const float d0 = v[q].x - o.x, d1 = v[q].z - o.z;
                            o.y = fmaf(32.0f * d0, d0, o.y);
                            o.w = fmaf(32.0f * d1, d1, o.w);
                        }
                        if (!wait.aborted())
                            ptx::st_async_f4(ptx::map_peer(stats + (uint32_t)(pair * n_ctas + rank) * 16, peer), o,
                                             ptx::map_peer(bar_stat, peer));
                    }
                    Tile sh, u;                          // (u: the scale, then the result)
                    mods(k, b, 0, sh);
                    mods(k, b, 1, u);
                    const bool there = wait.mbar(bar_stat, ph_stat);
                    ph_stat ^= 1;
                    __syncwarp();
                    // (never twice in a phase: not after a wait that gave up, nor after one that came too early because
                    // of it)
                    if (quarter == 0 && lane == 0 && there && !wait.aborted())
                        ptx::mbar_arrive_expect_tx(bar_stat, 4 * G * n_ctas * 16);
#pragma unroll
                    for (int g = 0; g < G; ++g) {
                        float4 v[2];
#pragma unroll
                        for (int s = 0; s < 2; ++s) {
                            v[s] = make_float4(0.f, 0.f, 0.f, 0.f);
                            if (r8 + 8 * s < n_ctas) v[s] = ptx::lds_f4(stats + (uint32_t)((4 * g + c4) * n_ctas + r8 + 8 * s) * 16);
                        }
                        const float mean[2] = {add8(v[0].x + v[1].x) * inv_ctas, add8(v[0].z + v[1].z) * inv_ctas};
                        float q0 = v[0].y + v[1].y, q1 = v[0].w + v[1].w;
#pragma unroll
                        for (int s = 0; s < 2; ++s)
                            if (r8 + 8 * s < n_ctas) {
                                const float d0 = v[s].x - mean[0], d1 = v[s].z - mean[1];
                                q0 = fmaf((float)ROWS * d0, d0, q0);
                                q1 = fmaf((float)ROWS * d1, d1, q1);
                            }
                        const float rstd[2] = {rsqrtf(add8(q0) * inv_w + 1e-6f), rsqrtf(add8(q1) * inv_w + 1e-6f)};
#pragma unroll
                        for (int i = 0; i < 2; ++i)
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                u[g][i][e] = fmaf((h[g][i][e] - mean[e & 1]) * rstd[e & 1], 1.0f + u[g][i][e], sh[g][i][e]);
                    }
                    publish(lay.u, B.src_u, &B.sig[0], xch, u);
                }
                if (me == 0 && ptx::elect_one()) {
                    if (b < L) {
                        fetch(k, b, 2);
                        fetch(k, b + 1, 0);
                        fetch(k, b + 1, 1);
                    } else if (k + 1 < K) {
                        fetch(k + 1, 0, 0);
                        fetch(k + 1, 0, 1);
                    }
                }
                __syncwarp();
                if (b == L) break;
                const float* b_blk = P.bias_cat + (size_t)b * 5 * W + ch0;
                {   // a = SiLU(W1 u + b1)
                    float b1[2][2];
                    bias(b_blk + 3 * (size_t)W, b1);
                    Tile a;
                    next_acc(a);
#pragma unroll
                    for (int g = 0; g < G; ++g)
#pragma unroll
                        for (int i = 0; i < 2; ++i)
#pragma unroll
                            for (int e = 0; e < 4; ++e) a[g][i][e] = silu_f(a[g][i][e] + b1[i][e >> 1]);
                    publish(lay.a, B.src_a, &B.sig[1], xch + lay.act, a);
                }
                {   // h += gate * (W2 a + b2)
                    Tile gate;
                    mods(k, b, 2, gate);
                    float b2[2][2];
                    bias(b_blk + 4 * (size_t)W, b2);
                    Tile v;
                    next_acc(v);
#pragma unroll
                    for (int g = 0; g < G; ++g)
#pragma unroll
                        for (int i = 0; i < 2; ++i)
#pragma unroll
                            for (int e = 0; e < 4; ++e) h[g][i][e] = fmaf(gate[g][i][e], v[g][i][e] + b2[i][e >> 1], h[g][i][e]);
                }
            }
            if (!has_x) { ++n_acc; continue; }
            {   // x <- ax x + av (Wout u + bout) + an z
                Tile z;
                if (P.step_noise) rows_of(P.step_noise + (size_t)k * (size_t)P.step_stride, z);
                float bo[2][2];
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int j = 0; j < 2; ++j) bo[i][j] = cx + 16 * i + 8 * j < C ? __ldg(P.bias_cat + P.out_row0 + cx + 16 * i + 8 * j) : 0.f;
                const float ax = P.ax[k], av = P.av[k], an = P.an[k];
                Tile v;
                next_acc(v);
#pragma unroll
                for (int g = 0; g < G; ++g)
#pragma unroll
                    for (int i = 0; i < 2; ++i)
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            const bool have = cx + 16 * i + 8 * j < C;
                            float2 x = make_float2(0.f, 0.f);
                            if (have) x = ptx::lds_f2(x_at + (uint32_t)((16 * i + 8 * j) * N + 8 * g) * 4);
                            x.x *= ax;                                    // ax = 1: exactly x
                            x.y *= ax;
                            if (P.step_noise) {
                                x.x = fmaf(an, z[g][i][2 * j], x.x);
                                x.y = fmaf(an, z[g][i][2 * j + 1], x.y);
                            }
                            v[g][i][2 * j] = have ? fmaf(av, v[g][i][2 * j] + bo[i][j], x.x) : 0.f;
                            v[g][i][2 * j + 1] = have ? fmaf(av, v[g][i][2 * j + 1] + bo[i][j], x.y) : 0.f;
                        }
                if (k + 1 < K) store_x(v);
                else if (rank == 0) {
#pragma unroll
                    for (int g = 0; g < G; ++g)
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const int rw = row_of(g, e);
#pragma unroll
                            for (int i = 0; i < 2; ++i)
#pragma unroll
                                for (int j = 0; j < 2; ++j)
                                    if (cx + 16 * i + 8 * j < C && rw >= 0)
                                        P.out[(size_t)rw * C + cx + 16 * i + 8 * j] = v[g][i][2 * j + e];
                        }
                }
            }
        }
    }
};

// One thread: the weight slices in the order they are used. A layer's K slices start with the CTA's own channels, whose
// activations are there first.
template <int ROWS>
__device__ __forceinline__ void cluster_feed(const ClusterParams& P, int cluster, int rank, const ClusterLayout& lay, uint32_t ring,
                                             ClusterBars& B, ClusterWait& wait) {
    const uint32_t full = ptx::smem_u32(B.full), empty = ptx::smem_u32(B.empty);
    constexpr int SL = cl_slices(ROWS), SRCS = SL * CL_KS / ROWS;
    const int W = P.W, stages = W / (CL_KS * SL), layers = 2 * P.L + 2;
    int st = 0;
    uint32_t ph = 0, issued = 0, parity = 0;
    bool ok = true;
    // (one loop over the layers of a step with one copy in it: see cluster_mma)
    for (int k = 0; ok && k < P.K; ++k)
        for (int l = 0; ok && l < layers; ++l) {
            const bool in = l == 0, out = l == layers - 1;
            const int n = in ? 1 : stages, sl = in ? 1 : SL;
            const void* map = P.maps + (in ? P.map_in : out ? P.map_out : P.map_cat);
            const int row = in ? rank * ROWS : out ? (int)P.out_row0 : (5 * ((l - 1) >> 1) + 3 + ((l - 1) & 1)) * W + rank * ROWS;
            const uint32_t bytes = (uint32_t)(out ? P.C : ROWS) * CL_KS * 2 * sl;
            int kp = in ? 0 : rank / SRCS;
            if (l == 2 && cluster == P.stall_cluster && rank == P.n_ctas - 1) {      // self-test (nothing ends this wait in time)
                wait.mbar(ptx::smem_u32(&B.drain), 0);
                ok = false;
                break;
            }
            for (int i = 0; i < n; ++i) {
                ok = wait.mbar(empty + 8 * st, ph ^ 1u);
                if (!ok) break;
                ptx::mbar_arrive_expect_tx(full + 8 * st, bytes);
                const uint32_t dst = ring + (uint32_t)st * lay.stage;
                for (int j = 0; j < sl; ++j)
                    ptx::tma_load_2d(dst + (uint32_t)j * (ROWS * CL_KS * 2), map, full + 8 * st, (kp * SL + j) * CL_KS, row);
                issued |= 1u << st;
                parity = (parity & ~(1u << st)) | (ph << st);
                if (++st == lay.stages) { st = 0; ph ^= 1u; }
                if (++kp == n) kp = 0;
            }
        }
    // copies in flight land before the CTA may leave (bounded by time: an aborted call has slices nobody waits for)
    for (int s = 0; s < lay.stages; ++s)
        if (issued & (1u << s)) drain_mbar(full + 8 * s, (parity >> s) & 1u);
}

// One thread: the products. Weights are the A operand (128 rows of it, ROWS of them this CTA's), the activations of all
// CTAs the B operand, which lies in shared memory as [8 channels][token][16 bytes].
template <int ROWS>
__device__ __forceinline__ void cluster_mma(const ClusterParams& P, int units, int rank, const ClusterLayout& lay, uint32_t smem,
                                            uint32_t tmem, ClusterBars& B, ClusterWait& wait) {
    const uint32_t full = ptx::smem_u32(B.full), empty = ptx::smem_u32(B.empty), acc = ptx::smem_u32(B.acc);
    constexpr int SL = cl_slices(ROWS), SRCS = SL * CL_KS / ROWS;
    const int stages = P.W / (CL_KS * SL);
    const uint32_t N = (uint32_t)units * CL_UNIT, idesc = ptx::idesc_bf16_f32(128, N);
    const uint32_t part = ROWS * 2 * N;
    const bool direct = lay.act <= P.direct_bytes;
    int st = 0;
    uint32_t ph = 0, n_acc = 0, ph_x = 0, ph_u = 0, ph_a = 0;
    for (int p = 0; direct && p < P.n_ctas; ++p)
        if (p != rank) {
            ptx::mbar_arrive_expect_tx(ptx::smem_u32(&B.src_u[p]), part);
            ptx::mbar_arrive_expect_tx(ptx::smem_u32(&B.src_a[p]), part);
        }
    const int layers = 2 * P.L + 2;              // of a step: in-projection, W1 and W2 of every block, out-projection
    const uint32_t bar_u = ptx::smem_u32(B.src_u), bar_a = ptx::smem_u32(B.src_a);
    bool ok = true;
    // One loop with one set of asynchronous instructions in it: called from several places the body becomes a function, in
    // which the compiler no longer knows that one thread is active (see ptx::elect_one).
    for (int k = 0; ok && k < P.K; ++k)
        for (int l = 0; ok && l < layers; ++l) {
            const bool in = l == 0, odd = l & 1;         // odd: operand u, even: operand a
            const int n = in ? 1 : stages;
            const uint32_t act = smem + (in ? lay.xb : odd ? lay.u : lay.a), src = odd ? bar_u : bar_a;
            const uint32_t phase = odd ? ph_u : ph_a, d = tmem + (n_acc & 1) * 64;
            // a layer's stages start with the one that holds this CTA's own channels: they are there first
            int kp = in ? 0 : rank / SRCS;
            if (in) ok = wait.mbar(ptx::smem_u32(&B.x), ph_x);
            for (int i = 0; ok && i < n; ++i) {
                ok = wait.mbar(full + 8 * st, ph);
                const uint32_t a0 = smem + (uint32_t)st * lay.stage, b0 = act + (uint32_t)(kp * SL) * (8 * N * 16);
#pragma unroll
                for (int j = 0; j < SL; ++j) {
                    if (in && j > 0) break;
                    // the CTAs whose channels the slice holds
                    if (!in && SRCS == SL) ok = ok && wait.mbar(src + 8 * (kp * SRCS + j), phase);
                    else if (!in && j == 0)
                        for (int q = 0; q < SRCS; ++q) ok = ok && wait.mbar(src + 8 * (kp * SRCS + q), phase);
                    if (!ok) break;
                    ptx::tc_fence_after();
                    const uint64_t da = ptx::smem_desc_sw128(a0 + (uint32_t)j * (ROWS * CL_KS * 2));
                    const uint64_t db = ptx::smem_desc_plain(b0 + (uint32_t)j * (8 * N * 16), N * 16, 128);
#pragma unroll
                    for (int q = 0; q < CL_KS / 16; ++q)
                        ptx::mma_f16_ss(d, da + (uint64_t)(2 * q), db + (uint64_t)(q * 2) * N, idesc, (i | j | q) != 0 ? 1u : 0u);
                }
                if (!ok) break;
                ptx::mma_commit(empty + 8 * st);
                if (++st == lay.stages) { st = 0; ph ^= 1u; }
                if (++kp == n) kp = 0;
            }
            if (ok) ptx::mma_commit(acc + 8 * (n_acc & 1));
            ++n_acc;
            // what the next exchange of this operand brings (its first bytes may come before this, but not its last:
            // the barrier waits for this arrival)
            for (int p = 0; direct && ok && !in && p < P.n_ctas; ++p)
                if (p != rank) ptx::mbar_arrive_expect_tx(src + 8 * p, part);
            if (in) ph_x ^= 1;
            else if (odd) ph_u ^= 1;
            else ph_a ^= 1;
        }
    // all products are done before tensor memory is freed
    ptx::mma_commit(ptx::smem_u32(&B.drain));
    drain_mbar(ptx::smem_u32(&B.drain), 0);
}

// One thread: u and a of the other CTAs from L2, when all have said that their parts are there (a wait for each, with the
// fences it needs, took 1000 cycles a CTA).
template <int ROWS>
__device__ __forceinline__ void cluster_fetch(const ClusterParams& P, int units, int cluster, int rank, const ClusterLayout& lay,
                                              uint32_t smem, ClusterBars& B, ClusterWait& wait) {
    if (lay.act <= P.direct_bytes) return;
    const uint32_t part = ROWS * 2 * (uint32_t)units * CL_UNIT, acc = ptx::smem_u32(B.acc);
    const uint8_t* xch = P.xch + (size_t)cluster * 2 * lay.act;
    uint32_t ph_u = 0, ph_a = 0, n_acc = 0;
    bool ok = true;
    for (int k = 0; ok && k < P.K; ++k) {
        ++n_acc;                                          // the in-projection
        for (int l = 1; ok && l < 2 * P.L + 2; ++l, ++n_acc) {
            const bool odd = l & 1;                       // u, else a
            const uint32_t act = smem + (odd ? lay.u : lay.a), src = ptx::smem_u32(odd ? B.src_u : B.src_a);
            const uint32_t sig = ptx::smem_u32(&B.sig[odd ? 0 : 1]), phase = odd ? ph_u : ph_a;
            const uint8_t* from = odd ? xch : xch + lay.act;
            // where they share a buffer a takes u's place when the products of u are done (u takes a's when all CTAs
            // have sent their partials of the LayerNorm that it comes from, this one among them: after its products)
            if (!odd && lay.bufs == 1) ok = wait.mbar(acc + 8 * ((n_acc - 1) & 1), ((n_acc - 1) >> 1) & 1);
            ok = ok && wait.template mbar<true>(sig, phase);
            if (ok) ptx::fence_proxy_async();
            int s = rank;
            for (int i = 1; ok && i < P.n_ctas; ++i) {
                if (++s == P.n_ctas) s = 0;
                ptx::mbar_arrive_expect_tx(src + 8 * s, part);
                ptx::bulk_load(act + (uint32_t)s * part, from + (size_t)s * part, part, src + 8 * s);
            }
            if (odd) ph_u ^= 1;
            else ph_a ^= 1;
        }
    }
    // (after a normal run all of them have landed: the products waited for them; after an abort the kernel waits)
}

template <int ROWS>
__global__ void __launch_bounds__(CL_THREADS, 1) cluster_kernel(const __grid_constant__ ClusterParams P) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ ClusterBars B;
    __shared__ int s_abort;
    __shared__ uint32_t s_tmem;
    // Launched while the modulations are still made: its start hides behind their last items. A call for the chain or the tile
    // schedule pays for a launch all the same. The count is there already (this kernel starts after head_kernel has, and that
    // after the kernels before it are done), so all CTAs but one leave as they come, and that one keeps the stream's order:
    // what follows waits for this launch. Behind the chain 1.9 -> 0.9 us, behind tiles 2.5 .. 6 -> 1.3 .. 5 (W = 512, 1024,
    // 2048: 2.3 -> 1.3, 5.6 -> 4.2, 6.3 -> 5.1 at K = 1).
    const int S = min(ptx::ld_relaxed_gpu(P.count), P.max_tokens);
    if (S <= P.above || S > P.limit) {
        if (blockIdx.x == 0) ptx::wait_for_prior_kernel();
        return;
    }
    ptx::wait_for_prior_kernel();
    const int n_ctas = P.n_ctas, rank = (int)blockIdx.x % n_ctas, cluster = (int)blockIdx.x / n_ctas;
    // units of 16 tokens dealt evenly to the clusters (one round of groups: the host's limit, cluster_survivors)
    const int n_clusters = (int)gridDim.x / n_ctas, all_units = (S + CL_UNIT - 1) / CL_UNIT;
    const int units = (all_units + n_clusters - 1) / n_clusters;
    if (cluster * units >= all_units) return;   // (all CTAs of the cluster)
    const ClusterLayout lay(P.W, P.C, ROWS, units);
    const uint32_t smem = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        s_abort = ptx::ld_relaxed_gpu(P.abort_flag) != 0;       // what made the modulations gave up
        const uint32_t bars = ptx::smem_u32(&B);
        for (uint32_t i = 0; i < sizeof(ClusterBars) / 8; ++i) {
            const uint32_t bar = bars + 8 * i;
            const bool sig = bar == ptx::smem_u32(&B.sig[0]) || bar == ptx::smem_u32(&B.sig[1]);
            const bool own = bar == ptx::smem_u32(&B.src_u[rank]) || bar == ptx::smem_u32(&B.src_a[rank]);
            // (ROWS / 16: the epilogue's warps)
            ptx::mbar_init(bar, bar == ptx::smem_u32(&B.x) ? 4 : sig ? (n_ctas - 1) * ROWS / 16 : own ? ROWS / 16 : 1);
        }
        ptx::fence_mbar_init();
        for (int i = 0; i < 2; ++i)
            ptx::mbar_arrive_expect_tx(ptx::smem_u32(&B.stat[i]), 4 * units * n_ctas * 16);
    }
    if (warp == 1) {
        ptx::tmem_alloc(ptx::smem_u32(&s_tmem), 128);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    const bool gave_up = s_abort != 0;
    ptx::cluster_sync_all();
    ptx::tc_fence_after();
    const uint32_t tmem = s_tmem;
    ClusterWait wait(P, &s_abort);

    if (gave_up) {
        // nothing to work on
    } else if (warp == 0) {
        if (ptx::elect_one()) cluster_feed<ROWS>(P, cluster, rank, lay, smem, B, wait);
        __syncwarp();
    } else if (warp == 1) {
        if (ptx::elect_one()) cluster_mma<ROWS>(P, units, rank, lay, smem, tmem, B, wait);
        __syncwarp();
    } else if (warp == 10) {
        if (ptx::elect_one()) cluster_fetch<ROWS>(P, units, cluster, rank, lay, smem, B, wait);
        __syncwarp();
    } else {
        constexpr int M = cl_most_units(ROWS);
        switch (units) {
            case 1: ClusterEpilogue<ROWS, 1>::run(P, S, cluster, rank, smem, tmem, B, warp - 2, lane, wait); break;
            case 2: if constexpr (M >= 2) ClusterEpilogue<ROWS, 2>::run(P, S, cluster, rank, smem, tmem, B, warp - 2, lane, wait); break;
            case 3: if constexpr (M >= 3) ClusterEpilogue<ROWS, 3>::run(P, S, cluster, rank, smem, tmem, B, warp - 2, lane, wait); break;
            case 4: if constexpr (M >= 4) ClusterEpilogue<ROWS, 4>::run(P, S, cluster, rank, smem, tmem, B, warp - 2, lane, wait); break;
            default: break;
        }
        __syncwarp();
    }
    // After a normal run every copy between the CTAs has been waited for where it landed; after an abort some may be on their
    // way: their latency is waited out.
    __syncthreads();
    if (s_abort) {
        const uint64_t t0 = ptx::globaltimer_ns();
        while (ptx::globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::cluster_sync_all();
    if (warp == 1) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem, 128);
    }
}
