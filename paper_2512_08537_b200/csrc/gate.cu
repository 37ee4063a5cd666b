// Entropy gate + stream compaction for sm_100a.
//
// Kernel 1 (gate_rows_kernel): 4 to 32 lanes per token. The whole bf16 row is fetched with
// 128-bit streaming loads into registers (one HBM pass), the row maximum is taken with packed
// bf16x2 max, then S = sum 2^t and T = sum t 2^t with t = (x - m) log2(e) are accumulated in
// fp32, and H = ln S - ln2 * T / S. One lane writes the mask byte (and the entropy, if asked)
// and each block leaves its number of kept tokens in a small scratch array.
// Kernel 2 (compact_kernel): every block sums the counts of the blocks before it and writes the
// ascending token ids of its own contiguous token range (ballot + prefix), the last block
// writes the total.
//
// Definition being computed: the softmax-row entropy indicator of the paper's entropy-informed
// speculative decoding (H = -L_entropy of one row, natural log) and Algorithm 1's threshold test
// (a token is dropped iff H < tau).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <string.h>
#include <math_constants.h>
#include <stdint.h>

#include <atomic>
#include <mutex>
#include <type_traits>

#include "../../include/ardiff.h"
#include "common.cuh"
#include "gate_plan.h"

namespace {

constexpr int kGateThreads = 256;
constexpr int kGateWarps = kGateThreads / 32;
constexpr int kMaxGateBlocks = 4096;  // capacity of the per-device block-count scratch
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

__device__ __forceinline__ uint4 ld_stream_v4(const uint4* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// NaN-propagating packed max of two bf16 pairs held in 32-bit words
__device__ __forceinline__ uint32_t max_bf16x2_nan(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("max.NaN.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

// over the G lanes that share a row
template <int G = 32>
__device__ __forceinline__ float warp_max_nan(float v) {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
        float other = __shfl_xor_sync(0xffffffffu, v, o);
        // NaN-propagating max
        v = (v != v || other != other) ? CUDART_NAN_F : fmaxf(v, other);
    }
    return v;
}

template <int G = 32>
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// accumulate one 32-bit word (two bf16 values) into S and T; mneg = -m*log2e
__device__ __forceinline__ void acc_word(uint32_t w, float mneg, float& S, float& T) {
    float t0 = fmaf(bf16_lo(w), kLog2e, mneg);
    float t1 = fmaf(bf16_hi(w), kLog2e, mneg);
    float e0 = ex2_approx(t0);
    float e1 = ex2_approx(t1);
    S += e0;
    S += e1;
    T = fmaf(t0, e0, T);
    T = fmaf(t1, e1, T);
}

// the same for words that may hold -inf (fill, or a real channel): e is 0 there, and t, which e multiplies, stays finite.
// NaN, +inf and rows of -inf alone still give S = NaN through the row maximum.
__device__ __forceinline__ void acc_word_safe(uint32_t w, float mneg, float& S, float& T) {
    float t0 = fmaf(bf16_lo(w), kLog2e, mneg);
    float t1 = fmaf(bf16_hi(w), kLog2e, mneg);
    float e0 = ex2_approx(t0);
    float e1 = ex2_approx(t1);
    S += e0;
    S += e1;
    T = fmaf(fmaxf(t0, -1e30f), e0, T);
    T = fmaf(fmaxf(t1, -1e30f), e1, T);
}

// (S, T) of one 16-byte chunk of such words.
__device__ __forceinline__ float2 chunk_sums(const uint4& v, float mneg) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    float s[4], t = 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float t0 = fmaf(bf16_lo(w[q]), kLog2e, mneg), t1 = fmaf(bf16_hi(w[q]), kLog2e, mneg);
        const float e0 = ex2_approx(t0), e1 = ex2_approx(t1);
        s[q] = e0 + e1;
        const float p0 = fmaxf(t0, -1e30f);
        t = q == 0 ? p0 * e0 : fmaf(p0, e0, t);
        t = fmaf(fmaxf(t1, -1e30f), e1, t);
    }
    return make_float2((s[0] + s[1]) + (s[2] + s[3]), t);
}
// Sum of f(0) .. f(NCH - 1) as a tree over the bits of the index, the highest first. Chunk l + G j of a row sits with lane l,
// and the G lanes are added the same way (warp_sum), so a narrow row's sums are one tree over its chunks however many lanes
// hold it: its entropy does not depend, to the bit, on how many rows the call has (see few_rows). It is also the more exact
// order: one chain over a lane's 64 elements was off by 5.3e-8 of the norm at 16384 rows of 256, the tree is by 4.0e-8.
// A part of the tree whose first index is not wanted(j) holds nothing and is left out (272 channels use 34 of 64 chunks).
template <int NCH, int J = 0, int STEP = 1, typename F, typename W>
__device__ __forceinline__ float2 chunk_tree(F&& f, W&& wanted) {
    if constexpr (STEP >= NCH) {
        return f(std::integral_constant<int, J>());
    } else {
        float2 a = chunk_tree<NCH, J, 2 * STEP>(f, wanted);
        if constexpr (J + STEP < NCH) {
            if (wanted(J + STEP)) {
                const float2 b = chunk_tree<NCH, J + STEP, 2 * STEP>(f, wanted);
                a.x += b.x;
                a.y += b.y;
            }
        }
        return a;
    }
}

// Rows of a width that is no multiple of 8 start at any even address. They are read as the 16-byte chunks that cover
// them: the first chunk starts with `head` elements of the row before, the last one ends with elements of the row
// after; both are replaced by -inf once the chunk has arrived. 65536 x 777: 57 us (1.8 TB/s) with scalar loads in two
// passes, 39 us this way, 34 to 37 us with the tests for the matrix's edges and for the two partial chunks out of the loop
// over the chunks (bound by instruction issue).
constexpr uint32_t kFill = 0xff80ff80u;
struct RowSpan {
    const uint4* base;       // first chunk
    int nch, head;
};
// (width: channels; of aligned rows chunks)
template <bool RAGGED>
__device__ __forceinline__ RowSpan row_span(const void* feat, int64_t row, int32_t width) {
    if (!RAGGED) return RowSpan{static_cast<const uint4*>(feat) + row * (int64_t)width, width, 0};
    const uintptr_t at = reinterpret_cast<uintptr_t>(feat) + (uintptr_t)row * (uintptr_t)width * 2;
    const int head = (int)(at & 15u) / 2;
    return RowSpan{reinterpret_cast<const uint4*>(at & ~(uintptr_t)15), (head + width + 7) / 8, head};
}
// A partial chunk of a row at an edge of the matrix, element by element: nothing outside the caller's array is touched.
__device__ __noinline__ uint4 load_edge_chunk(const uint4* base, int head, int c, int32_t d) {
    const uint16_t* e = reinterpret_cast<const uint16_t*>(base + c);
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        w[q] = kFill;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = 8 * c + 2 * q + h - head;
            if (i >= 0 && i < d) w[q] = (w[q] & (h ? 0x0000ffffu : 0xffff0000u)) | ((uint32_t)e[2 * q + h] << (16 * h));
        }
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}
template <bool RAGGED>
__device__ __forceinline__ uint4 load_chunk(const RowSpan& r, int c, int32_t d, bool edge) {
    if (RAGGED && edge && (c == 0 || c == r.nch - 1)) return load_edge_chunk(r.base, r.head, c, d);
    return ld_stream_v4(r.base + c);
}
// elements lo .. hi - 1 of a chunk kept, the others -inf
__device__ __forceinline__ uint4 keep_elements(uint4 v, int lo, int hi) {
    uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (2 * q < lo || 2 * q >= hi) w[q] = (w[q] & 0xffff0000u) | 0xff80u;
        if (2 * q + 1 < lo || 2 * q + 1 >= hi) w[q] = (w[q] & 0x0000ffffu) | 0xff800000u;
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}
template <bool RAGGED>
__device__ __forceinline__ uint4 own_elements(uint4 v, const RowSpan& r, int c, int32_t d) {
    if (RAGGED && (c == 0 || c == r.nch - 1)) return keep_elements(v, c == 0 ? r.head : 0, min(8, r.head + d - 8 * c));
    return v;
}

// Whether a row's chunks may stick out of the matrix: fewer than 8 elements before it or after it.
template <bool RAGGED>
__device__ __forceinline__ bool edge_row(int64_t row, int64_t n, int32_t d) {
    return RAGGED && (row * d < 8 || (n - 1 - row) * d < 8);
}

// Slow exact-semantics path for one row: used when the fast path meets a non-finite
// intermediate (a -inf channel makes t*e = -inf*0). Re-reads the row from memory (rare), so the
// register-resident copy of the fast path never needs an address. Terms with e == 0 contribute 0.
__device__ __noinline__ float row_entropy_careful(const uint4* row, int nchunks, int lane, float m) {
    float S = 0.f, T = 0.f;
    const float mneg = -m * kLog2e;
    for (int c = lane; c < nchunks; c += 32) {
        const uint4 v = ld_stream_v4(row + c);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float t0 = fmaf(bf16_lo(w[q]), kLog2e, mneg), t1 = fmaf(bf16_hi(w[q]), kLog2e, mneg);
            float e0 = ex2_approx(t0), e1 = ex2_approx(t1);
            S += e0 + e1;
            if (e0 > 0.f || e0 != e0) T = fmaf(t0, e0, T);
            if (e1 > 0.f || e1 != e1) T = fmaf(t1, e1, T);
        }
    }
    S = warp_sum(S);
    T = warp_sum(T);
    return logf(S) - kLn2 * (T / S);
}

// Entropy of the aligned row that a warp holds in v (NCH 16-byte chunks per lane). Each chunk is refilled with the warp's
// NEXT row as soon as the exponentials of the current row have consumed it, so a warp always has loads in flight while
// it computes (with 128 registers per thread only 16 warps fit an SM: they cannot hide HBM latency by
// switching alone). Plain pointers and the chunk count as an argument: the same through RowSpan and d / 8 took 77 us
// instead of 55 at 16384 x 8192.
template <int NCH>
__device__ __forceinline__ float whole_row_entropy(uint4 (&v)[NCH], const uint4* row, const uint4* next_row,
                                                   bool has_next, int32_t nchunks, int lane) {
    // row maximum (packed, exact in bf16)
    uint32_t mx = kFill;
#pragma unroll
    for (int j = 0; j < NCH; ++j) {
        mx = max_bf16x2_nan(mx, max_bf16x2_nan(max_bf16x2_nan(v[j].x, v[j].y), max_bf16x2_nan(v[j].z, v[j].w)));
    }
    float ml = bf16_lo(mx), mh = bf16_hi(mx);
    float m = (ml != ml || mh != mh) ? CUDART_NAN_F : fmaxf(ml, mh);
    m = warp_max_nan(m);
    const float mneg = -m * kLog2e;
    float S = 0.f, T = 0.f;
#pragma unroll
    for (int j = 0; j < NCH; ++j) {
        const int c = lane + 32 * j;
        if (c < nchunks) {
            acc_word(v[j].x, mneg, S, T);
            acc_word(v[j].y, mneg, S, T);
            acc_word(v[j].z, mneg, S, T);
            acc_word(v[j].w, mneg, S, T);
            if (has_next) v[j] = ld_stream_v4(next_row + c);
        }
    }
    S = warp_sum(S);
    T = warp_sum(T);
    float H = logf(S) - kLn2 * (T / S);
    if (H != H) {
        // a -inf channel (t*e = -inf*0) lands here, as do genuinely undefined rows
        H = row_entropy_careful(row, nchunks, lane, m);
    }
    return H;
}
template <int NCH>
__device__ __forceinline__ void load_whole_row(uint4 (&v)[NCH], const uint4* row, int32_t nchunks, int lane) {
#pragma unroll
    for (int j = 0; j < NCH; ++j) {
        const int c = lane + 32 * j;
        v[j] = c < nchunks ? ld_stream_v4(row + c) : make_uint4(kFill, kFill, kFill, kFill);
    }
}

// The least chunk counts that the instances of dispatch_row serve, and the first of a lane's chunks that a row's last one may
// be (a row of a width that is no multiple of 8 may have one less than others of it). Instances of 5 and 7 chunks a lane, and
// the last chunk looked for in two of them instead of in the upper half: 65536 x 777 33.2 -> 32.3 us, 500000 x 777 210 -> 203,
// 65536 x 800 27.5 -> 26.8. (At 8 a lane the upper half: two take 36.2 us at 65536 x 900, five 35.4.)
__host__ __device__ constexpr int least_chunks(int nch, int g) {
    return g == 4 ? (nch == 2 ? 1 : nch == 4 ? 9 : 17)
         : g == 8 ? 33
         : g == 16 ? 16 * (nch - 1) + 1
         : nch <= 2 ? 32 * (nch - 1) + 1 : nch == 4 ? 65 : nch == 8 ? 129 : nch == 32 ? 769 : 32 * (nch - 4) + 1;
}
__host__ __device__ constexpr int last_chunk_from(int nch, int g) {
    return nch == 8 && g == 16 ? 3 : least_chunks(nch, g) < 2 ? 0 : (least_chunks(nch, g) - 2) / g;
}

// The same for rows at any even address (RAGGED) and for 32 / G rows to a warp, G lanes each. Where rows share a warp, what
// a row costs beside its elements (three reductions by shuffle, a logarithm, a division, the loop) is paid once for all of
// them: one row per warp takes 242 us for 2^20 x 64 and 20 us for 65536 x 256, this 43 and 12. `step` rows lie between a
// lane's row and its next one.
template <int NCH, int G, bool RAGGED>
__device__ __forceinline__ float resident_row_entropy(uint4 (&v)[NCH], const RowSpan& row, const RowSpan& next, int step,
                                                      bool has_next, bool next_edge, int32_t width, int l) {
    if (RAGGED) {
        if (l == 0) v[0] = keep_elements(v[0], row.head, 8);
        const int last = row.nch - 1, keep = row.head + width - 8 * last;
#pragma unroll
        for (int j = last_chunk_from(NCH, G); j < NCH; ++j)
            if (l + G * j == last) v[j] = keep_elements(v[j], 0, keep);
    }
    uint32_t mx = kFill;
#pragma unroll
    for (int j = 0; j < NCH; ++j) {
        mx = max_bf16x2_nan(mx, max_bf16x2_nan(max_bf16x2_nan(v[j].x, v[j].y), max_bf16x2_nan(v[j].z, v[j].w)));
    }
    float ml = bf16_lo(mx), mh = bf16_hi(mx);
    float m = (ml != ml || mh != mh) ? CUDART_NAN_F : fmaxf(ml, mh);
    m = warp_max_nan<G>(m);
    const float mneg = -m * kLog2e;
    float S = 0.f, T = 0.f;
    const int lo = RAGGED && next_edge ? 1 : 0, hi = !has_next ? 0 : RAGGED && next_edge ? next.nch - 1 : next.nch;
    auto refill = [&](uint4& w, int c, bool first_chunk) {
        // by the distance from this row: fewer registers than the next row's own pointer (16384 x 1024 11.3 us, not 12.3)
        if (!RAGGED && has_next && c < row.nch) w = ld_stream_v4(row.base + (int64_t)step * row.nch + c);
        // neighbouring rows may differ by a chunk; at an edge the partial chunks follow after the others
        if (RAGGED) {
            w = make_uint4(kFill, kFill, kFill, kFill);
            if (c < hi && (!first_chunk || c >= lo)) w = ld_stream_v4(next.base + c);
        }
    };
    if constexpr (NCH * G <= 128) {
        const float2 sums = chunk_tree<NCH>([&](auto J) {
            constexpr int j = decltype(J)::value;
            const int c = l + G * j;
            float2 x = make_float2(0.f, 0.f);
            if (c < row.nch) x = chunk_sums(v[j], mneg);
            refill(v[j], c, j == 0);
            return x;
        }, [&](int j) { return RAGGED || l + G * j < row.nch; });      // (a ragged row's next one may need the chunk)
        S = sums.x;
        T = sums.y;
    } else {
#pragma unroll
        for (int j = 0; j < NCH; ++j) {
            const int c = l + G * j;
            if (c < row.nch) {
                acc_word_safe(v[j].x, mneg, S, T);
                acc_word_safe(v[j].y, mneg, S, T);
                acc_word_safe(v[j].z, mneg, S, T);
                acc_word_safe(v[j].w, mneg, S, T);
            }
            refill(v[j], c, j == 0);
        }
    }
    if (RAGGED && has_next && next_edge) {
#pragma unroll
        for (int j = 0; j < NCH; ++j)
            if (l + G * j == 0 || l + G * j == next.nch - 1) v[j] = load_edge_chunk(next.base, next.head, l + G * j, width);
    }
    S = warp_sum<G>(S);
    T = warp_sum<G>(T);
    return logf(S) - kLn2 * (T / S);
}

template <int NCH, int G, bool RAGGED>
__device__ __forceinline__ void load_resident_row(uint4 (&v)[NCH], const RowSpan& row, int32_t width, bool edge, bool have,
                                                  int l) {
#pragma unroll
    for (int j = 0; j < NCH; ++j) {
        const int c = l + G * j;
        v[j] = have && c < row.nch ? load_chunk<RAGGED>(row, c, width, edge) : make_uint4(kFill, kFill, kFill, kFill);
    }
}

// f(row, its entropy, whether this lane answers for it) over rows begin + first row of the warp .. end - 1 of n, NCH chunks
// per lane and G lanes per row, in registers. `width` is d of ragged rows, the chunk count of aligned ones.
template <int NCH, int G, bool RAGGED, typename F>
__device__ __forceinline__ void for_each_row(const void* __restrict__ feat, int64_t begin, int64_t end, int64_t n,
                                             int32_t width, int warp, int lane, F&& f) {
    uint4 v[NCH];
    if constexpr (!RAGGED && NCH * G > 128) {
        const uint4* base = static_cast<const uint4*>(feat);
        if (begin + warp < end) load_whole_row(v, base + (begin + warp) * (int64_t)width, width, lane);
        for (int64_t i = begin + warp; i < end; i += kGateWarps) {
            const uint4* row = base + i * (int64_t)width;
            f(i, whole_row_entropy(v, row, row + (int64_t)kGateWarps * width, i + kGateWarps < end, width, lane), lane == 0);
        }
    } else {
        constexpr int R = 32 / G, STEP = kGateWarps * R;         // rows of a warp, of the CTA
        const int l = lane % G, sub = lane / G;
        auto edge = [&](int64_t i) { return edge_row<RAGGED>(i, n, width); };
        const int64_t first = begin + warp * R + sub;
        RowSpan row = row_span<RAGGED>(feat, first, width);
        load_resident_row<NCH, G, RAGGED>(v, row, width, edge(first), first < end, l);
        for (int64_t i0 = begin + warp * R; i0 < end; i0 += STEP) {
            const int64_t i = i0 + sub, nx = i + STEP;
            const RowSpan next = row_span<RAGGED>(feat, nx, width);
            const float H = resident_row_entropy<NCH, G, RAGGED>(v, row, next, STEP, nx < end, edge(nx), width, l);
            row = next;
            f(i, H, l == 0 && i < end);
        }
    }
}

// Count, sum and sum of squares (fp64) of the entropies a CTA has seen, one slot per warp, merged in warp order.
struct WarpStats { double n, s, q; };
__device__ __forceinline__ void cta_merge_stats(const WarpStats& mine, int warp, int lane, double* out3) {
    __shared__ double s_st[kGateWarps][3];
    if (lane == 0) { s_st[warp][0] = mine.n; s_st[warp][1] = mine.s; s_st[warp][2] = mine.q; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double n = 0, sm = 0, q = 0;
        for (int w = 0; w < kGateWarps; ++w) { n += s_st[w][0]; sm += s_st[w][1]; q += s_st[w][2]; }
        out3[0] = n; out3[1] = sm; out3[2] = q;
    }
}

// G lanes per token, row resident in registers: NCH 16-byte chunks per lane.
template <int NCH, int G, bool RAGGED>
__global__ void __launch_bounds__(kGateThreads)
gate_rows_kernel(const void* __restrict__ feat, int64_t n, int32_t width, float tau,
                 uint8_t* __restrict__ mask, float* __restrict__ entropy,
                 int32_t* __restrict__ block_counts, double* __restrict__ cta_stats, int64_t tokens_per_block) {
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    // the compaction kernel may be launched as soon as every block of this grid has started: its launch
    // latency then hides under this kernel's tail (it waits for this grid's completion before reading)
    asm volatile("griddepcontrol.launch_dependents;");
    const int64_t t_begin = (int64_t)blockIdx.x * tokens_per_block;
    const int64_t t_end = min(n, t_begin + tokens_per_block);
    int kept = 0;
    WarpStats st{0.0, 0.0, 0.0};
    for_each_row<NCH, G, RAGGED>(feat, t_begin, t_end, n, width, warp, lane, [&](int64_t tok, float H, bool mine) {
        const bool keep = (H >= tau);  // false for NaN
        if (mine) {
            if (mask) mask[tok] = keep ? 1 : 0;
            if (entropy) entropy[tok] = H;
        }
        // (lane 0 speaks for the warp at the end: where a row has all lanes they all count it)
        if (G == 32 || mine) {
            kept += keep ? 1 : 0;
            st.n += 1.0; st.s += (double)H; st.q += (double)H * (double)H;
        }
    });
    if (G < 32) {                            // the warp's rows together, in a fixed order
#pragma unroll
        for (int o = 16; o >= G; o >>= 1) {
            kept += __shfl_xor_sync(0xffffffffu, kept, o);
            if (cta_stats) {
                st.n += __shfl_xor_sync(0xffffffffu, st.n, o);
                st.s += __shfl_xor_sync(0xffffffffu, st.s, o);
                st.q += __shfl_xor_sync(0xffffffffu, st.q, o);
            }
        }
    }
    // block count (lane 0 holds the warp's)
    __shared__ int s_cnt[kGateWarps];
    if (lane == 0) s_cnt[warp] = kept;
    __syncthreads();
    if (threadIdx.x == 0) {
        int tot = 0;
#pragma unroll
        for (int w = 0; w < kGateWarps; ++w) tot += s_cnt[w];
        if (block_counts) block_counts[blockIdx.x] = tot;
    }
    if (cta_stats) cta_merge_stats(st, warp, lane, cta_stats + 3 * (size_t)blockIdx.x);
}

// Block-prefix form (Algorithm 1, Step 1, in one pass over the features): a CTA owns whole draft blocks. Its
// warps leave the row entropies in shared memory; then one thread per draft block forms the token indicators
// (mean of the token's r row entropies, summed in row order), runs the prefix test, and writes mask, kept
// length and, if asked, the indicators. No row entropy goes through global memory unless the caller wants it.
template <int NCH, int G, bool RAGGED>
__global__ void __launch_bounds__(kGateThreads)
gate_blocks_kernel(const void* __restrict__ feat, int64_t n_tokens, int32_t r, int32_t gamma, int32_t width,
                   float tau, float* __restrict__ row_entropy, float* __restrict__ token_entropy,
                   uint8_t* __restrict__ mask, int32_t* __restrict__ block_len, int32_t* __restrict__ cta_counts,
                   int64_t blocks_per_cta, int64_t n_blocks) {
    extern __shared__ float s_H[];      // row entropies of this CTA's draft blocks
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    asm volatile("griddepcontrol.launch_dependents;");
    const int64_t b_begin = (int64_t)blockIdx.x * blocks_per_cta;
    const int64_t b_end = min(n_blocks, b_begin + blocks_per_cta);
    const int64_t t_begin = b_begin * gamma;
    const int64_t t_end = min(n_tokens, b_end * gamma);
    const int64_t r_begin = t_begin * r, r_end = t_end * r;
    for_each_row<NCH, G, RAGGED>(feat, r_begin, r_end, n_tokens * r, width, warp, lane, [&](int64_t i, float H, bool mine) {
        if (mine) {
            s_H[i - r_begin] = H;
            if (row_entropy) row_entropy[i] = H;
        }
    });
    __syncthreads();
    int kept_total = 0;
    const float inv = 1.0f / (float)r;
    for (int64_t b = b_begin + threadIdx.x; b < b_end; b += kGateThreads) {
        const int64_t t0 = b * gamma;
        const int64_t t1 = min(n_tokens, t0 + gamma);
        bool speculate = true;
        int kept = 0;
        for (int64_t t = t0; t < t1; ++t) {
            const float* src = s_H + (t - t_begin) * r;
            float acc = 0.f;
            for (int j = 0; j < r; ++j) acc += src[j];
            const float hs = acc * inv;
            if (token_entropy) token_entropy[t] = hs;
            if (speculate && !(hs >= tau)) speculate = false;   // H < tau, or NaN
            mask[t] = speculate ? 1 : 0;
            kept += speculate ? 1 : 0;
        }
        if (block_len) block_len[b] = kept;
        kept_total += kept;
    }
    __shared__ int s_cnt[kGateWarps];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) kept_total += __shfl_xor_sync(0xffffffffu, kept_total, o);
    if (lane == 0) s_cnt[warp] = kept_total;
    __syncthreads();
    if (threadIdx.x == 0) {
        int tot = 0;
        for (int w = 0; w < kGateWarps; ++w) tot += s_cnt[w];
        cta_counts[blockIdx.x] = tot;
    }
}

// Partial sums (S, T) of a lane whose maximum so far was `from`, brought to the larger maximum `to`. Where 2^D is 0 nothing
// is left of them, also when they are not finite: from * log2 e overflows for the type's lowest values, which serve as masks.
__device__ __forceinline__ void rescale_sums(float from, float to, float& S, float& T) {
    const float D = (from - to) * kLog2e;
    const float f = ex2_approx(D);
    T = f > 0.f ? (T + D * S) * f : 0.f;
    S = f > 0.f ? S * f : 0.f;
}

// Rows longer than the registers hold: still one pass with 128-bit loads. Every lane keeps a running maximum of its own
// share of the row and rescales its partial sums when the maximum grows
// (S <- S 2^D, T <- (T + D S) 2^D with D = (m_old - m_new) log2 e <= 0); the lanes' partials are merged the
// same way at the end. The next four chunks are asked for before the present four are worked on.
template <bool RAGGED>
__global__ void __launch_bounds__(kGateThreads)
gate_rows_long_kernel(const void* __restrict__ feat, int64_t n, int32_t d, float tau,
                      uint8_t* __restrict__ mask, float* __restrict__ entropy,
                      int32_t* __restrict__ block_counts, double* __restrict__ cta_stats, int64_t tokens_per_block) {
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    asm volatile("griddepcontrol.launch_dependents;");
    const int64_t t_begin = (int64_t)blockIdx.x * tokens_per_block;
    const int64_t t_end = min(n, t_begin + tokens_per_block);
    int kept = 0;
    WarpStats st{0.0, 0.0, 0.0};
    constexpr int G = 4;
    auto load_group = [&](uint4 (&v)[G], const RowSpan& row, bool edge, int c0) {
#pragma unroll
        for (int j = 0; j < G; ++j)
            v[j] = c0 + 32 * j < row.nch ? load_chunk<RAGGED>(row, c0 + 32 * j, d, edge) : make_uint4(kFill, kFill, kFill, kFill);
    };
    for (int64_t tok = t_begin + warp; tok < t_end; tok += kGateWarps) {
        const RowSpan row = row_span<RAGGED>(feat, tok, RAGGED ? d : d / 8);
        const bool edge = edge_row<RAGGED>(tok, n, d);
        float ml = -CUDART_INF_F, S = 0.f, T = 0.f;
        uint4 v[G], nv[G];
        load_group(v, row, edge, lane);
        for (int c0 = lane; c0 < row.nch; c0 += 32 * G) {
            load_group(nv, row, edge, c0 + 32 * G);
            if (RAGGED) {
#pragma unroll
                for (int j = 0; j < G; ++j) v[j] = own_elements<true>(v[j], row, c0 + 32 * j, d);
            }
            uint32_t mx = kFill;
#pragma unroll
            for (int j = 0; j < G; ++j)
                mx = max_bf16x2_nan(mx, max_bf16x2_nan(max_bf16x2_nan(v[j].x, v[j].y), max_bf16x2_nan(v[j].z, v[j].w)));
            const float a = bf16_lo(mx), b = bf16_hi(mx);
            const float mc = (a != a || b != b) ? CUDART_NAN_F : fmaxf(a, b);
            if (mc != mc) ml = CUDART_NAN_F;
            else if (mc > ml) {
                rescale_sums(ml, mc, S, T);
                ml = mc;
            }
            // a lane whose elements so far are all -inf has nothing to add (and no finite maximum to subtract)
            if (!RAGGED || ml != -CUDART_INF_F) {
                const float mneg = -ml * kLog2e;
#pragma unroll
                for (int j = 0; j < G; ++j) {
                    if (c0 + 32 * j < row.nch) {
                        if (RAGGED) {
                            acc_word_safe(v[j].x, mneg, S, T);
                            acc_word_safe(v[j].y, mneg, S, T);
                            acc_word_safe(v[j].z, mneg, S, T);
                            acc_word_safe(v[j].w, mneg, S, T);
                        } else {
                            acc_word(v[j].x, mneg, S, T);
                            acc_word(v[j].y, mneg, S, T);
                            acc_word(v[j].z, mneg, S, T);
                            acc_word(v[j].w, mneg, S, T);
                        }
                    }
                }
            }
#pragma unroll
            for (int j = 0; j < G; ++j) v[j] = nv[j];
        }
        const float m = warp_max_nan(ml);
        if (ml < m) rescale_sums(ml, m, S, T);      // bring this lane's partials to the row maximum
        S = warp_sum(S);
        T = warp_sum(T);
        float H = logf(S) - kLn2 * (T / S);
        if (RAGGED) {
            if (!(fabsf(m) < CUDART_INF_F)) H = CUDART_NAN_F;       // NaN, +inf, or -inf alone
        } else if (H != H) {
            H = row_entropy_careful(row.base, row.nch, lane, m);
        }
        const bool keep = (H >= tau);
        if (lane == 0) {
            if (mask) mask[tok] = keep ? 1 : 0;
            if (entropy) entropy[tok] = H;
        }
        kept += keep ? 1 : 0;
        st.n += 1.0; st.s += (double)H; st.q += (double)H * (double)H;
    }
    __shared__ int s_cnt[kGateWarps];
    if (lane == 0) s_cnt[warp] = kept;
    __syncthreads();
    if (threadIdx.x == 0) {
        int tot = 0;
        for (int w = 0; w < kGateWarps; ++w) tot += s_cnt[w];
        if (block_counts) block_counts[blockIdx.x] = tot;
    }
    if (cta_stats) cta_merge_stats(st, warp, lane, cta_stats + 3 * (size_t)blockIdx.x);
}

// Stable compaction: block b writes the ids of kept tokens of its own range at the offset given
// by the counts of blocks 0..b-1.
__global__ void __launch_bounds__(kGateThreads)
compact_kernel(const uint8_t* mask, int64_t n, const int32_t* block_counts, int64_t tokens_per_block, int32_t* idx,
               int32_t* count, const double* cta_stats, double* stats_out3) {
    __shared__ int s_warp[kGateWarps];
    __shared__ int s_base;
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    // launched with programmatic stream serialization: its blocks may be resident before the kernel that
    // writes mask and block_counts has finished; nothing of that kernel's output is read before this wait, and none of it
    // through the read-only path (no __restrict__), which wants data that does not change while this kernel runs
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // What a thread reads first is asked for at once, and a tile's mask before the tile ahead of it is written: across the
    // barriers the compiler moves no load of data that may change. (us, gate / with statistics, those before all else and
    // loads where they are used: 8192 x 64 5.2 / 8.0, 8192 x 2048 11.2 / 12.5, 8192 x 16384 51.6 / 53.6, 2^20 x 64 41.6 / 44.4; now
    // 5.0 / 7.8, 11.0 / 12.2, 51.2 / 53.3, 41.1 / 43.4.)
    const int64_t t_begin = (int64_t)blockIdx.x * tokens_per_block;
    const int64_t t_end = min(n, t_begin + tokens_per_block);
    bool next = t_begin + threadIdx.x < t_end && mask[t_begin + threadIdx.x] != 0;
    // offset = sum of counts of the blocks before this one
    int part = 0;
    for (int b = threadIdx.x; b < (int)blockIdx.x; b += kGateThreads) part += block_counts[b];
    const int own = block_counts[blockIdx.x];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if (lane == 0) s_warp[warp] = part;
    __syncthreads();
    if (threadIdx.x == 0) {
        int tot = 0;
        for (int w = 0; w < kGateWarps; ++w) tot += s_warp[w];
        s_base = tot;
        if (blockIdx.x == gridDim.x - 1) *count = tot + own;
    }
    __syncthreads();
    int base = s_base;
    for (int64_t t0 = t_begin; t0 < t_end; t0 += kGateThreads) {
        const int64_t tok = t0 + threadIdx.x;
        const bool keep = next;
        next = tok + kGateThreads < t_end && mask[tok + kGateThreads] != 0;
        const unsigned bal = __ballot_sync(0xffffffffu, keep);
        const int rank = __popc(bal & ((1u << lane) - 1u));
        __syncthreads();  // s_warp reuse
        if (lane == 0) s_warp[warp] = __popc(bal);
        __syncthreads();
        int woff = 0, tot = 0;
#pragma unroll
        for (int w = 0; w < kGateWarps; ++w) {
            const int cw = s_warp[w];
            woff += (w < warp) ? cw : 0;
            tot += cw;
        }
        if (keep) idx[base + woff + rank] = (int32_t)tok;
        base += tot;
    }
    // Threshold statistics of the entropies (the tau equation): the per-CTA partial sums of the row kernel,
    // merged in a fixed order (lane-strided, then a fixed tree) so that the result is reproducible run to run. (Last: nothing in
    // this kernel waits for them, and one lane's square root in 64 bits is long.)
    if (cta_stats && blockIdx.x == 0 && warp == 0) {
        double cn = 0, cs = 0, cq = 0;
        for (int b = lane; b < (int)gridDim.x; b += 32) {
            cn += cta_stats[3 * b]; cs += cta_stats[3 * b + 1]; cq += cta_stats[3 * b + 2];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            cn += __shfl_xor_sync(0xffffffffu, cn, o);
            cs += __shfl_xor_sync(0xffffffffu, cs, o);
            cq += __shfl_xor_sync(0xffffffffu, cq, o);
        }
        if (lane == 0) {
            const double mean = cs / cn;
            const double var = fmax(cq / cn - mean * mean, 0.0);
            stats_out3[0] = mean;
            stats_out3[1] = sqrt(var);
            stats_out3[2] = 0.3 * mean - 0.1 * sqrt(var);
        }
    }
}

__global__ void write_zero_count_kernel(int32_t* count) { *count = 0; }

// ---- per-device scratch: one slice per stream ---------------------------------------------------
// A slice holds what the two kernels of a call hand to each other: per-block kept counts and, for the calls
// that ask for the threshold statistics, per-block partial sums. Two gate calls may run on the GPU at the same
// time only when they were enqueued on different streams, so every stream gets a slice of its own (calls on
// one stream are ordered and share theirs). The table holds kGateSlices - 1 streams per device; any further
// stream shares the last slice.
constexpr int kMaxDevices = 64;
constexpr int kGateSlices = 32;
constexpr size_t kSliceBytes = (size_t)kMaxGateBlocks * (sizeof(int32_t) + 3 * sizeof(double));
struct GateScratch {
    char* base = nullptr;
    int n_sm = 0;
    int used = 0;
    cudaStream_t key[kGateSlices];
};
GateScratch g_scratch[kMaxDevices];
std::mutex g_scratch_mutex;

void load_gate_kernels();

int gate_scratch(cudaStream_t st, int32_t** counts, double** stats, int* sms) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return ARDIFF_ERR_CUDA;
    if (dev < 0 || dev >= kMaxDevices) return ARDIFF_ERR_UNSUPPORTED;
    std::lock_guard<std::mutex> lock(g_scratch_mutex);
    GateScratch& g = g_scratch[dev];
    if (!g.base) {
        int n_sm = 0;
        if (cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return ARDIFF_ERR_CUDA;
        void* p = nullptr;
        if (cudaMalloc(&p, kSliceBytes * kGateSlices) != cudaSuccess) {
            (void)cudaGetLastError();
            return ARDIFF_ERR_NOMEM;
        }
        load_gate_kernels();
        g.n_sm = n_sm;
        g.base = static_cast<char*>(p);
    }
    int slice = -1;
    for (int i = 0; i < g.used; ++i)
        if (g.key[i] == st) { slice = i; break; }
    if (slice < 0) {
        if (g.used < kGateSlices - 1) {
            g.key[g.used] = st;
            slice = g.used++;
        } else {
            slice = kGateSlices - 1;
        }
    }
    char* sl = g.base + (size_t)slice * kSliceBytes;
    *stats = reinterpret_cast<double*>(sl);                                        // 8-byte aligned part first
    *counts = reinterpret_cast<int32_t*>(sl + (size_t)kMaxGateBlocks * 3 * sizeof(double));
    *sms = g.n_sm;
    return ARDIFF_OK;
}

// compact_kernel behind programmatic stream serialization (see the wait at its top)
cudaError_t launch_compact(int grid, cudaStream_t st, const uint8_t* mask, int64_t n, const int32_t* block_counts,
                           int64_t tpb, int32_t* idx, int32_t* count, const double* cta_stats, double* out3) {
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3(grid); cfg.blockDim = dim3(kGateThreads); cfg.dynamicSmemBytes = 0; cfg.stream = st;
    cfg.attrs = at; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, compact_kernel, mask, n, block_counts, tpb, idx, count, cta_stats, out3);
}

// 16-byte pieces that a row of d channels may cover: rows of a width that is no multiple of 8 start anywhere in a piece.
// Up to kResidentChunks the row is held in registers, above it the long-row kernel runs.
constexpr int kResidentChunks = 1024;
int row_chunks(int32_t d) { return d % 8 == 0 ? d / 8 : (d + 14) / 8; }
// what the kernels of resident rows take as their width
int32_t kernel_width(int32_t d) { return d % 8 == 0 ? d / 8 : d; }

// The row kernel for rows of up to `chunks` sixteen-byte pieces: f(integral_constant<NCH>, integral_constant<G>). Narrow rows
// share a warp with 5 to 8 pieces per lane (fewer in the narrowest) and at least 4 lanes per row, so that a load still
// covers whole 32-byte sectors; above 128 pieces, and where there are few rows (`alone`), a row has a warp of its own.
template <typename F>
void dispatch_row(int chunks, bool alone, F&& f) {
    auto call = [&](auto nch, auto g) { f(nch, g); };
#define ROW(n, g) call(std::integral_constant<int, n>(), std::integral_constant<int, g>())
    if (alone && chunks <= 32) ROW(1, 32);
    else if (alone && chunks <= 64) ROW(2, 32);
    else if (alone && chunks <= 128) ROW(4, 32);
    else if (chunks <= 8) ROW(2, 4);
    else if (chunks <= 16) ROW(4, 4);
    else if (chunks <= 32) ROW(8, 4);
    else if (chunks <= 64) ROW(8, 8);
    else if (chunks <= 80) ROW(5, 16);
    else if (chunks <= 96) ROW(6, 16);
    else if (chunks <= 112) ROW(7, 16);
    else if (chunks <= 128) ROW(8, 16);
    else if (chunks <= 256) ROW(8, 32);
    else if (chunks <= 384) ROW(12, 32);
    else if (chunks <= 512) ROW(16, 32);
    else if (chunks <= 640) ROW(20, 32);
    else if (chunks <= 768) ROW(24, 32);
    else ROW(32, 32);
#undef ROW
}
constexpr int kRowClasses = 17;
int row_class(int chunks, bool alone) {
    const int up_to[kRowClasses - 4] = {8, 16, 32, 64, 80, 96, 112, 128, 256, 384, 512, 640, 768};
    if (alone && chunks <= 128) return kRowClasses - 3 + (chunks > 32) + (chunks > 64);
    int c = 0;
    while (c < kRowClasses - 4 && chunks > up_to[c]) ++c;
    return c;
}

// Whether n rows of d channels, narrow enough to share warps, get one each: a call of few rows lasts as long as the chain of
// one row's instructions, which is shorter with 32 lanes on it. Measured, alone / shared, us: 1000 x 256 4.1 / 4.8, 3000 x
// 256 5.0 / 5.4, 5000 x 256 6.0 / 6.3, 6000 x 256 6.6 / 6.4, 4000 x 1024 6.4 / 6.6, 5000 x 1024 7.4 / 7.5; 2000 x 128
// 4.3 / 4.5, 3000 x 128 5.0 / 4.8, 2000 x 65 5.0 / 5.4, 4000 x 65 6.4 / 6.1; 1500 x 64 4.3 / 4.4, 4000 x 64 5.3 / 4.8.
// Up to 64 aligned channels the two are even at the few rows and sharing wins from there on.
bool few_rows(int32_t d, int64_t n, int n_sm) {
    const int chunks = row_chunks(d);
    if (chunks > 128 || (chunks <= 8 && d % 8 == 0)) return false;
    const bool long_lanes = (chunks > 16 && chunks <= 64) || chunks > 96;      // 8 chunks per lane where warps are shared
    return n <= (int64_t)n_sm * (long_lanes ? 36 : 14);
}

// Launches the row kernel for any d.
void launch_rows(int grid, cudaStream_t st, const void* feat, int64_t n, int32_t d, float tau, uint8_t* mask,
                 float* entropy, int32_t* counts, double* cta_stats, int64_t tpb, bool alone) {
    const int chunks = row_chunks(d);
    if (chunks > kResidentChunks) {
        if (d % 8 == 0)
            gate_rows_long_kernel<false><<<grid, kGateThreads, 0, st>>>(feat, n, d, tau, mask, entropy, counts, cta_stats, tpb);
        else
            gate_rows_long_kernel<true><<<grid, kGateThreads, 0, st>>>(feat, n, d, tau, mask, entropy, counts, cta_stats, tpb);
        return;
    }
    dispatch_row(chunks, alone, [&](auto nch, auto g) {
        constexpr int NCH = decltype(nch)::value, G = decltype(g)::value;
        auto kern = d % 8 == 0 ? gate_rows_kernel<NCH, G, false> : gate_rows_kernel<NCH, G, true>;
        kern<<<grid, kGateThreads, 0, st>>>(feat, n, kernel_width(d), tau, mask, entropy, counts, cta_stats, tpb);
    });
}

// Resident blocks per SM of the row kernel that serves rows of d channels.
// One block per resident slot, i.e. a grid of exactly one wave, measured best: with more blocks the later
// waves start against a full memory system and the kernel grows a tail (32768 x 5120: 74.8 -> 68.6 us).
int rows_blocks_per_sm(int32_t d, bool alone) {
    static std::atomic<int> cache[2][kRowClasses + 1] = {};
    const int chunks = row_chunks(d);
    const bool ragged = d % 8 != 0;
    const int slot = chunks > kResidentChunks ? kRowClasses : row_class(chunks, alone);
    const int known = cache[ragged][slot].load(std::memory_order_relaxed);
    if (known > 0) return known;
    int occ = 0;
    cudaError_t e = cudaSuccess;
    auto ask = [&](auto kern) { e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kGateThreads, 0); };
    if (slot == kRowClasses) {
        if (ragged) ask(gate_rows_long_kernel<true>);
        else ask(gate_rows_long_kernel<false>);
    } else {
        dispatch_row(chunks, alone, [&](auto nch, auto g) {
            constexpr int NCH = decltype(nch)::value, G = decltype(g)::value;
            if (ragged) ask(gate_rows_kernel<NCH, G, true>);
            else ask(gate_rows_kernel<NCH, G, false>);
        });
    }
    if (e != cudaSuccess || occ < 1) {
        (void)cudaGetLastError();
        occ = 2;
    }
    if (occ > 8) occ = 8;
    cache[ragged][slot].store(occ, std::memory_order_relaxed);
    return occ;
}

// Loads every kernel that a gate call may launch on the current device (the runtime loads a kernel when it is first used,
// and takes device memory for it: 2 MB for all of these). So a device's first gate call is the only one that does so, and
// any other shape may follow inside a stream capture. (That first call takes 11 to 12 ms with and without this.)
void load_gate_kernels() {
    auto load = [](auto kern) {
        cudaFuncAttributes a;
        if (cudaFuncGetAttributes(&a, kern) != cudaSuccess) (void)cudaGetLastError();
    };
    for (int chunks : {8, 16, 32, 64, 80, 96, 112, 128, 256, 384, 512, 640, 768, kResidentChunks})
        for (bool alone : {false, true})
            if (!alone || chunks <= 128)
                dispatch_row(chunks, alone, [&](auto nch, auto g) {
                    constexpr int NCH = decltype(nch)::value, G = decltype(g)::value;
                    load(gate_rows_kernel<NCH, G, false>);
                    load(gate_rows_kernel<NCH, G, true>);
                    load(gate_blocks_kernel<NCH, G, false>);
                    load(gate_blocks_kernel<NCH, G, true>);
                });
    load(gate_rows_long_kernel<false>);
    load(gate_rows_long_kernel<true>);
    load(compact_kernel);
    load(write_zero_count_kernel);
    ardiff::load_prefix_kernel();
}

// Waves of blocks: one while a block's share of the input stays small (then ramp and tail dominate and a
// single wave is fastest), up to four once a block would stream more than 4 MB (then finer blocks even out
// the finish: 2^19 x 5120 is 1 % faster with four waves than with one).
int grid_waves(int64_t rows, int32_t d, int64_t resident_blocks) {
    const int64_t per_block = rows * (int64_t)d * 2 / (resident_blocks > 0 ? resident_blocks : 1);
    const int64_t w = per_block / (4ll << 20);
    return w < 1 ? 1 : (w > 4 ? 4 : (int)w);
}

int check_feat(const void* feat, int32_t d) {
    const bool vec = (d % 8 == 0);
    if (vec && (reinterpret_cast<uintptr_t>(feat) & 15u)) return ARDIFF_ERR_ALIGN;
    if (!vec && (reinterpret_cast<uintptr_t>(feat) & 1u)) return ARDIFF_ERR_ALIGN;
    return ARDIFF_OK;
}

}  // namespace

namespace ardiff {

// Shared by the allocating entry points and by variants that bring their own block-count
// scratch: validates, picks the row kernel, launches gate + compaction on `st`. With cta_stats and
// stats_out3 the entropies' mean, standard deviation and threshold are produced on the way.
int gate_launch(const void* feat, int64_t n, int32_t d, float tau, uint8_t* mask, int32_t* idx,
                int32_t* count, float* entropy, int32_t* block_counts, double* cta_stats, double* stats_out3,
                int max_blocks, int n_sm, cudaStream_t st) {
    if (!count) return ARDIFF_ERR_NULL;
    if (n < 0 || n >= (int64_t)1 << 31 || d < 1 || d > 65536) return ARDIFF_ERR_SHAPE;
    if (n == 0) {
        write_zero_count_kernel<<<1, 1, 0, st>>>(count);
        set_launch_count(1);
        return cudaGetLastError() == cudaSuccess ? ARDIFF_OK : ARDIFF_ERR_CUDA;
    }
    if (!feat || !mask || !idx || !block_counts) return ARDIFF_ERR_NULL;
    const int rc = check_feat(feat, d);
    if (rc != ARDIFF_OK) return rc;

    // contiguous token range per block; one block per resident slot of the GPU, each with at least 8 tokens (one per warp;
    // where warps are shared, one warp's worth: spread thin, few rows start their loads on as many SMs as there are)
    const bool alone = few_rows(d, n, n_sm);
    int64_t want = (int64_t)n_sm * rows_blocks_per_sm(d, alone);
    want *= grid_waves(n, d, want);
    if (want > max_blocks) want = max_blocks;
    int64_t tpb = (n + want - 1) / want;
    if (tpb < kGateWarps) tpb = kGateWarps;
    const int grid = (int)((n + tpb - 1) / tpb);

    launch_rows(grid, st, feat, n, d, tau, mask, entropy, block_counts, stats_out3 ? cta_stats : nullptr, tpb, alone);
    (void)launch_compact(grid, st, mask, n, block_counts, tpb, idx, count, stats_out3 ? cta_stats : nullptr,
                         stats_out3);
    set_launch_count(2);
    return cudaGetLastError() == cudaSuccess ? ARDIFF_OK : ARDIFF_ERR_CUDA;
}

// Row entropies only (no threshold, no compaction): entropy[i] = H of row i.
int entropy_rows_launch(const void* feat, int64_t rows, int32_t d, float* entropy, int n_sm, cudaStream_t st) {
    if (rows < 0 || rows >= (int64_t)1 << 31 || d < 1 || d > 65536) return ARDIFF_ERR_SHAPE;
    if (rows == 0) return ARDIFF_OK;
    if (!feat || !entropy) return ARDIFF_ERR_NULL;
    const int rc = check_feat(feat, d);
    if (rc != ARDIFF_OK) return rc;
    const bool alone = few_rows(d, rows, n_sm);
    int64_t want = (int64_t)n_sm * rows_blocks_per_sm(d, alone);
    want *= grid_waves(rows, d, want);
    int64_t tpb = (rows + want - 1) / want;
    if (tpb < kGateWarps) tpb = kGateWarps;
    const int grid = (int)((rows + tpb - 1) / tpb);
    launch_rows(grid, st, feat, rows, d, 0.f, nullptr, entropy, nullptr, nullptr, tpb, alone);
    return cudaGetLastError() == cudaSuccess ? ARDIFF_OK : ARDIFF_ERR_CUDA;
}

// The block-prefix gate in one pass over the features (gate_blocks_kernel + compaction). Returns
// ARDIFF_ERR_UNSUPPORTED, with nothing launched, when the shape does not fit it: rows that do not fit the
// registers, or a draft block whose row entropies exceed a CTA's shared memory.
int gate_blocks_fused_launch(const void* feat, int64_t n, int32_t r, int32_t d, int32_t gamma, float tau,
                             float* row_entropy, float* token_entropy, uint8_t* mask, int32_t* idx, int32_t* count,
                             int32_t* block_len, int32_t* cta_counts, int max_blocks, int n_sm, cudaStream_t st) {
    if (row_chunks(d) > kResidentChunks || (int64_t)gamma * r > kMaxRowsPerCta) return ARDIFF_ERR_UNSUPPORTED;
    const int rc = check_feat(feat, d);
    if (rc != ARDIFF_OK) return rc;
    const int64_t n_blocks = (n + gamma - 1) / gamma;
    const int64_t rows = n * r;
    const int64_t rows_per_block = (int64_t)gamma * r;
    // with more rows in a draft block than the CTA has warps, shared warps take fewer rounds (8 blocks of 128 rows of 1024
    // channels: 15.1 us, 16.7 with one row per warp; 64 blocks of 8 rows: 6.2 and 5.8)
    const bool alone = rows_per_block <= kGateWarps && few_rows(d, rows, n_sm);
    int64_t want = (int64_t)n_sm * rows_blocks_per_sm(d, alone);
    want *= grid_waves(rows, d, want);
    int64_t rows_per_round = 0;
    dispatch_row(row_chunks(d), alone, [&](auto, auto g) { rows_per_round = kGateThreads / decltype(g)::value; });
    const DraftPlan plan = plan_draft_blocks(n_blocks, rows_per_block, rows_per_round, want, max_blocks);
    if (plan.grid == 0) return ARDIFF_ERR_UNSUPPORTED;               // too many CTAs for the count scratch
    const int grid = (int)plan.grid;
    const int64_t bpc = plan.blocks_per_cta;
    const size_t smem = (size_t)(bpc * rows_per_block) * sizeof(float);
    cudaError_t e = cudaSuccess;
    dispatch_row(row_chunks(d), alone, [&](auto nch, auto g) {
        constexpr int NCH = decltype(nch)::value, G = decltype(g)::value;
        auto kern = d % 8 == 0 ? gate_blocks_kernel<NCH, G, false> : gate_blocks_kernel<NCH, G, true>;
        if (smem > 48 * 1024) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
        if (e == cudaSuccess)
            kern<<<grid, kGateThreads, smem, st>>>(feat, n, r, gamma, kernel_width(d), tau,
                                                  row_entropy, token_entropy, mask, block_len, cta_counts, bpc,
                                                  n_blocks);
    });
    if (e != cudaSuccess) return ARDIFF_ERR_CUDA;
    (void)launch_compact(grid, st, mask, n, cta_counts, bpc * gamma, idx, count, nullptr, nullptr);
    set_launch_count(2);
    return cudaGetLastError() == cudaSuccess ? ARDIFF_OK : ARDIFF_ERR_CUDA;
}

// Stable compaction of a mask whose per-block kept counts (blocks of tokens_per_block tokens) are known.
int compact_launch(const uint8_t* mask, int64_t n, const int32_t* block_counts, int64_t tokens_per_block, int grid,
                   int32_t* idx, int32_t* count, cudaStream_t st) {
    (void)launch_compact(grid, st, mask, n, block_counts, tokens_per_block, idx, count, nullptr, nullptr);
    return cudaGetLastError() == cudaSuccess ? ARDIFF_OK : ARDIFF_ERR_CUDA;
}

int gate_scratch_get(cudaStream_t st, int32_t** counts, int* max_blocks, int* sms) {
    *max_blocks = kMaxGateBlocks;
    double* stats = nullptr;
    return gate_scratch(st, counts, &stats, sms);
}

void gate_load_kernels() { load_gate_kernels(); }

int write_zero_count(int32_t* count, cudaStream_t st) {
    write_zero_count_kernel<<<1, 1, 0, st>>>(count);
    return cudaGetLastError() == cudaSuccess ? ARDIFF_OK : ARDIFF_ERR_CUDA;
}

}  // namespace ardiff

namespace {
int gate_entry(const void* feat, int64_t n, int32_t d, float tau, uint8_t* mask, int32_t* idx, int32_t* count,
               float* entropy, double* stats_out3, void* stream) {
    int32_t* counts = nullptr;
    double* stats = nullptr;
    int sms = 0;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int rc = gate_scratch(st, &counts, &stats, &sms);
    if (rc != ARDIFF_OK) return rc;
    return ardiff::gate_launch(feat, n, d, tau, mask, idx, count, entropy, counts, stats, stats_out3,
                               kMaxGateBlocks, sms, st);
}
}  // namespace

extern "C" int ardiff_entropy_gate_ex(const void* feat, int64_t n, int32_t d, float tau,
                                      uint8_t* mask, int32_t* idx, int32_t* count, float* entropy,
                                      void* stream) {
    return gate_entry(feat, n, d, tau, mask, idx, count, entropy, nullptr, stream);
}

extern "C" int ardiff_entropy_gate(const void* feat, int64_t n, int32_t d, float tau, uint8_t* mask,
                                   int32_t* idx, int32_t* count, void* stream) {
    return gate_entry(feat, n, d, tau, mask, idx, count, nullptr, nullptr, stream);
}

extern "C" int ardiff_entropy_gate_stats(const void* feat, int64_t n, int32_t d, float tau, uint8_t* mask,
                                         int32_t* idx, int32_t* count, float* entropy, double* out3,
                                         void* stream) {
    if (!out3) return ARDIFF_ERR_NULL;
    if (n < 1) return ARDIFF_ERR_SHAPE;
    return gate_entry(feat, n, d, tau, mask, idx, count, entropy, out3, stream);
}
