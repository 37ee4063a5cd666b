// Later stages of the entropy-gated pipeline, built on the row-entropy kernel of gate.cu:
//   ardiff_entropy_gate_blocks  the early stop of Algorithm 1, Step 1 as written: per draft block, the
//                               first token whose indicator falls below tau drops itself and the rest
//                               of the block; the indicator is the mean of the token's row entropies
//                               (the entropy-loss equation's mean over rows and heads);
//   ardiff_tau_calibrate        the threshold equation tau = 0.3 mean(H) - 0.1 std(H);
//   ardiff_accept_prefix        Algorithm 1, Step 4: accepted draft length per block.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <atomic>

#include "../../include/ardiff.h"
#include "common.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int kThreads = 256;

// One thread per draft block: token indicators (mean over rows_per_token row entropies, summed in row
// order), prefix test, mask, kept length. A CTA covers blocks_per_cta consecutive blocks and leaves
// its kept-token count for the compaction pass.
__global__ void __launch_bounds__(kThreads)
block_prefix_kernel(const float* __restrict__ row_entropy, int64_t n, int32_t r, int32_t gamma, float tau,
                    float* __restrict__ token_entropy, uint8_t* __restrict__ mask, int32_t* __restrict__ block_len,
                    int32_t* __restrict__ cta_counts, int64_t blocks_per_cta, int64_t n_blocks) {
    __shared__ int s_cnt[kThreads / 32];
    int kept_total = 0;
    const int64_t b_begin = (int64_t)blockIdx.x * blocks_per_cta;
    const int64_t b_end = min(n_blocks, b_begin + blocks_per_cta);
    for (int64_t b = b_begin + threadIdx.x; b < b_end; b += kThreads) {
        const int64_t t0 = b * gamma;
        const int64_t t1 = min(n, t0 + gamma);
        bool speculate = true;
        int kept = 0;
        const float inv = 1.0f / (float)r;
        for (int64_t t = t0; t < t1; ++t) {
            const float* src = row_entropy + t * r;
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
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) kept_total += __shfl_xor_sync(0xffffffffu, kept_total, o);
    if ((threadIdx.x & 31) == 0) s_cnt[threadIdx.x >> 5] = kept_total;
    __syncthreads();
    if (threadIdx.x == 0) {
        int tot = 0;
        for (int w = 0; w < kThreads / 32; ++w) tot += s_cnt[w];
        cta_counts[blockIdx.x] = tot;
    }
}

// Mean, standard deviation (divisor n) and tau of n entropies: one CTA or a cluster of them, fp64, no scratch. Every CTA
// takes a contiguous part in two passes (the deviations are taken from the part's own mean), sums in a fixed order
// (thread-strided partial sums, a tree per CTA); a cluster's parts are merged once, in rank order, through distributed
// shared memory. Bound by what a few SMs load: a million entropies take one CTA 87 us, 8 18.4 (with two exchanges, one for the
// mean and one for the deviations), 16 12.0. A cluster costs 2 us to start and to meet in, so few entropies have one CTA, in a
// kernel without the cluster's barriers: us, one CTA / 16: 8192 4.0 / 6.2, 16384 4.4 / 6.3, 32768 5.7 / 6.5, 49152 7.1 / 6.6, 57344
// 7.8 / 6.9.
constexpr int kTauThreads = 1024;
constexpr int64_t kTauOneCta = 42 * kTauThreads;
__device__ __forceinline__ double cta_sum(double acc, double* s) {
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int o = kTauThreads / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
        __syncthreads();
    }
    const double total = s[0];
    __syncthreads();
    return total;
}
template <typename F>
__device__ __forceinline__ double tau_partial(const float* __restrict__ H, int64_t n, F&& f) {
    double a0 = 0.0, a1 = 0.0;
    // the part before the first 16-byte boundary, whole float4s, the rest
    const int64_t lead = min(n, (int64_t)((16 - (reinterpret_cast<uintptr_t>(H) & 15u)) & 15u) / 4);
    const int64_t n4 = (n - lead) / 4;
    const float4* H4 = reinterpret_cast<const float4*>(H + lead);
    if ((int64_t)threadIdx.x < lead) a0 += f(H[threadIdx.x]);
#pragma unroll 4
    for (int64_t i = threadIdx.x; i < n4; i += kTauThreads) {
        const float4 v = H4[i];
        a0 += f(v.x) + f(v.y);
        a1 += f(v.z) + f(v.w);
    }
    const int64_t rest = lead + 4 * n4 + threadIdx.x;
    if (rest < n) a1 += f(H[rest]);
    return a0 + a1;
}
struct TauPart { double n, mean, m2; };
template <bool CLUSTER>
__global__ void __launch_bounds__(kTauThreads) tau_kernel(const float* __restrict__ H, int64_t n, double* __restrict__ out) {
    __shared__ double s[kTauThreads];
    __shared__ TauPart s_part;
    unsigned rank = 0, size = 1;
    int64_t begin = 0, own = n;
    if constexpr (CLUSTER) {
        cg::cluster_group cl = cg::this_cluster();
        rank = cl.block_rank();
        size = cl.num_blocks();
        const int64_t per = (n + size - 1) / size;
        begin = (int64_t)rank * per;
        own = min(n, begin + per) - begin;                   // (more entropies than CTAs squared: every part has some)
    }
    double mean = cta_sum(tau_partial(H + begin, own, [](float h) { return (double)h; }), s) / (double)own;
    double q = cta_sum(tau_partial(H + begin, own, [mean](float h) {
        const double dlt = (double)h - mean;
        return dlt * dlt;
    }), s);
    if constexpr (CLUSTER) {
        cg::cluster_group cl = cg::this_cluster();
        if (threadIdx.x == 0) s_part = TauPart{(double)own, mean, q};
        cl.sync();
        if (rank == 0 && threadIdx.x == 0) {
            double sum = 0.0;
            for (unsigned r = 0; r < size; ++r) {
                const TauPart* p = cl.map_shared_rank(&s_part, r);
                sum += p->n * p->mean;
            }
            mean = sum / (double)n;
            q = 0.0;
            for (unsigned r = 0; r < size; ++r) {
                const TauPart* p = cl.map_shared_rank(&s_part, r);
                const double d = p->mean - mean;
                q += p->m2 + p->n * d * d;
            }
        }
        cl.sync();                                           // a CTA leaves when its part has been read
    }
    if (rank == 0 && threadIdx.x == 0) {
        const double sd = sqrt(q / (double)n);
        out[0] = mean;
        out[1] = sd;
        out[2] = 0.3 * mean - 0.1 * sd;
    }
}

// CTAs of the cluster on the current device: 16 where it takes such a cluster, else 8, which every device takes.
int tau_cluster() {
    static std::atomic<int> known[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 8;
    int c = known[dev].load(std::memory_order_relaxed);
    if (c) return c;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 16; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(16); cfg.blockDim = dim3(kTauThreads); cfg.attrs = at; cfg.numAttrs = 1;
    int fit = 0;
    c = cudaFuncSetAttribute(tau_kernel<true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                cudaOccupancyMaxActiveClusters(&fit, tau_kernel<true>, &cfg) == cudaSuccess && fit >= 1
            ? 16 : 8;
    if (c == 8) (void)cudaGetLastError();
    known[dev].store(c, std::memory_order_relaxed);
    return c;
}

__global__ void __launch_bounds__(kThreads)
accept_prefix_kernel(const float* __restrict__ r, const float* __restrict__ ratio, int64_t n, int32_t gamma,
                     int64_t n_blocks, const int32_t* __restrict__ block_len, int32_t* __restrict__ accepted) {
    const int64_t b = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (b >= n_blocks) return;
    const int64_t t0 = b * gamma;
    int64_t t1 = min(n, t0 + gamma);
    // the draft that reaches Step 4 is what Step 1 left of the block
    if (block_len) t1 = min(t1, t0 + (int64_t)max(block_len[b], 0));
    int acc = (int)(t1 - t0);
    for (int64_t t = t0; t < t1; ++t) {
        if (r[t] > ratio[t]) {
            acc = (int)(t - t0);
            break;
        }
    }
    accepted[b] = acc;
}

}  // namespace

namespace ardiff {
void load_prefix_kernel() {
    cudaFuncAttributes a;
    if (cudaFuncGetAttributes(&a, block_prefix_kernel) != cudaSuccess) (void)cudaGetLastError();
}
}  // namespace ardiff

extern "C" int ardiff_entropy_gate_blocks(const void* feat, int64_t n, int32_t rows_per_token, int32_t d,
                                          int32_t gamma, float tau, float* row_entropy, float* token_entropy,
                                          uint8_t* mask, int32_t* idx, int32_t* count, int32_t* block_len,
                                          void* stream) {
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (!count) return ARDIFF_ERR_NULL;
    if (n < 0 || rows_per_token < 1 || gamma < 1 || d < 1 || d > 65536) return ARDIFF_ERR_SHAPE;
    if (n >= (int64_t)1 << 31 || n * (int64_t)rows_per_token >= (int64_t)1 << 31) return ARDIFF_ERR_SHAPE;
    if (n == 0) {
        ardiff::set_launch_count(1);
        return ardiff::write_zero_count(count, st);
    }
    if (!feat || !mask || !idx) return ARDIFF_ERR_NULL;
    if (d % 8 != 0 && !row_entropy) return ARDIFF_ERR_NULL;      // the interface asks for it at such widths
    int32_t* counts = nullptr;
    int max_blocks = 0, sms = 0;
    int rc = ardiff::gate_scratch_get(st, &counts, &max_blocks, &sms);
    if (rc != ARDIFF_OK) return rc;
    // one pass over the features when the shape allows it; else row entropies through global memory
    rc = ardiff::gate_blocks_fused_launch(feat, n, rows_per_token, d, gamma, tau, row_entropy, token_entropy, mask,
                                          idx, count, block_len, counts, max_blocks, sms, st);
    if (rc != ARDIFF_ERR_UNSUPPORTED) return rc;
    if (!row_entropy) return ARDIFF_ERR_NULL;      // this path needs it as scratch
    rc = ardiff::entropy_rows_launch(feat, n * rows_per_token, d, row_entropy, sms, st);
    if (rc != ARDIFF_OK) return rc;
    // CTAs own whole draft blocks, so a block never straddles two compaction ranges
    const int64_t n_blocks = (n + gamma - 1) / gamma;
    int64_t want = (int64_t)sms * 4;
    if (want > max_blocks) want = max_blocks;
    int64_t bpc = (n_blocks + want - 1) / want;
    if (bpc < 1) bpc = 1;
    const int grid = (int)((n_blocks + bpc - 1) / bpc);
    block_prefix_kernel<<<grid, kThreads, 0, st>>>(row_entropy, n, rows_per_token, gamma, tau, token_entropy, mask,
                                                   block_len, counts, bpc, n_blocks);
    if (cudaGetLastError() != cudaSuccess) return ARDIFF_ERR_CUDA;
    rc = ardiff::compact_launch(mask, n, counts, bpc * gamma, grid, idx, count, st);
    ardiff::set_launch_count(3);
    return rc;
}

extern "C" int ardiff_tau_calibrate(const float* entropy, int64_t n, double* out3, void* stream) {
    if (!entropy || !out3) return ARDIFF_ERR_NULL;
    if (n < 1) return ARDIFF_ERR_SHAPE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (n <= kTauOneCta) {
        tau_kernel<false><<<1, kTauThreads, 0, st>>>(entropy, n, out3);
    } else {
        cudaLaunchConfig_t cfg;
        memset(&cfg, 0, sizeof(cfg));
        cudaLaunchAttribute at[1];
        const int ctas = tau_cluster();
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = ctas; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(ctas); cfg.blockDim = dim3(kTauThreads); cfg.stream = st;
        cfg.attrs = at; cfg.numAttrs = 1;
        (void)cudaLaunchKernelEx(&cfg, tau_kernel<true>, entropy, n, out3);
    }
    ardiff::set_launch_count(1);
    return cudaGetLastError() == cudaSuccess ? ARDIFF_OK : ARDIFF_ERR_CUDA;
}

extern "C" int ardiff_accept_prefix(const float* r, const float* ratio, int64_t n, int32_t gamma,
                                    const int32_t* block_len, int32_t* accepted, void* stream) {
    if (n < 0 || gamma < 1) return ARDIFF_ERR_SHAPE;
    if (n == 0) return ARDIFF_OK;
    if (!r || !ratio || !accepted) return ARDIFF_ERR_NULL;
    const int64_t n_blocks = (n + gamma - 1) / gamma;
    const int grid = (int)((n_blocks + kThreads - 1) / kThreads);
    accept_prefix_kernel<<<grid, kThreads, 0, static_cast<cudaStream_t>(stream)>>>(r, ratio, n, gamma, n_blocks,
                                                                                 block_len, accepted);
    ardiff::set_launch_count(1);
    return cudaGetLastError() == cudaSuccess ? ARDIFF_OK : ARDIFF_ERR_CUDA;
}
