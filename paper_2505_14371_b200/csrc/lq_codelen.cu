// Code-length accounting (the paper's appendix on the coding framework): the probability that each
// level of a layer is emitted, from the same histogram-based CDF estimate the level fit uses, and a
// count of the level indices a message actually carries, to set against those probabilities.
//
//   p^_j = int hat_j(u) dF~(u):  stochastic rounding sends u in [l_tau, l_{tau+1}] to l_tau with
//   probability (l_{tau+1} - u) / (l_{tau+1} - l_tau) and to l_{tau+1} otherwise, so level j collects
//   the rising half of its hat function from [l_{j-1}, l_j] and the falling half from [l_j, l_{j+1}].
//   F~ is piecewise linear inside the histogram bins, plus the point mass at u = 1 of the last bin.
// Compiled without FMA contraction: the sequence of fp64 roundings is the plain one.
#include "lq_internal.cuh"

namespace lq {
namespace {

constexpr int kBins = 385;            // bins 0..384 carry density; bin 385 is the point mass at u = 1

__device__ __forceinline__ double edge_of(int i)
{
    if (i <= 0) return 0.0;
    const int o = (i - 1) >> 4, m = (i - 1) & 15;
    return ldexp(1.0 + (double)m * 0.0625, o - 24);
}

// One CTA per layer, one warp per level at a time: the lanes take the bins that lie under the level's hat function (the
// first intervals of a level set span most of the 385 bins) and the warp adds their pieces.  One thread per level walking
// all bins took 152 us for 4-bit levels, the latency of its divisions throughout; this takes 11.
__global__ void __launch_bounds__(kMaxLevels) level_probabilities_kernel(PlanDev p, const uint32_t* hist,
                                                                         const float* norms, int Z,
                                                                         const float* levels,
                                                                         double* probs)
{
    __shared__ double mass[LQ_NUM_BINS];
    __shared__ double edge[kBins + 1];
    __shared__ double lev[kMaxLevels];
    __shared__ double weight[LQ_MAX_WORKERS];
    __shared__ double wsum_s;
    const int m = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
    const LayerDesc L = p.layers[m];
    const int n = L.nlevels;
    double* out = probs + (int64_t)m * kMaxLevels;
    pdl_launch_next();
    pdl_wait();
    for (int z = tid; z < Z; z += blockDim.x) {
        const double x = (double)norms[(int64_t)z * p.num_layers + m];
        weight[z] = x * x;
    }
    if (tid < n) lev[tid] = (double)levels[(int64_t)m * kLevelStride + tid];
    for (int i = tid; i <= kBins; i += blockDim.x) edge[i] = edge_of(i);
    __syncthreads();
    if (tid == 0) {
        double w = 0.0;
        for (int z = 0; z < Z; ++z) w += weight[z];
        wsum_s = w;
    }
    __syncthreads();
    const double wsum = wsum_s;
    if (tid >= n || !(wsum > 0.0) || L.size <= 0) out[tid] = 0.0;
    if (!(wsum > 0.0) || L.size <= 0) return;
    for (int i = tid; i < LQ_NUM_BINS; i += blockDim.x) {
        double acc = 0.0;
        for (int z = 0; z < Z; ++z)
            acc += (weight[z] / wsum) * (double)hist[((int64_t)z * p.num_layers + m) * LQ_HIST_STRIDE + i];
        mass[i] = acc / (double)L.size;
    }
    __syncthreads();
    // the bin that holds x: the largest i <= 384 with edge[i] <= x
    auto bin_of = [&](double x) {
        int lo = 0, hi = kBins - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (edge[mid] <= x) lo = mid; else hi = mid - 1;
        }
        return lo;
    };
    for (int j = tid >> 5; j < n; j += kMaxLevels / 32) {
        const double prev = j > 0 ? lev[j - 1] : 0.0, at = lev[j], next = j + 1 < n ? lev[j + 1] : 1.0;
        const int last = bin_of(next);
        double pj = 0.0;
        for (int i = bin_of(prev) + lane; i <= last; i += 32) {
            if (mass[i] == 0.0) continue;
            const double lo = edge[i], hi = edge[i + 1], dens = mass[i] / (hi - lo);
            if (j >= 1) {                                      // rising half on [l_{j-1}, l_j]
                const double x0 = fmax(lo, prev), x1 = fmin(hi, at);
                if (x1 > x0) pj += dens * (x1 - x0) * (0.5 * (x0 + x1) - prev) / (at - prev);
            }
            if (j <= n - 2) {                                  // falling half on [l_j, l_{j+1}]
                const double x0 = fmax(lo, at), x1 = fmin(hi, next);
                if (x1 > x0) pj += dens * (x1 - x0) * (next - 0.5 * (x0 + x1)) / (next - at);
            }
        }
        pj = warp_sum(pj);
        if (lane == 0) out[j] = j == n - 1 ? pj + mass[LQ_NUM_BINS - 1] : pj;      // the last level also has the point mass at u = 1
    }
}

// One CTA per (sub-tile, worker): counts the level indices of the message's real coordinates.
__global__ void __launch_bounds__(kThreads) symbol_counts_kernel(PlanDev p, const uint32_t* __restrict__ packed,
                                                                 uint32_t* __restrict__ counts)
{
    __shared__ uint32_t cnt[kMaxLevels];
    Tile tile = p.tiles[blockIdx.x >> p.sub_shift];
    const int sub0 = (blockIdx.x & (p.sub_tiles - 1)) * p.sub_blocks;
    if (sub0 >= tile.nblocks) return;
    const int sub1 = min(sub0 + p.sub_blocks, tile.nblocks);
    const int layer = tile.layer, k = blockIdx.y;
    const LayerDesc L = p.layers[layer];
    const int C = L.bits + 1, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < kMaxLevels; i += blockDim.x) cnt[i] = 0;
    __syncthreads();
    const uint32_t* msg = packed + (int64_t)k * p.packed_words + L.word_off;
    for (int b = sub0 + warp; b < sub1; b += kWarps) {
        const int64_t blk = tile.block0 + b;
        uint32_t w[LQ_MAX_BITS + 2];
        for (int i = 0; i < C; ++i) w[i] = msg[blk * (int64_t)C * 32 + i * 32 + lane];
        w[C] = 0u;
        for (int pp = 0; pp < 32; ++pp) {
            const int64_t coord = blk * kBlockCoords + 128 * (pp >> 2) + 4 * lane + (pp & 3);
            if (coord >= L.size) continue;
            const int off = pp * C, i = off >> 5, s = off & 31;
            const uint64_t two = ((uint64_t)w[i + 1] << 32) | w[i];
            const uint32_t sym = (uint32_t)(two >> s) & ((1u << C) - 1u);
            atomicAdd(&cnt[sym >> 1], 1u);
        }
    }
    __syncthreads();
    uint32_t* out = counts + ((int64_t)k * p.num_layers + layer) * kMaxLevels;
    for (int i = threadIdx.x; i < L.nlevels; i += blockDim.x)
        if (cnt[i]) atomicAdd(out + i, cnt[i]);
}

}  // namespace

cudaError_t launch_level_probabilities(const PlanDev& p, const uint32_t* hist, const float* norms, int num_samples,
                                       const float* levels, double* probs, cudaStream_t s)
{
    if (p.num_layers == 0) return cudaSuccess;
    return launch(level_probabilities_kernel, (unsigned)p.num_layers, kMaxLevels, 0, s, p, hist, norms, num_samples, levels, probs);
}

cudaError_t launch_symbol_counts(const PlanDev& p, const uint32_t* packed, uint32_t* counts, cudaStream_t s)
{
    if (p.num_tiles == 0) return cudaSuccess;
    const dim3 grid((unsigned)p.num_tiles * p.sub_tiles, (unsigned)p.num_workers);
    symbol_counts_kernel<<<grid, kThreads, 0, s>>>(p, packed, counts);
    return cudaGetLastError();
}

}  // namespace lq
