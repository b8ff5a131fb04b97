// ENCODE in the layer norm scope for plans whose layers are all small: one cluster of up to 16 CTAs takes a whole (layer,
// worker), so the norm, which every coordinate of the layer needs before its first symbol, is exchanged inside the
// cluster (distributed shared memory, a cluster barrier) instead of through kernel boundaries: one launch where the
// general path has four (norm partials, norms, encoder, statistic).  Such plans are a chain of launches of a few us each,
// with nothing to fill the GPU, so latency is what bounds them, and more than that of sums and look-ups the latency of fetching
// code: warp j of a CTA takes row j of each of its blocks, and all warps run the same code.
// (Which plans: lq_small_rule.h.)
#include <algorithm>
#include <mutex>

#include "lq_quantize_rows.cuh"

namespace lq {

namespace {

// room for the words of a CTA's blocks
__host__ __device__ constexpr int kSmallWords(int blocks, int C) { return blocks * C * 32; }

// ---- cluster exchange
__device__ __forceinline__ void st_peer(const double* mine, uint32_t rank, double v)
{
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(mine)), "r"(rank));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// Warp j takes row j of all of the CTA's blocks.  `rows` (zeroed): bit j of a block's word says whether its row j holds anything
// but zeros.  `first`: the lane's values of the first block's row.
template <int kMode>
__device__ __forceinline__ double norm_of_rows(const PlanDev& p, const float* g, int64_t size, int block0, int nblocks,
                                               uint32_t* rows, double* scratch, float4& first)
{
    const int lane = threadIdx.x & 31, j = threadIdx.x >> 5;
    double acc = 0.0;
    uint32_t maxbits = 0;
    constexpr int kAhead = 4;
    for (int b0 = 0; b0 < nblocks; b0 += kAhead) {
        float4 v[kAhead];
#pragma unroll
        for (int i = 0; i < kAhead; ++i)
            v[i] = b0 + i < nblocks ? row_values(g, block0 + b0 + i, j, size, lane) : make_float4(0.f, 0.f, 0.f, 0.f);
        if (b0 == 0) first = v[0];
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
            accumulate<kMode>(acc, maxbits, v[i].x, p.q);
            accumulate<kMode>(acc, maxbits, v[i].y, p.q);
            accumulate<kMode>(acc, maxbits, v[i].z, p.q);
            accumulate<kMode>(acc, maxbits, v[i].w, p.q);
            const float mag = (fabsf(v[i].x) + fabsf(v[i].y)) + (fabsf(v[i].z) + fabsf(v[i].w));
            if (__any_sync(0xffffffffu, mag != 0.0f) && lane == 0) atomicOr(rows + b0 + i, 1u << j);
        }
    }
    return norm_cta_total<kMode>(acc, maxbits, scratch);
}

// What a CTA of a cluster takes of its layer: an equal share of consecutive blocks.
__device__ __forceinline__ Tile cluster_share(const LayerDesc& L, int layer, int rank, int ranks)
{
    const int per = (L.nblocks + ranks - 1) / ranks;
    Tile t;
    t.layer = layer; t.block0 = rank * per; t.nblocks = max(0, min(per, L.nblocks - t.block0)); t.pad_ = 0;
    return t;
}

// The layer's norm from all CTAs of the cluster: each sends its sum to every other, and all add them in rank order.  What
// is done between the two calls overlaps the exchange.  (The caller has arrived at the cluster's barrier once before.)
__device__ __forceinline__ void cluster_norm_send(const PlanDev& p, const float* g, const LayerDesc& L, const Tile& t, int rank,
                                                  int ranks, uint32_t* rows, double* scratch, double* part, float4& first)
{
    const double mine = p.q == 0   ? norm_of_rows<0>(p, g, L.size, t.block0, t.nblocks, rows, scratch, first)
                        : p.q == 1 ? norm_of_rows<1>(p, g, L.size, t.block0, t.nblocks, rows, scratch, first)
                        : p.q == 2 ? norm_of_rows<2>(p, g, L.size, t.block0, t.nblocks, rows, scratch, first)
                                   : norm_of_rows<3>(p, g, L.size, t.block0, t.nblocks, rows, scratch, first);
    cluster_wait();                                          // every CTA of the cluster runs
    if (threadIdx.x == 0)
        for (int r = 0; r < ranks; ++r) st_peer(&part[rank], r, mine);
    cluster_arrive();
}
__device__ __forceinline__ LayerNorm cluster_norm_receive(const PlanDev& p, int ranks, const double* part)
{
    cluster_wait();
    double total = 0.0;
    bool bad = false;
    for (int r = 0; r < ranks; ++r) {
        const double v = part[r];
        if (!(fabs(v) <= 1.7976931348623157e308)) bad = true;
        total = p.q == 0 ? fmax(total, v) : total + v;
    }
    return layer_norm_of_total(total, bad, p.q);
}
__device__ __forceinline__ void store_norm(const PlanDev& p, const LayerNorm& n, float* norms, int64_t kl)
{
    norms[kl] = n.norm; p.rnorm[kl] = n.rnorm; p.status[kl] = n.status;
}

// The norms alone, in the encoder's order (lq_layer_norms gives the very norms that lq_quantize_pack sends).
__global__ void __launch_bounds__(kQThreads) layer_norms_small_kernel(PlanDev p, const float* grads, float* norms)
{
    __shared__ double part[kSmallRanks], scratch[kQWarps];
    __shared__ uint32_t rows[kSmallShare];                    // (not used)
    float4 first;
    pdl_launch_next();
    const int ranks = gridDim.x, rank = blockIdx.x, layer = blockIdx.y, k = blockIdx.z + p.worker0;
    cluster_arrive();
    const LayerDesc L = p.layers[layer];
    const Tile t = cluster_share(L, layer, rank, ranks);
    pdl_wait();
    cluster_norm_send(p, fresh(grads + (int64_t)blockIdx.z * p.padded_elems + L.elem_off), L, t, rank, ranks, rows, scratch, part, first);
    const LayerNorm n = cluster_norm_receive(p, ranks, part);
    if (rank == 0 && threadIdx.x == 0) store_norm(p, n, norms, (int64_t)k * p.num_layers + layer);
}

template <bool kHist, bool kStat>
__global__ void __launch_bounds__(kQThreads, 3) quantize_small_kernel(
    PlanDev p, const float* grads, uint32_t step, uint32_t* packed, float* norms, uint32_t* hist,
    const uint32_t* prev_packed, const float* prev_norms, const float* levels_cur, const float* levels_prev, SearchTables st)
{
    extern __shared__ unsigned char dyn_smem[];
    __shared__ double norm_part[kSmallRanks], stat_part[kSmallRanks];             // per CTA of the cluster
    __shared__ uint32_t rows[kSmallShare];
    uint32_t base;
    unsigned char* sm = table_base(dyn_smem, base);
    pdl_launch_next();
    // grid: x = CTA of the cluster, y = layer, z = worker
    const int ranks = gridDim.x, rank = blockIdx.x, layer = blockIdx.y, k = blockIdx.z + p.worker0;
    cluster_arrive();                                         // (waited for before the first store into a peer)
    const LayerDesc L = p.layers[layer];
    const Tile tile = cluster_share(L, layer, rank, ranks);
    const int lane = threadIdx.x & 31, C = L.bits + 1;
    const int64_t kl = (int64_t)k * p.num_layers + layer;
    uint32_t* words = reinterpret_cast<uint32_t*>(sm + kSmRing);                // the blocks' words, behind them the histogram
    uint32_t* counts = words + kSmallWords(tile.nblocks, C);
    if (threadIdx.x < tile.nblocks) rows[threadIdx.x] = 0u;
    for (int i = threadIdx.x; i < tile.nblocks * C * 32; i += kQThreads) words[i] = 0u;
    if (kHist)
        for (int i = threadIdx.x; i < LQ_HIST_STRIDE; i += kQThreads) counts[i] = 0u;
    __syncthreads();
    pdl_wait();
    const float* g = fresh(grads + (int64_t)blockIdx.z * p.padded_elems + L.elem_off);
    if (rank == 0 && layer == 0 && blockIdx.z == 0 && threadIdx.x == 0) p.scalars[1] = p.scalars[0];

    // everything that does not need the norm is requested before the values
    const float nprev = prev_norms ? load_f32(prev_norms + kl) : 0.0f;
    const int2 how = load_i32x2(st.how + layer);
    const uint4* lsrc = reinterpret_cast<const uint4*>(st.lut + (int64_t)layer * kLutEntries);
    const uint4 lut0 = load_u32x4(lsrc + threadIdx.x), lut1 = load_u32x4(lsrc + kQThreads + threadIdx.x);
    const int64_t mask_at = (int64_t)k * p.total_blocks + L.block_off + tile.block0 + threadIdx.x;
    uint32_t mprev = 0;
    if (threadIdx.x < tile.nblocks)
        mprev = (!kStat || !prev_packed) ? 0u : (p.row_mask_prev ? load_u8(p.row_mask_prev + mask_at) : 0xffu);
    float lc = 0.f, lp = 0.f;
    float2 lg = make_float2(0.f, 0.f);
    if (threadIdx.x < L.nlevels) {
        lc = load_f32(levels_cur + (int64_t)layer * kLevelStride + threadIdx.x);
        lp = load_f32(levels_prev + (int64_t)layer * kLevelStride + threadIdx.x);
        lg = load_f32x2(st.ld + (int64_t)layer * kMaxLevels + threadIdx.x);
    }
    double* scratch = reinterpret_cast<double*>(sm + kSmScratch);
    float4 first;
    cluster_norm_send(p, g, L, tile, rank, ranks, rows, scratch, norm_part, first);
    {
        uint4* ldst = reinterpret_cast<uint4*>(sm + kSmLut);
        ldst[threadIdx.x] = lut0;
        ldst[kQThreads + threadIdx.x] = lut1;
    }
    const LayerNorm ln = cluster_norm_receive(p, ranks, norm_part);
    if (threadIdx.x < L.nlevels) {
        const float cv = __fmul_rn(ln.norm, lc), pv = __fmul_rn(nprev, lp);
        reinterpret_cast<float2*>(sm + kSmLd)[threadIdx.x] = lg;
        reinterpret_cast<float2*>(sm + kSmTcur)[threadIdx.x] = make_float2(cv, -cv);
        reinterpret_cast<float2*>(sm + kSmTprev)[threadIdx.x] = make_float2(pv, -pv);
    }
    if (threadIdx.x == 0) *reinterpret_cast<int2*>(sm + kSmHow) = how;
    if (threadIdx.x < tile.nblocks) {                        // (the rows' bits lie behind norm_cta_total's barriers)
        const uint32_t live = rows[threadIdx.x];
        p.row_mask[mask_at] = (uint8_t)live;
        rows[threadIdx.x] = (ln.rnorm != 0.0f ? live : 0u) | (mprev << 8);        // a layer without a norm sends zeros
    }
    if (rank == 0 && threadIdx.x == 0) store_norm(p, ln, norms, kl);
    __syncthreads();

    RowsJob job;
    job.g = g;
    job.prev = prev_packed ? fresh(prev_packed + (int64_t)k * p.packed_words + L.word_off) : nullptr;
    job.size = L.size;
    job.block0 = tile.block0; job.nblocks = tile.nblocks;
    job.rows = rows;
    job.words = base + kSmRing;
    job.counts = ln.rnorm != 0.0f;
    QuantEnv ev;
    ev.lut = base + kSmLut; ev.ld = base + kSmLd; ev.tprev = base + kSmTprev;
    ev.r = ln.rnorm;
    ev.hist = counts;
    if (step == LQ_STEP_AUTO) step = (uint32_t)p.scalars->t;      // the plan's own iteration counter (graph replays)
    const PhiloxConsts pc = philox_fold((uint32_t)layer, (uint32_t)k, step, p.seed_lo, p.seed_hi);
    double stat = 0.0;
    if (tile.nblocks > 0) {
        switch (L.bits) {
#define LQ_CASE(BB) case BB: stat = quantize_rows_by<BB, kHist, kStat>(p, pc, job, ev, how.x & 3, first, lane, (int)(threadIdx.x >> 5)); break;
            LQ_CASE(1) LQ_CASE(2) LQ_CASE(3) LQ_CASE(4) LQ_CASE(5) LQ_CASE(6) LQ_CASE(7) LQ_CASE(8)
#undef LQ_CASE
            default: break;
        }
    }
    const double sum = block_reduce<false>(kStat ? stat : 0.0, scratch);
    if (threadIdx.x == 0) st_peer(&stat_part[rank], 0, sum);
    cluster_arrive();
    // (block_reduce's barriers lie behind the last word and the last count)
    uint32_t* out = packed + (int64_t)k * p.packed_words + L.word_off + (int64_t)tile.block0 * (C * 32);
    for (int i = threadIdx.x; i < tile.nblocks * C * 32; i += kQThreads) __stcs(out + i, words[i]);
    if (kHist) {
        uint32_t* h = hist + kl * LQ_HIST_STRIDE;
        for (int i = threadIdx.x; i < LQ_NUM_BINS; i += blockDim.x)
            if (counts[i]) atomicAdd(h + i, counts[i]);
    }
    cluster_wait();
    if (rank == 0 && threadIdx.x == 0) {
        double s = 0.0;
        for (int r = 0; r < ranks; ++r) s += stat_part[r];
        p.sq_diff[kl] = s;
    }
}

}  // namespace

// The most shared memory that the kernel asks for.
constexpr unsigned kSmallTables = kSmRing + kSmSlack, kSmallMost = kSmallTables + kSmallWords(kSmallShare, LQ_MAX_BITS + 1) * 4 + LQ_HIST_STRIDE * 4;

namespace {

cudaError_t allow_small()
{
    static std::atomic<uint64_t> memory{0}, clusters{0};
    cudaError_t e = opt_in_shared_memory(memory, (int)kSmallMost, quantize_small_kernel<true, true>,
                                         quantize_small_kernel<false, true>, quantize_small_kernel<false, false>);
    if (e == cudaSuccess)
        e = allow_clusters(clusters, layer_norms_small_kernel, quantize_small_kernel<true, true>, quantize_small_kernel<false, true>,
                           quantize_small_kernel<false, false>);
    return e;
}

}  // namespace

ClusterRoom small_cluster_room()
{
    static std::mutex guard;
    static ClusterRoom rooms[64];                                // asked for once per device
    static uint64_t known = 0;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return ClusterRoom{}; }
    const std::lock_guard<std::mutex> lock(guard);
    if (dev < 64 && ((known >> dev) & 1u)) return rooms[dev];
    ClusterRoom room{};
    cudaError_t e = allow_small();
    for (int i = 0; i < 5 && e == cudaSuccess; ++i) {
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = 1u << i; at.val.clusterDim.y = 1; at.val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(1u << i, 1, 1); cfg.blockDim = kQThreads; cfg.dynamicSmemBytes = kSmallMost;
        cfg.attrs = &at; cfg.numAttrs = 1;
        int least = INT32_MAX;
        for (auto kernel : {quantize_small_kernel<true, true>, quantize_small_kernel<false, true>, quantize_small_kernel<false, false>}) {
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) { n = 0; cudaGetLastError(); }
            least = std::min(least, n);
        }
        room.clusters[i] = least;
    }
    if (e != cudaSuccess) cudaGetLastError();
    else if (dev < 64) { rooms[dev] = room; known |= 1ull << dev; }
    return room;
}

cudaError_t launch_layer_norms_small(const PlanDev& p, const float* grads, float* norms, cudaStream_t s)
{
    const cudaError_t e = allow_small();
    if (e != cudaSuccess) return e;
    const unsigned ranks = (unsigned)p.small_ranks;
    return launch_cluster(layer_norms_small_kernel, dim3(ranks, (unsigned)p.num_layers, (unsigned)p.worker_count), kQThreads, 0, ranks,
                          s, p, grads, norms);
}

cudaError_t launch_quantize_small(const PlanDev& p, const float* grads, uint32_t step, uint32_t* packed, float* norms,
                                  uint32_t* hist, const uint32_t* prev_packed, const float* prev_norms,
                                  const float* levels_cur, const float* levels_prev, SearchTables t, bool need_stat, cudaStream_t s)
{
    if (p.num_layers == 0) return cudaSuccess;
    const cudaError_t e = allow_small();
    if (e != cudaSuccess) return e;
    const auto kernel = hist ? quantize_small_kernel<true, true>
                        : need_stat ? quantize_small_kernel<false, true> : quantize_small_kernel<false, false>;
    const unsigned ranks = (unsigned)p.small_ranks;
    const unsigned smem = kSmallTables + kSmallWords(p.small_share, p.most_bits + 1) * 4 + (hist ? LQ_HIST_STRIDE * 4 : 0);
    return launch_cluster(kernel, dim3(ranks, (unsigned)p.num_layers, (unsigned)p.worker_count), kQThreads, smem, ranks, s, p, grads, step,
                          packed, norms, hist, prev_packed, prev_norms, levels_cur, levels_prev, t);
}

}  // namespace lq
