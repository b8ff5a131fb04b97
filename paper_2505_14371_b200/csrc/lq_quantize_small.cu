// ENCODE in the layer norm scope for plans whose layers are all small: one cluster of up to 8 CTAs takes a whole (layer,
// worker), so the norm, which every coordinate of the layer needs before its first symbol, is exchanged inside the
// cluster (distributed shared memory, a cluster barrier) instead of through kernel boundaries: one launch where the
// general path has four (norm partials, norms, encoder, statistic).  Such plans are a chain of launches of a few us each,
// with nothing to fill the GPU, so latency is what bounds them.
//
// The rule (use_small): every layer has at most 256 blocks of 1024 coordinates (8 CTAs of 32), and the clusters of all
// layers and all of the plan's workers run at once: 3 CTAs per SM, or for whole clusters, which have to fit an SM group
// each, 352 CTAs.  It asks for nothing but the plan's constants: a worker range does not change which kernel encodes a
// layer, nor the order in which the layer's sums are formed.  A cluster has as many CTAs as its plan's largest layer needs
// for one block per warp; the values are read twice, the second time from L2.
// lq_quantize_pack at 3 bits and 4 workers, this kernel and the general path: layers of one block 18.9 and 25.0 us at 444
// CTAs, 34.8 and 26.9 at 592; of 64 blocks 27.5 and 38.9 at 352 CTAs, 46.7 and 40.1 at 416; of 256 blocks 52.0 and 60.6 at
// 352, 75.7 and 65.7 at 416 (there the second wave waits for whole clusters).
#include "lq_quantize_tile.cuh"

namespace lq {

namespace {

// ---- cluster exchange
__device__ __forceinline__ void st_peer(const double* mine, uint32_t rank, double v)
{
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(mine)), "r"(rank));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

template <int kMode>
__device__ __forceinline__ double norm_of_blocks(const PlanDev& p, const float* g, int64_t size, int block0, int nblocks,
                                                 uint8_t* rows, double* scratch)
{
    double acc = 0.0;
    uint32_t maxbits = 0;
    for (int b = threadIdx.x >> 5; b < nblocks; b += kQWarps) {
        const uint32_t r = norm_block<kMode>(g, block0 + b, size, threadIdx.x & 31, p.q, acc, maxbits);
        if ((threadIdx.x & 31) == 0) rows[b] = (uint8_t)r;
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
                                                  int ranks, uint8_t* rows, double* scratch, double* part)
{
    const double mine = p.q == 0   ? norm_of_blocks<0>(p, g, L.size, t.block0, t.nblocks, rows, scratch)
                        : p.q == 1 ? norm_of_blocks<1>(p, g, L.size, t.block0, t.nblocks, rows, scratch)
                        : p.q == 2 ? norm_of_blocks<2>(p, g, L.size, t.block0, t.nblocks, rows, scratch)
                                   : norm_of_blocks<3>(p, g, L.size, t.block0, t.nblocks, rows, scratch);
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
    __shared__ double part[8], scratch[kQWarps];
    __shared__ uint8_t rows[32];                             // (8 CTAs for up to 256 blocks)
    pdl_launch_next();
    const int ranks = gridDim.x, rank = blockIdx.x, layer = blockIdx.y, k = blockIdx.z + p.worker0;
    cluster_arrive();
    const LayerDesc L = p.layers[layer];
    const Tile t = cluster_share(L, layer, rank, ranks);
    pdl_wait();
    cluster_norm_send(p, fresh(grads + (int64_t)blockIdx.z * p.padded_elems + L.elem_off), L, t, rank, ranks, rows, scratch, part);
    const LayerNorm n = cluster_norm_receive(p, ranks, part);
    if (rank == 0 && threadIdx.x == 0) store_norm(p, n, norms, (int64_t)k * p.num_layers + layer);
}

template <bool kHist, bool kStat>
__global__ void __launch_bounds__(kQThreads, 3) quantize_small_kernel(
    PlanDev p, const float* grads, uint32_t step, uint32_t* packed, float* norms, uint32_t* hist,
    const uint32_t* prev_packed, const float* prev_norms, const float* levels_cur, const float* levels_prev, SearchTables st)
{
    extern __shared__ unsigned char dyn_smem[];
    __shared__ double norm_part[8], stat_part[8];             // per CTA of the cluster
    uint32_t base;
    unsigned char* sm = table_base(dyn_smem, base);
    pdl_launch_next();
    // grid: x = CTA of the cluster, y = layer, z = worker
    const int ranks = gridDim.x, rank = blockIdx.x, layer = blockIdx.y, k = blockIdx.z + p.worker0;
    cluster_arrive();                                         // (waited for before the first store into a peer)
    const LayerDesc L = p.layers[layer];
    const Tile tile = cluster_share(L, layer, rank, ranks);
    const int lane = threadIdx.x & 31;
    const int64_t kl = (int64_t)k * p.num_layers + layer;
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
    uint8_t* rows_cur = sm + kSmRows;
    uint8_t* rows_prev = rows_cur + kTileBlocks;
    double* scratch = reinterpret_cast<double*>(sm + kSmScratch);
    cluster_norm_send(p, g, L, tile, rank, ranks, rows_cur, scratch, norm_part);
    {
        uint4* ldst = reinterpret_cast<uint4*>(sm + kSmLut);
        ldst[threadIdx.x] = lut0;
        ldst[kQThreads + threadIdx.x] = lut1;
        if (kHist) {
            uint32_t* h = reinterpret_cast<uint32_t*>(sm + kSmHist);
            for (int i = threadIdx.x; i < LQ_HIST_STRIDE; i += kQThreads) h[i] = 0;
        }
    }
    const LayerNorm ln = cluster_norm_receive(p, ranks, norm_part);
    if (threadIdx.x < L.nlevels) {
        const float cv = __fmul_rn(ln.norm, lc), pv = __fmul_rn(nprev, lp);
        reinterpret_cast<float2*>(sm + kSmLd)[threadIdx.x] = lg;
        reinterpret_cast<float2*>(sm + kSmTcur)[threadIdx.x] = make_float2(cv, -cv);
        reinterpret_cast<float2*>(sm + kSmTprev)[threadIdx.x] = make_float2(pv, -pv);
    }
    if (threadIdx.x == 0) *reinterpret_cast<int2*>(sm + kSmHow) = how;
    if (threadIdx.x < tile.nblocks) {
        rows_prev[threadIdx.x] = (uint8_t)mprev;
        p.row_mask[mask_at] = rows_cur[threadIdx.x];
    }
    if (rank == 0 && threadIdx.x == 0) store_norm(p, ln, norms, kl);
    __syncthreads();

    WarpCtx c;
    c.g = g;
    c.size = L.size;
    c.nfull = L.size / kBlockCoords;
    c.lane = lane;
    QuantEnv ev;
    ev.lut = base + kSmLut; ev.ld = base + kSmLd; ev.tprev = base + kSmTprev;
    ev.r = ln.rnorm;
    ev.hist = reinterpret_cast<uint32_t*>(sm + kSmHist);
    if (step == LQ_STEP_AUTO) step = (uint32_t)p.scalars->t;      // the plan's own iteration counter (graph replays)
    const PhiloxConsts pc = philox_fold((uint32_t)layer, (uint32_t)k, step, p.seed_lo, p.seed_hi);
    uint32_t* out = packed + (int64_t)k * p.packed_words + L.word_off;
    const uint32_t* prev = prev_packed ? fresh(prev_packed + (int64_t)k * p.packed_words + L.word_off) : nullptr;
    const double stat = quantize_blocks<0, kHist, kStat>(p, pc, c, tile, L.bits, how.x & 3, (uint32_t)layer, (uint32_t)k, step, out, prev, ev,
                                                      rows_cur, rows_prev, base + kSmRing);
    const double sum = block_reduce<false>(stat, scratch);
    if (threadIdx.x == 0) st_peer(&stat_part[rank], 0, sum);
    cluster_arrive();
    if (kHist) {                                             // (block_reduce's barriers lie behind the last count)
        uint32_t* h = hist + kl * LQ_HIST_STRIDE;
        for (int i = threadIdx.x; i < LQ_NUM_BINS; i += blockDim.x)
            if (ev.hist[i]) atomicAdd(h + i, ev.hist[i]);
    }
    cluster_wait();
    if (rank == 0 && threadIdx.x == 0) {
        double s = 0.0;
        for (int r = 0; r < ranks; ++r) s += stat_part[r];
        p.sq_diff[kl] = s;
    }
}

int small_ranks(const PlanDev& p)
{
    int r = 1;
    while (r < 8 && r * kQWarps < p.most_blocks) r *= 2;
    return r;
}

}  // namespace

bool use_small(const PlanDev& p)
{
    const int ranks = small_ranks(p);
    return !p.global_norm && !p.bucket_norm && p.most_blocks <= 256 &&
           (int64_t)p.num_workers * p.num_layers * ranks <= (ranks == 1 ? 3 * kSms : 352);
}

cudaError_t launch_layer_norms_small(const PlanDev& p, const float* grads, float* norms, cudaStream_t s)
{
    const unsigned ranks = (unsigned)small_ranks(p);
    return launch_cluster(layer_norms_small_kernel, dim3(ranks, (unsigned)p.num_layers, (unsigned)p.worker_count), kQThreads, 0, ranks,
                          s, p, grads, norms);
}

cudaError_t launch_quantize_small(const PlanDev& p, const float* grads, uint32_t step, uint32_t* packed, float* norms,
                                  uint32_t* hist, const uint32_t* prev_packed, const float* prev_norms,
                                  const float* levels_cur, const float* levels_prev, SearchTables t, bool need_stat, cudaStream_t s)
{
    if (p.num_layers == 0) return cudaSuccess;
    constexpr unsigned smem = kSmTables + kRingBytes + kSmSlack, smem_hist = smem + LQ_HIST_STRIDE * 4;
    static std::atomic<uint64_t> configured{0};
    const cudaError_t e = opt_in_shared_memory(configured, (int)smem_hist, quantize_small_kernel<true, true>,
                                               quantize_small_kernel<false, true>, quantize_small_kernel<false, false>);
    if (e != cudaSuccess) return e;
    const auto kernel = hist ? quantize_small_kernel<true, true>
                        : need_stat ? quantize_small_kernel<false, true> : quantize_small_kernel<false, false>;
    const unsigned ranks = (unsigned)small_ranks(p);
    return launch_cluster(kernel, dim3(ranks, (unsigned)p.num_layers, (unsigned)p.worker_count), kQThreads,
                          hist ? smem_hist : smem, ranks, s, p, grads, step, packed, norms, hist, prev_packed, prev_norms,
                          levels_cur, levels_prev, t);
}

}  // namespace lq
