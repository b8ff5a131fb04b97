// ENCODE for all workers in the layer and global norm scopes: normalise, round stochastically between
// neighbouring levels, pack one (b+1)-bit symbol per coordinate (Section 3.1 quantizer, Section 3.2 message;
// Algorithm 1 line 12), with the optional histogram of normalised magnitudes (Algorithm 1 line 4) and the
// sender-side term of the adaptive step size, sum ||V^_{k,t+1/2} - V^_{k,t-1/2}||^2 (Eq. general_stepsize).
//
// Work decomposition: one CTA of 8 warps per (tile, worker); a tile is up to 128 blocks of 1024
// coordinates of one layer, taken round-robin by the warps.  A lane owns the 32 coordinates
// {128 j + 4 lane + e} of a block (row j = one float4 per lane, 512 contiguous bytes per warp).  Rows
// travel from global memory into a per-warp ring of 8 rows in shared memory with 16-byte
// asynchronous copies, so a warp always has up to 4 KB in flight and the values never sit in registers
// while they wait; every lane reads back only the bytes it copied itself, so the ring needs no
// barrier.  Per row the lane draws one Philox4x32-10 block (4 uniforms); after 8 rows it holds
// exactly b+1 words of symbols, which it stores plane by plane (128 contiguous bytes per warp and
// plane).  No shuffles, ballots or atomics on the per-coordinate path.  The kernel is bound by its
// arithmetic pipes and the issue of some 40 instructions per coordinate (10 Philox, 7 the statistic), not by DRAM.
//
// The level search and the tables are described in lq_quantize.cuh.  Layers whose levels are denser than the
// search table's bins take finer bins, or a byte table and steps up from its entry (build_search_kernel).
//
// The norm pass, which reads the same values just before, leaves one bit per row of 128 values
// that says whether the row holds anything but zeros.  An all-zero row (untouched embedding rows)
// is never fetched, draws no random numbers and needs no search: its symbols are 0.  If the
// previous message is all zero there as well, the row adds nothing to the statistic and is
// skipped entirely.  The masks are made warp-uniform by a reduction, so the per-row tests are uniform
// branches.  The unrolled code handles whole blocks only; a layer's last, partial block is taken by all warps, a row
// each (once per layer and worker).
#include "lq_quantize_tile.cuh"

namespace lq {

// The layer's last, partial block, by all warps of the CTA that has it, a row each, once they are done with their whole blocks; its
// words are gathered where the rings were.  It looks everything up again, so that the whole blocks' code carries nothing for it
// (as arguments it took that code 844 -> 950 us on the Transformer-XL shapes).  Returns the thread's statistic term.
// One warp that went through the 32 positions of its lanes one by one, each with a load and a binary search to wait for, took some 20
// us, behind the last whole block of its layer: steps of 1 365 blocks in 40 layers and 2 workers 53.9 -> 39.6, of 504 blocks in
// 30 layers 53.7 -> 32.1 us.
template <int B, bool kHist, bool kStat>
__device__ __noinline__ double quantize_last_block(const PlanDev& p, const float* grads, uint32_t step, uint32_t* packed,
                                                   const uint32_t* prev_packed)
{
    extern __shared__ unsigned char dyn_smem[];
    constexpr int C = B + 1;
    uint32_t base;
    unsigned char* sm = table_base(dyn_smem, base);
    const int flat = blockIdx.y * gridDim.x + blockIdx.x, slot = flat / (int)gridDim.y, kk = flat - slot * (int)gridDim.y;
    const TileJob J = p.jobs[slot];
    const int k = kk + p.worker0, b = J.nblocks - 1, lane = threadIdx.x & 31, j = threadIdx.x >> 5;
    uint32_t* words = reinterpret_cast<uint32_t*>(sm + kSmRing);
    RowsJob job;
    job.g = fresh(grads + (int64_t)kk * p.padded_elems + J.elem_off);
    job.prev = kStat && prev_packed ? fresh(prev_packed + (int64_t)k * p.packed_words + J.word_off) : nullptr;
    job.size = J.size;
    job.block0 = J.block0 + b; job.nblocks = 1;
    job.rows = words + C * 32;
    job.words = base + kSmRing;
    job.counts = true;
    const float4 first = row_values(job.g, job.block0, j, job.size, lane);
    __syncthreads();
    for (int i = threadIdx.x; i < C * 32; i += kQThreads) words[i] = 0u;
    if (threadIdx.x == 0) words[C * 32] = (uint32_t)sm[kSmRows + b] | ((uint32_t)sm[kSmRows + kTileBlocks + b] << 8);
    __syncthreads();
    QuantEnv ev;
    ev.lut = base + kSmLut; ev.ld = base + kSmLd; ev.tprev = base + kSmTprev;
    ev.r = p.rnorm[(int64_t)k * p.num_layers + J.layer];
    ev.hist = reinterpret_cast<uint32_t*>(sm + kSmHist);
    if (step == LQ_STEP_AUTO) step = (uint32_t)p.scalars->t;
    const PhiloxConsts pc = philox_fold((uint32_t)J.layer, (uint32_t)k, step, p.seed_lo, p.seed_hi);
    const double stat = quantize_rows_by<B, kHist, kStat>(p, pc, job, ev, reinterpret_cast<const int2*>(sm + kSmHow)->x & 3, first, lane, j);
    __syncthreads();
    uint32_t* out = packed + (int64_t)k * p.packed_words + J.word_off + (int64_t)job.block0 * (C * 32);
    for (int i = threadIdx.x; i < C * 32; i += kQThreads) __stcs(out + i, words[i]);
    return stat;
}

// kWidth: the code width of every layer of the plan, or 0 when they differ (a kernel of one width has less code to fetch).
// The plan is a grid constant: a function that is handed it by reference otherwise makes every thread copy it to its stack (288
// bytes: WGAN step 166 -> 180 us).  With it and the partial block out of the way the widths but 8 have no spills (0 to 52 bytes
// before): Transformer-XL step 1938 -> 1911 us, low-rank factors 322 -> 267, widths 2, 3, 4 and 8 side by side 2396 -> 2280.
template <int kWidth, bool kHist, bool kStat>
__global__ void __launch_bounds__(kQThreads, 4) quantize_pack_kernel(
    const __grid_constant__ PlanDev p, const float* grads, uint32_t step, uint32_t* packed, const float* norms, uint32_t* hist,
    const uint32_t* prev_packed, const float* prev_norms, const float* levels_cur, const float* levels_prev, SearchTables st)
{
    extern __shared__ unsigned char dyn_smem[];
    uint32_t base;
    unsigned char* sm = table_base(dyn_smem, base);
    // CTAs start in the order of their flat index: the workers of one tile next to each other, tiles in the plan's
    // launch order, so that the last CTAs to start are every worker's short tiles (the ends of the layers) and not
    // one worker's whole message
    const int flat = blockIdx.y * gridDim.x + blockIdx.x;
    const int slot = flat / (int)gridDim.y, kk = flat - slot * (int)gridDim.y;
    pdl_launch_next();
    const TileJob J = p.jobs[slot];
    const int tile_id = J.tile, layer = J.layer;
    Tile tile;
    tile.layer = J.layer; tile.block0 = J.block0; tile.nblocks = J.nblocks; tile.pad_ = 0;
    LayerDesc L;
    L.elem_off = J.elem_off; L.word_off = J.word_off; L.size = J.size; L.bits = J.bits; L.nlevels = 1 << J.bits;
    L.block_off = J.block_off;
    const int k = kk + p.worker0;
    const int lane = threadIdx.x & 31;
    const int64_t kl = (int64_t)k * p.num_layers + layer;
    pdl_wait();

    // Everything below depends on the job record only, so all of it is requested at once: the norms, this thread's
    // two pieces of the search table, the zero-row masks of its block, the levels of its table entries.
    const float ncur = load_f32(norms + kl);
    const float nprev = prev_norms ? load_f32(prev_norms + kl) : 0.0f;
    const float rn = load_f32(p.rnorm + kl);
    const int2 how = load_i32x2(st.how + layer);
    const uint4* lsrc = reinterpret_cast<const uint4*>(st.lut + (int64_t)layer * kLutEntries);
    const uint4 lut0 = load_u32x4(lsrc + threadIdx.x), lut1 = load_u32x4(lsrc + kQThreads + threadIdx.x);
    uint32_t mcur = 0, mprev = 0;
    if (threadIdx.x < tile.nblocks) {
        // a previous message whose masks are unknown is taken as nonzero everywhere
        const int64_t mb = (int64_t)k * p.total_blocks + L.block_off + tile.block0 + threadIdx.x;
        mcur = load_u8(p.row_mask + mb);
        mprev = (!kStat || !prev_packed) ? 0u : (p.row_mask_prev ? load_u8(p.row_mask_prev + mb) : 0xffu);
    }
    float lc = 0.f, lp = 0.f;
    float2 lg = make_float2(0.f, 0.f);
    if (threadIdx.x < L.nlevels) {
        lc = load_f32(levels_cur + (int64_t)layer * kLevelStride + threadIdx.x);
        lp = load_f32(levels_prev + (int64_t)layer * kLevelStride + threadIdx.x);
        lg = load_f32x2(st.ld + (int64_t)layer * kMaxLevels + threadIdx.x);
    }
    {
        uint4* ldst = reinterpret_cast<uint4*>(sm + kSmLut);
        ldst[threadIdx.x] = lut0;
        ldst[kQThreads + threadIdx.x] = lut1;
        if (threadIdx.x < L.nlevels) {
            const float cv = __fmul_rn(ncur, lc), pv = __fmul_rn(nprev, lp);
            reinterpret_cast<float2*>(sm + kSmLd)[threadIdx.x] = lg;
            reinterpret_cast<float2*>(sm + kSmTcur)[threadIdx.x] = make_float2(cv, -cv);
            reinterpret_cast<float2*>(sm + kSmTprev)[threadIdx.x] = make_float2(pv, -pv);
        }
        if (kHist) {
            uint32_t* h = reinterpret_cast<uint32_t*>(sm + kSmHist);
            for (int i = threadIdx.x; i < LQ_HIST_STRIDE; i += kQThreads) h[i] = 0;
        }
    }
    if (threadIdx.x == 0) {
        *reinterpret_cast<int2*>(sm + kSmHow) = how;
        // whether the tile ends in the layer's partial block, which is not part of a message of zeros
        *reinterpret_cast<int*>(sm + kSmLast) = rn != 0.0f && (J.block0 + J.nblocks) * (int64_t)kBlockCoords > J.size;
    }
    uint8_t* rows_cur = sm + kSmRows;
    uint8_t* rows_prev = rows_cur + kTileBlocks;
    if (threadIdx.x < tile.nblocks) {
        rows_cur[threadIdx.x] = (uint8_t)mcur;
        rows_prev[threadIdx.x] = (uint8_t)mprev;
    }
    __syncthreads();

    WarpCtx c;
    c.g = fresh(grads + (int64_t)kk * p.padded_elems + L.elem_off);
    c.nfull = L.size / kBlockCoords;
    c.lane = lane;
    QuantEnv ev;
    ev.lut = base + kSmLut; ev.ld = base + kSmLd; ev.tprev = base + kSmTprev;
    ev.r = rn;
    ev.hist = reinterpret_cast<uint32_t*>(sm + kSmHist);
    if (step == LQ_STEP_AUTO) step = (uint32_t)p.scalars->t;      // the plan's own iteration counter (graph replays)
    const PhiloxConsts pc = philox_fold((uint32_t)layer, (uint32_t)k, step, p.seed_lo, p.seed_hi);
    uint32_t* out = packed + (int64_t)k * p.packed_words + L.word_off;
    const uint32_t* prev = prev_packed ? fresh(prev_packed + (int64_t)k * p.packed_words + L.word_off) : nullptr;

    double stat = quantize_blocks<kWidth, kHist, kStat>(p, pc, c, tile, L.bits, how.x & 3, out, prev, ev, rows_cur, rows_prev, base + kSmRing);
    if (*reinterpret_cast<volatile int*>(sm + kSmLast)) {
        if constexpr (kWidth != 0) {
            stat += quantize_last_block<kWidth, kHist, kStat>(p, grads, step, packed, prev_packed);
        } else {
            switch (L.bits) {
#define LQ_CASE(BB) case BB: stat += quantize_last_block<BB, kHist, kStat>(p, grads, step, packed, prev_packed); break;
                LQ_CASE(1) LQ_CASE(2) LQ_CASE(3) LQ_CASE(4) LQ_CASE(5) LQ_CASE(6) LQ_CASE(7) LQ_CASE(8)
#undef LQ_CASE
                default: break;
            }
        }
    }
    const double total = block_reduce<false>(stat, reinterpret_cast<double*>(sm + kSmScratch));
    if (threadIdx.x == 0) p.stat_partial[(int64_t)k * p.num_tiles + tile_id] = total;

    if (kHist) {
        __syncthreads();
        uint32_t* h = hist + kl * LQ_HIST_STRIDE;
        for (int i = threadIdx.x; i < LQ_NUM_BINS; i += blockDim.x)
            if (ev.hist[i]) atomicAdd(h + i, ev.hist[i]);
    }
}

// Adds the per-tile statistic partials of one (layer, worker) in a fixed order, and keeps the scalars as this message
// found them.
__global__ void __launch_bounds__(128) stat_finalize_kernel(PlanDev p)
{
    __shared__ double scratch[4];
    pdl_launch_next();
    const int m = blockIdx.x, k = blockIdx.y + p.worker0;
    const LayerDesc L = p.layers[m];
    pdl_wait();
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) p.scalars[1] = p.scalars[0];
    const double* part = p.stat_partial + (int64_t)k * p.num_tiles + L.first_tile;
    double acc = 0.0;
    for (int i = threadIdx.x; i < L.ntiles; i += blockDim.x) acc += part[i];
    const double total = block_reduce<false>(acc, scratch);
    if (threadIdx.x == 0) p.sq_diff[(int64_t)k * p.num_layers + m] = total;
}

// One CTA per layer: derives the encode-side tables from the layer's levels, which it also copies to `kept` (the level
// table of the messages to come).
//   ld[tau]  = {l_tau, l_{tau+1} - l_tau}                 tau = 0..n-2 (other entries: {l_tau, 0})
//   lut[bin] = (tau0 << 19) - (bin << 19) + (2^19 - low)    bin = bits(u) >> 19, i.e. the values [lo, hi) with bits(lo) = bin <<
//              19; tau0 = last level (<= n-2) at or below lo; low = the low 19 bits of l_{tau0+1} if that level
//              (<= n-2) lies inside the bin, else 2^19, so that  (lut[bin] + bits(u)) >> 19 = tau
// Layers with two levels in such a bin and 5 bits or more get bins of 2^s patterns from just below the first level up to
// 1.0, with the finest s that 2048 bins allow and the same entries (s for 19, bits(u) counted from the first bin's edge).  If two
// levels still share a bin, or below 5 bits, a byte table over the top 15 bits takes the same 8 KB:
//   lut8[bits(u) >> 17] = tau0 of that finer bin; tau is found by stepping up while l_{tau+1} <= u, at most R times,
//   R = the most levels inside one bin.
// (8-bit uniform levels took the byte table and 3 steps before: 201 M coordinates in 593 us, 419 us with one lookup.)
__global__ void __launch_bounds__(256) build_search_kernel(PlanDev p, const float* levels, float* kept, SearchTables t)
{
    __shared__ float lev[kMaxLevels];
    __shared__ int shared_bin, most;
    pdl_launch_next();
    pdl_wait();
    const int m = blockIdx.x;
    const int n = p.layers[m].nlevels;
    if (threadIdx.x == 0) { shared_bin = 0; most = 0; }
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        lev[i] = levels[(int64_t)m * kLevelStride + i];
        kept[(int64_t)m * kLevelStride + i] = lev[i];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kMaxLevels; i += blockDim.x) {
        float2 e = make_float2(i < n ? lev[i] : 0.f, 0.f);
        if (i <= n - 2) e.y = __fsub_rn(lev[i + 1], lev[i]);
        t.ld[(int64_t)m * kMaxLevels + i] = e;
    }
    // the last level <= n - 2 at or below x
    auto tau_of = [&](float x) {
        int tau = 0;
        for (int s = n >> 1; s > 0; s >>= 1)
            if (lev[tau + s] <= x) tau += s;
        return min(tau, n - 2);
    };
    constexpr uint32_t kOne = 0x3f800000u;               // bins past 1.0 (and Inf / NaN) behave like the bin of 1.0
    uint32_t* lut = t.lut + (int64_t)m * kLutEntries;
    // bins of 2^s patterns, bin i from off + i 2^s on; returns whether two levels share one
    auto fill = [&](int s, uint32_t off) {
        const uint32_t mask = (1u << s) - 1u;
        for (int bin = threadIdx.x; bin < kLutEntries; bin += blockDim.x) {
            const uint32_t lob = off + ((uint32_t)bin << s);
            const bool top = lob >= kOne;
            const int tau0 = tau_of(__uint_as_float(top ? kOne : lob));
            uint32_t low = mask + 1u;
            if (!top && tau0 + 1 <= n - 2) {
                const uint32_t nb = __float_as_uint(lev[tau0 + 1]);
                if ((nb >> s) == (lob >> s)) {                              // l_{tau0+1} > lo lies inside this bin
                    low = nb & mask;
                    if (tau0 + 2 <= n - 2 && (__float_as_uint(lev[tau0 + 2]) >> s) == (lob >> s)) atomicOr(&shared_bin, 1);
                }
            }
            lut[bin] = (((uint32_t)tau0 - (uint32_t)bin) << s) + (mask + 1u - low);
        }
        __syncthreads();
        const int r = shared_bin;
        __syncthreads();
        if (threadIdx.x == 0) shared_bin = 0;
        __syncthreads();
        return r != 0;
    };
    int2 how = make_int2(kSearchOctave, 0);
    bool dense = fill(19, 0u);
    if (dense && n >= 1 << kWindowBits) {
        const uint32_t first = __float_as_uint(lev[1]);
        int s = 3;                                                         // (quantize_coord shifts by s - 3)
        while ((kOne >> s) - (first >> s) + 1u >= (uint32_t)kLutEntries) ++s;
        const uint32_t off = ((first >> s) - 1u) << s;                     // (a level is at least 2^-100: no wrap)
        how = make_int2(kSearchWindow | (s << 2), (int)off);
        dense = fill(s, off);
    }
    if (dense) {
        uint8_t* lut8 = reinterpret_cast<uint8_t*>(lut);
        for (int bin = threadIdx.x; bin < 4 * kLutEntries; bin += blockDim.x) {
            const uint32_t lob = (uint32_t)bin << 17;
            const bool top = lob >= kOne;
            const int tau0 = tau_of(__uint_as_float(top ? kOne : lob));
            lut8[bin] = (uint8_t)tau0;
            int inside = 0;
            while (!top && tau0 + 1 + inside <= n - 2 && (__float_as_uint(lev[tau0 + 1 + inside]) >> 17) == (uint32_t)bin) ++inside;
            if (inside) atomicMax(&most, inside);
        }
        __syncthreads();
        how = make_int2(kSearchStep | (most << 2), 0);
    }
    if (threadIdx.x == 0) t.how[m] = how;
}

cudaError_t launch_build_search(const PlanDev& p, const float* levels, float* kept, SearchTables t, cudaStream_t s)
{
    if (p.num_layers == 0) return cudaSuccess;
    return launch(build_search_kernel, (unsigned)p.num_layers, 256, 0, s, p, levels, kept, t);
}

cudaError_t launch_quantize(const PlanDev& p, const float* grads, uint32_t step, uint32_t* packed,
                            const float* norms, uint32_t* hist, const uint32_t* prev_packed,
                            const float* prev_norms, const float* levels_cur,
                            const float* levels_prev, SearchTables t, bool need_stat, cudaStream_t s)
{
    if (p.num_tiles == 0) return cudaSuccess;
    // the ring follows the tables; the histogram (histogram mode only) follows the ring
    constexpr unsigned smem = kSmTables + kRingBytes + kSmSlack, smem_hist = smem + LQ_HIST_STRIDE * 4;
    using Kernel = void (*)(PlanDev, const float*, uint32_t, uint32_t*, const float*, uint32_t*, const uint32_t*, const float*,
                            const float*, const float*, SearchTables);
#define LQ_ALL(H, S) {quantize_pack_kernel<0, H, S>, quantize_pack_kernel<1, H, S>, quantize_pack_kernel<2, H, S>, \
                      quantize_pack_kernel<3, H, S>, quantize_pack_kernel<4, H, S>, quantize_pack_kernel<5, H, S>, \
                      quantize_pack_kernel<6, H, S>, quantize_pack_kernel<7, H, S>, quantize_pack_kernel<8, H, S>}
    static const Kernel kernels[3][9] = {LQ_ALL(false, false), LQ_ALL(false, true), LQ_ALL(true, true)};
#undef LQ_ALL
    static std::atomic<uint64_t> configured[3][9];
    const int mode = hist ? 2 : need_stat ? 1 : 0;
    const int width = p.least_bits == p.most_bits ? p.most_bits : 0;
    const Kernel kernel = kernels[mode][width];
    const cudaError_t e = opt_in_shared_memory(configured[mode][width], (int)smem_hist, kernel);
    if (e != cudaSuccess) return e;
    return launch_as(encoder_dependent(p), kernel, dim3((unsigned)p.num_tiles, (unsigned)p.worker_count), kQThreads,
                     hist ? smem_hist : smem, 1, s, p, grads, step, packed, norms, hist, prev_packed, prev_norms, levels_cur,
                     levels_prev, t);
}

cudaError_t launch_stat_finalize(const PlanDev& p, cudaStream_t s)
{
    return launch(stat_finalize_kernel, dim3((unsigned)p.num_layers, (unsigned)p.worker_count), 128, 0, s, p);
}

}  // namespace lq
