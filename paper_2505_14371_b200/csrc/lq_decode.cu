// DECODE + aggregate of the K workers' messages, alone or fused with the optimistic dual averaging
// update (Algorithm 1 lines 15-18 and line 10 of the next iteration; Eq. ODA; Eq. general_stepsize).
//
// One CTA of 4 warps per piece of a layer (up to 32 blocks of 1024 coordinates, one block per warp at a time; in plans
// with fewer blocks than the GPU has warps to give them, the 4 warps share a block, 2 rows each).  A lane owns the same 32
// coordinates it owned at encode time: it looks the signed decoded values up by symbol in a per-(worker, layer) table in
// shared memory, sums them in worker order in registers, and finishes with float4 reads of Y and X_1 and float4 writes of
// Y and X_{t+3/2}.  Every packed word and every state element is touched once.
//
// Everything a warp reads from global memory travels by 16-byte asynchronous copies into shared memory of its own: the
// words of a few workers at a time (a unit), two units deep, and the block's rows of Y and X_1, which arrive while the
// words are being decoded.  So 16 warps per SM keep up to 210 KB in flight, no load waits in a register, and the accumulators
// of a whole block fit: per symbol remain shift, mask (which also adds the table's address: tables start at multiples of
// their size), look-up and add.  The look-ups bound it for many narrow messages (one pass of the SM's shared-memory
// pipe per 32 symbols), DRAM otherwise.
#include <algorithm>

#include "lq_internal.cuh"

namespace lq {

constexpr int kUnitPlanes = 20;                          // 128-byte planes of words in a unit, most
constexpr uint32_t kUnitBytes = kUnitPlanes * 128;
constexpr uint32_t kStateBytes = 2 * kBlockCoords * 4;   // a block's rows of Y, then of X_1
constexpr uint32_t kTableBytes = 32 * 1024;              // most shared memory for value tables

// workers per unit, and bytes of one worker's words of a block
template <int B>
constexpr int kUnitWorkers = kUnitPlanes / (B + 1) < 16 ? kUnitPlanes / (B + 1) : 16;
template <int B>
constexpr uint32_t kBlockBytes = (B + 1) * 128;
// workers whose value tables (2^(b+1) floats each) are in shared memory at once: whole units
template <int B>
constexpr int kTableWorkers = ((int)(kTableBytes >> (B + 3)) / kUnitWorkers<B>) * kUnitWorkers<B>;

// The rates one QODA update uses: X_{t+1} = X_1 + eta Y_{t+1}, X_{t+3/2} = X_{t+1} - gamma gbar; eta_cur made X_t.
struct Rates { float eta, gamma, eta_cur; };

struct DecodeArgs {
    const uint8_t* masks;    // [K][total_blocks] zero-row masks of the message's input (K <= 32), or nullptr
    const uint32_t* packed;
    const float* norms;
    const float* levels;
    const float* X1;
    float* Y;
    float* Xhalf;
    float* X;
    float* gbar;
    bool form_rates;         // mode 1: the CTAs form the step's rates (rates_in_decoder), else a kernel before has done it
    bool vec;                // packed (and in bucket scope norms) start on a 16-byte boundary
    uint32_t table_bytes;    // shared memory for the value tables, a multiple of their size
};

// Fills the value tables of workers k0 .. k0 + kc - 1 of one layer (all threads); in bucket scope one table of plain
// signed levels.  Symbol = 2 * idx + sign.
template <bool kBucket>
__device__ __forceinline__ void fill_tables(const PlanDev& p, const LayerDesc& L, int layer, const DecodeArgs& a,
                                            float2* table, int k0, int kc)
{
    const int n = (kBucket ? 1 : kc) << L.bits;
    for (int i = threadIdx.x; i < n; i += kDecThreads) {
        const int kk = i >> L.bits, j = i & (L.nlevels - 1);
        const float lv = load_f32(a.levels + (int64_t)layer * kLevelStride + j);
        const float mag = kBucket ? lv : __fmul_rn(load_f32(a.norms + (int64_t)(k0 + kk) * p.num_layers + layer), lv);
        table[i] = make_float2(mag, -mag);
    }
}

// What a warp needs to walk its blocks.
struct Walk {
    const uint32_t* words;       // the layer's words in worker 0's message
    const float* bnorms;         // bucket scope: the layer's bucket norms of worker 0
    int64_t base;                // the layer's first element in a state row
    int32_t block0, nblocks;     // the CTA's blocks of the layer
    int32_t size;                // d_m
    uint32_t tables, units, state;   // shared-memory addresses: value tables, this warp's two units, its state rows
    int lane, warp;
};

// Which 16-byte pieces of a unit a lane copies: piece 32 i + lane is piece (32 i + lane) % (8 C) of the words of the
// unit's worker (32 i + lane) / (8 C).  Worked out once per warp.
template <int B>
struct UnitPieces {
    static constexpr int kPer = (B + 1) * 8, kCount = (kUnitWorkers<B> * kPer + 31) / 32;
    int64_t off[kCount];         // bytes from the unit's first word
    uint32_t worker[kCount];     // the worker's bit (0: no such piece)
    __device__ __forceinline__ UnitPieces(int64_t packed_words, int lane)
    {
#pragma unroll
        for (int i = 0; i < kCount; ++i) {
            const int c = 32 * i + lane, kk = c / kPer;
            off[i] = kk * packed_words * 4 + (c - kk * kPer) * 16;
            worker[i] = kk < kUnitWorkers<B> ? 1u << kk : 0u;
        }
    }
};

// Starts the copies of the words of the workers k0 + (set bits of `live`) of block blk into a unit; in bucket scope
// every worker's 8 norms of the block go behind the words' space.
template <int B, bool kBucket>
__device__ __forceinline__ void request_unit(const PlanDev& p, const DecodeArgs& a, const Walk& w, const UnitPieces<B>& up,
                                             uint32_t unit, int64_t blk, int k0, uint32_t live)
{
    constexpr int C = B + 1;
    const uint32_t* src = w.words + (int64_t)k0 * p.packed_words + blk * (C * 32);
    const float* bn = kBucket ? w.bnorms + ((int64_t)k0 * p.total_blocks + blk) * 8 : nullptr;
    if (a.vec) {
        const char* from = reinterpret_cast<const char*>(src);
#pragma unroll
        for (int i = 0; i < UnitPieces<B>::kCount; ++i)
            if (live & up.worker[i]) cp_async16(unit + 16 * w.lane + 512 * i, from + up.off[i], 16);
        if (kBucket && w.lane < 2 * kUnitWorkers<B> && ((live >> (w.lane >> 1)) & 1u))
            cp_async16(unit + kUnitBytes + 16 * w.lane, bn + (w.lane >> 1) * p.total_blocks * 8 + 4 * (w.lane & 1), 16);
        return;
    }
    for (uint32_t m = live; m; m &= m - 1) {
        const int kk = __ffs(m) - 1;
#pragma unroll
        for (int i = 0; i < C; ++i)
            cp_async4(unit + kk * kBlockBytes<B> + 128 * i + 4 * w.lane, src + kk * p.packed_words + 32 * i + w.lane);
        if (kBucket && w.lane < 8)
            cp_async4(unit + kUnitBytes + 32 * kk + 4 * w.lane, bn + kk * p.total_blocks * 8 + w.lane);
    }
}

// symbol p of the lane's words as (4 * symbol) | table
template <int C>
__device__ __forceinline__ uint32_t value_addr(const uint32_t (&w)[C], int p, uint32_t table)
{
    const int off = p * C, i = off >> 5, s = off & 31;
    constexpr uint32_t mask4 = ((1u << C) - 1u) << 2;
    uint32_t v;
    if (s + C <= 32) v = s >= 2 ? (w[i] >> (s - 2)) : (w[i] << (2 - s));
    else             v = __funnelshift_r(w[i], w[i + 1], s - 2);      // s >= 2 whenever a symbol straddles
    return (v & mask4) | table;
}

// Adds a unit's workers to the sums of rows row0 .. row0 + kRows - 1, in worker order.  Two neighbours are added by one
// instruction: 33.6 M coordinates of 16 workers at 2 bits 102.7 -> 100.5 us (75 % of the issue slots are used, 5.1 warp
// instructions per 32 symbols).
// A clear bit of `live`: that worker's block is all zero words, which would add +0 to sums that are never -0.
// Of 2 rows (row0 = 2 x the warp) the words are first moved so that they start with the rows' symbols: the warps run the same code,
// which in such small grids takes longer to fetch than to run (8192 coordinates, 8 workers: the step 12.0 -> 10.0 us; 203 530 and
// 4: 20.5 -> 19.0).
template <int B, int kRows, bool kBucket>
__device__ __forceinline__ void add_unit(float (&acc)[4 * kRows], uint32_t unit, int lane, int row0, uint32_t table, uint32_t live)
{
    constexpr int C = B + 1, kWords = (4 * kRows * C + 31) >> 5;
    const int w0 = (4 * row0 * C) >> 5, shift = (4 * row0 * C) & 31;
    uint32_t at = unit + 4 * lane + 128 * w0, norm_at = unit + kUnitBytes + 4 * row0;
#pragma unroll 1
    for (; live; live >>= 1, at += kBlockBytes<B>, table += kBucket ? 0u : 8u << B, norm_at += 32) {
        if (!(live & 1u)) continue;
        uint32_t w[C];
#pragma unroll
        for (int i = 0; i < kWords; ++i) w[i] = lds_u32(at + 128 * i);
        if (kRows != 8 && (8 * C) % 32 != 0) {
            uint32_t behind = w0 + kWords < C ? lds_u32(at + 128 * kWords) : 0u;
#pragma unroll
            for (int i = 0; i < kWords; ++i) w[i] = __funnelshift_r(w[i], i + 1 < kWords ? w[i + 1] : behind, shift);
        }
        float nr[kRows];
        if (kBucket) {
#pragma unroll
            for (int j = 0; j < kRows; ++j) nr[j] = lds_f32(norm_at + 4 * j);
        }
#pragma unroll
        for (int i = 0; i < 4 * kRows; i += 2) {
            float v0 = lds_f32(value_addr<C>(w, i, table)), v1 = lds_f32(value_addr<C>(w, i + 1, table));
            if (kBucket) { v0 = __fmul_rn(v0, nr[i >> 2]); v1 = __fmul_rn(v1, nr[i >> 2]); }
            add_f32x2(acc[i], acc[i + 1], v0, v1);
        }
    }
}

template <int kRows>
__device__ __forceinline__ void request_state(const DecodeArgs& a, const Walk& w, int64_t blk, int row0)
{
#pragma unroll
    for (int jj = 0; jj < kRows; ++jj) {
        const int j = row0 + jj;
        const int64_t at = blk * kBlockCoords + 128 * j + 4 * w.lane;
        if (at < w.size) {
            cp_async16(w.state + 512 * j + 16 * w.lane, a.Y + w.base + at, 16);
            cp_async16(w.state + kStateBytes / 2 + 512 * j + 16 * w.lane, a.X1 + w.base + at, 16);
        }
    }
}

// The rows row0 .. of one block, from their sums: the mean, then the update.
template <int kMode, int kRows>
__device__ __forceinline__ void finish_block(const DecodeArgs& a, const Walk& w, int64_t blk, int row0, const float (&acc)[4 * kRows],
                                             float invK, const Rates& rt, bool sent, double& lam_acc, double& mu_acc)
{
    constexpr bool kQoda = kMode >= 1, kAlt = kMode == 2;
    const float eta = rt.eta, gamma = rt.gamma;
#pragma unroll
    for (int jj = 0; jj < kRows; ++jj) {
        const int64_t at = blk * kBlockCoords + 128 * (row0 + jj) + 4 * w.lane, pos = w.base + at;
        if (at >= w.size) continue;
        float4 g;
        g.x = __fmul_rn(acc[4 * jj + 0], invK);
        g.y = __fmul_rn(acc[4 * jj + 1], invK);
        g.z = __fmul_rn(acc[4 * jj + 2], invK);
        g.w = __fmul_rn(acc[4 * jj + 3], invK);
        if (a.gbar) *reinterpret_cast<float4*>(a.gbar + pos) = g;
        if (kQoda) {
            const float4 y0 = lds_f32x4(w.state + 512 * (row0 + jj) + 16 * w.lane);
            const float4 x1 = lds_f32x4(w.state + kStateBytes / 2 + 512 * (row0 + jj) + 16 * w.lane);
            float4 y, x, h;
            y.x = __fsub_rn(y0.x, g.x); y.y = __fsub_rn(y0.y, g.y);
            y.z = __fsub_rn(y0.z, g.z); y.w = __fsub_rn(y0.w, g.w);
            x.x = fmaf(eta, y.x, x1.x); x.y = fmaf(eta, y.y, x1.y);
            x.z = fmaf(eta, y.z, x1.z); x.w = fmaf(eta, y.w, x1.w);
            h.x = fmaf(-gamma, g.x, x.x); h.y = fmaf(-gamma, g.y, x.y);
            h.z = fmaf(-gamma, g.z, x.z); h.w = fmaf(-gamma, g.w, x.w);
            if (kAlt) {
                // this iteration's terms of lambda = sum ||gbar||^2 and mu = sum ||X_t - X_{t+1}||^2, with
                // X_t recomputed from Y_t and the rate that produced it; padding coordinates do not count
                const float gv[4] = {g.x, g.y, g.z, g.w};
                const float dv[4] = {__fsub_rn(fmaf(rt.eta_cur, y0.x, x1.x), x.x), __fsub_rn(fmaf(rt.eta_cur, y0.y, x1.y), x.y),
                                     __fsub_rn(fmaf(rt.eta_cur, y0.z, x1.z), x.z), __fsub_rn(fmaf(rt.eta_cur, y0.w, x1.w), x.w)};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (at + e < w.size) {
                        const double gd = (double)gv[e], dd = (double)dv[e];
                        lam_acc = fma(gd, gd, lam_acc);
                        mu_acc = fma(dd, dd, mu_acc);
                    }
                }
            }
            if (sent) *reinterpret_cast<float4*>(a.Y + pos) = y;         // no worker sent anything here: y = y0 - 0
            *reinterpret_cast<float4*>(a.Xhalf + pos) = h;
            if (a.X) *reinterpret_cast<float4*>(a.X + pos) = x;
        }
    }
}

// A warp's blocks: warp, warp + 4, ... of the CTA's (kRows = 8), or its two rows of all of them (kRows = 2).
// The next unit's words are always requested before the current unit is waited for; the rows of Y and X_1 as soon as
// the block before is finished.  Per unit one copy group, per block one more for the state, so a fixed number of
// younger groups may be under way at every wait.
template <int B, int kMode, bool kBucket, int kRows>
__device__ __forceinline__ void decode_blocks(const PlanDev& p, const LayerDesc& L, int layer, const DecodeArgs& a, const Walk& w,
                                           float2* table, const Rates* rates, uint32_t my_live, double* sums)
{
    constexpr bool kQoda = kMode >= 1;
    constexpr int kUW = kUnitWorkers<B>, kTW = kBucket ? 1 << 20 : kTableWorkers<B>;
    constexpr int kStep = kRows == 8 ? kDecWarps : 1;
    constexpr uint32_t kUnitStride = kUnitBytes + (kBucket ? 32 * 16 : 0);
    const int K = p.num_workers, nu = (K + kUW - 1) / kUW, row0 = kRows == 8 ? 0 : kRows * w.warp;
    const float invK = __fdiv_rn(1.0f, (float)K);
    // the workers of unit u that sent anything in a block with `live` (kept for up to 32 workers; of more, all are read)
    auto unit_live = [&](uint32_t live, int u) {
        const int k0 = u * kUW;
        const uint32_t m = K <= 32 ? live >> k0 : 0xffffffffu;
        return K - k0 < kUW ? m & ((1u << (K - k0)) - 1u) : m & ((1u << kUW) - 1u);
    };
    auto block_live = [&](int i) { return __reduce_or_sync(0xffffffffu, w.lane == i ? my_live : 0u); };   // uniform

    const UnitPieces<B> up(p.packed_words, w.lane);
    int b = kRows == 8 ? w.warp : 0, i = 0;
    uint32_t live = block_live(0);
    if (b < w.nblocks) request_unit<B, kBucket>(p, a, w, up, w.units, w.block0 + b, 0, unit_live(live, 0));
    cp_async_commit();
    if (kQoda) {
        if (b < w.nblocks) request_state<kRows>(a, w, w.block0 + b, row0);
        cp_async_commit();
    }
    fill_tables<kBucket>(p, L, layer, a, table, 0, min(K, kTW));
    __syncthreads();
    const Rates rt = *rates;
    double lam_acc = 0.0, mu_acc = 0.0;
    uint32_t stage = 0;
    // with more workers than tables fit, all warps take the same number of turns (the refills are CTA-wide)
    for (int b0 = 0; K > kTW ? b0 < w.nblocks : b < w.nblocks; b0 += kStep, b += kStep, ++i) {
        const bool active = b < w.nblocks;
        const int64_t blk = w.block0 + b;
        const uint32_t next_live = b + kStep < w.nblocks ? block_live(i + 1) : 0u;
        float acc[4 * kRows];
#pragma unroll
        for (int c = 0; c < 4 * kRows; ++c) acc[c] = 0.0f;
        for (int u = 0; u < nu; ++u) {
            const uint32_t other = w.units + (stage ^ 1u) * kUnitStride;
            if (u + 1 < nu) { if (active) request_unit<B, kBucket>(p, a, w, up, other, blk, (u + 1) * kUW, unit_live(live, u + 1)); }
            else if (b + kStep < w.nblocks) request_unit<B, kBucket>(p, a, w, up, other, blk + kStep, 0, unit_live(next_live, 0));
            cp_async_commit();
            const int k0 = u * kUW;
            int k_in = k0;                                        // index of the unit's first worker in the tables
            if (!kBucket && K > kTW) {
                k_in = k0 % kTW;
                if (k_in == 0 && (b0 > 0 || u > 0)) {
                    __syncthreads();
                    fill_tables<kBucket>(p, L, layer, a, table, k0, min(kTW, K - k0));
                    __syncthreads();
                }
            }
            if (kQoda && u == 0) cp_async_wait<2>(); else cp_async_wait<1>();
            __syncwarp();                                         // a lane reads what other lanes have copied
            if (active)
                add_unit<B, kRows, kBucket>(acc, w.units + stage * kUnitStride, w.lane, row0,
                                            w.tables + (kBucket ? 0 : (uint32_t)k_in << (B + 3)), unit_live(live, u));
            __syncwarp();                                         // ... and the unit may be overwritten
            stage ^= 1u;
        }
        if (kQoda) cp_async_wait<1>();
        if (active) finish_block<kMode, kRows>(a, w, blk, row0, acc, invK, rt, live != 0u, lam_acc, mu_acc);
        if (kQoda) {
            if (b + kStep < w.nblocks) request_state<kRows>(a, w, blk + kStep, row0);
            cp_async_commit();
        }
        live = next_live;
    }
    cp_async_wait<0>();
    if (kMode == 2) { sums[0] = lam_acc; sums[1] = mu_acc; }
}

// S_t = S_{t-1} + (sum over workers and layers of the squared differences) / K^2, eta_{t+1} = fp32((1 + S_t)^(-1/2)).
__device__ __forceinline__ QodaScalars next_scalars(const QodaScalars& q0, double total, int num_workers)
{
    QodaScalars q = q0;
    const double K = (double)num_workers;
    const double delta = total / (K * K);
    q.last_delta = delta;
    q.S = q.S + delta;
    q.eta = (float)(1.0 / sqrt(1.0 + q.S));
    q.gamma = q.eta;
    q.t = q.t + 1;
    return q;
}

// The sum of sq_diff over workers and layers in a fixed order (all threads of the CTA; valid in thread 0).
__device__ __forceinline__ double sum_sq_diff(const PlanDev& p, double* scratch)
{
    const int n = p.num_workers * p.num_layers;
    double acc = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) acc += p.sq_diff[i];
    return block_reduce<false>(acc, scratch);
}

// kSplit: the 4 warps share every block, 2 rows each.
template <int kMode, bool kBucket, bool kSplit>
__global__ void __launch_bounds__(kDecThreads, kMode == 0 ? 5 : 4) decode_kernel(PlanDev p, DecodeArgs a)
{
    extern __shared__ __align__(1024) unsigned char dec_smem[];
    constexpr bool kAlt = kMode == 2;
    constexpr uint32_t kUnitStride = kUnitBytes + (kBucket ? 32 * 16 : 0);
    constexpr uint32_t kWarpBytes = 2 * kUnitStride + (kMode >= 1 ? kStateBytes : 0);
    pdl_launch_next();
    const int ncta = p.num_tiles << p.dec_shift;
    const Tile tile = p.tiles[blockIdx.x >> p.dec_shift];              // this CTA takes a piece of it
    const int first = (blockIdx.x & ((1 << p.dec_shift) - 1)) * p.dec_blocks;
    if (first >= tile.nblocks) {
        pdl_wait();
        if (kAlt && threadIdx.x == 0) { p.alt_partial[blockIdx.x] = 0.0; p.alt_partial[ncta + blockIdx.x] = 0.0; }
        return;
    }
    const int layer = tile.layer;
    const LayerDesc L = p.layers[layer];
    // tables at a multiple of their size, then a few words for the reductions, then the warps' units and state rows
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(dec_smem);
    const uint32_t table_size = 8u << L.bits;
    const uint32_t tables = (base + table_size - 1) & ~(table_size - 1);
    unsigned char* after = dec_smem + a.table_bytes;
    double* scratch = reinterpret_cast<double*>(after);
    Rates* rates = reinterpret_cast<Rates*>(after + 64);
    Walk w;
    w.lane = threadIdx.x & 31; w.warp = threadIdx.x >> 5;
    w.words = a.packed + L.word_off;
    w.bnorms = a.norms + L.block_off * 8;
    w.base = L.elem_off;
    w.block0 = tile.block0 + first;
    w.nblocks = min(p.dec_blocks, tile.nblocks - first);
    w.size = (int32_t)L.size;
    w.tables = tables;
    w.units = base + a.table_bytes + 128 + w.warp * kWarpBytes;
    w.state = w.units + 2 * kUnitStride;
    float2* table = reinterpret_cast<float2*>(dec_smem + (tables - base));
    pdl_wait();

    // lane i: which workers sent anything in this warp's i-th block (all of them when that is not known)
    uint32_t my_live = 0xffffffffu;
    if (!kBucket && a.masks) {
        constexpr int kStep = kSplit ? 1 : kDecWarps;
        const uint8_t* mk = a.masks + (int64_t)min(w.lane, p.num_workers - 1) * p.total_blocks + L.block_off + w.block0;
        for (int i0 = 0; kStep * i0 < w.nblocks; i0 += 8) {
            uint32_t m[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int b = (kSplit ? 0 : w.warp) + kStep * (i0 + i);
                m[i] = b < w.nblocks && w.lane < p.num_workers ? load_u8(mk + b) : 0u;
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint32_t v = __ballot_sync(0xffffffffu, m[i] != 0u);
                if (w.lane == i0 + i) my_live = v;
            }
        }
    }
    if (kMode == 1 && a.form_rates) {
        const double total = sum_sq_diff(p, scratch);
        if (threadIdx.x == 0) {
            const QodaScalars q = next_scalars(p.scalars[1], total, p.num_workers);
            *rates = Rates{q.eta, q.eta, 0.0f};
            if (blockIdx.x == 0) p.scalars[0] = q;
        }
    } else if (kMode >= 1) {
        if (threadIdx.x == 0)
            *rates = Rates{p.scalars->eta, kAlt ? p.scalars->gamma : p.scalars->eta, kAlt ? p.scalars->eta_cur : 0.0f};
    }
    double sums[2] = {0.0, 0.0};
    switch (L.bits) {
#define LQ_CASE(BB) case BB: decode_blocks<BB, kMode, kBucket, kSplit ? 2 : 8>(p, L, layer, a, w, table, rates, my_live, sums); break;
        LQ_CASE(1) LQ_CASE(2) LQ_CASE(3) LQ_CASE(4) LQ_CASE(5) LQ_CASE(6) LQ_CASE(7) LQ_CASE(8)
#undef LQ_CASE
        default: break;
    }
    if (kAlt) {                                  // one term per CTA, added in CTA order by the finalize kernel
        const double lam = block_reduce<false>(sums[0], scratch);
        const double mu = block_reduce<false>(sums[1], scratch);
        if (threadIdx.x == 0) { p.alt_partial[blockIdx.x] = lam; p.alt_partial[ncta + blockIdx.x] = mu; }
    }
}

// Eq. (Alt), before the update of iteration t: eta_{t+1} and gamma_{t+1} from the sums through iteration t-1.
__global__ void alt_scalars_kernel(PlanDev p, double qhat)
{
    pdl_launch_next();
    pdl_wait();
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        QodaScalars* q = p.scalars;
        q->eta_cur = q->eta;
        q->eta = (float)(1.0 / sqrt(1.0 + q->lambda + q->mu));
        q->gamma = (float)pow(1.0 + q->lambda, qhat - 0.5);
        q->t = q->t + 1;
    }
}

// Eq. (Alt), after the update: adds the CTAs' terms of this iteration to lambda and mu in a fixed order.
__global__ void __launch_bounds__(256) alt_finalize_kernel(PlanDev p)
{
    __shared__ double scratch[8];
    pdl_launch_next();
    pdl_wait();
    const int n = p.num_tiles << p.dec_shift;
    double lam = 0.0, mu = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) { lam += p.alt_partial[i]; mu += p.alt_partial[n + i]; }
    const double lam_t = block_reduce<false>(lam, scratch);
    const double mu_t = block_reduce<false>(mu, scratch);
    if (threadIdx.x == 0) { p.scalars->lambda += lam_t; p.scalars->mu += mu_t; }
}

// The rates of a step in a kernel of their own (plans with many layers and workers); one CTA, fixed summation order.
__global__ void __launch_bounds__(kThreads) qoda_scalars_kernel(PlanDev p)
{
    __shared__ double scratch[kWarps];
    pdl_launch_next();
    pdl_wait();
    const double total = sum_sq_diff(p, scratch);
    if (threadIdx.x == 0) p.scalars[0] = next_scalars(p.scalars[0], total, p.num_workers);
}

__global__ void qoda_init_kernel(PlanDev p, const float* __restrict__ X1, float* __restrict__ Y,
                                 float* __restrict__ Xhalf)
{
    const int64_t n4 = p.padded_elems / 4;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n4;
         i += (int64_t)gridDim.x * blockDim.x) {
        reinterpret_cast<float4*>(Y)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        reinterpret_cast<float4*>(Xhalf)[i] = reinterpret_cast<const float4*>(X1)[i];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        QodaScalars* q = p.scalars;
        q->S = 0.0; q->last_delta = 0.0; q->t = 1; q->eta = 1.0f;
        q->gamma = 1.0f; q->eta_cur = 1.0f; q->lambda = 0.0; q->mu = 0.0;
    }
}

// xsum += Xhalf in fp64 (the running sum behind the ergodic average of the half iterates)
__global__ void __launch_bounds__(256) average_kernel(const float* __restrict__ Xhalf, double* __restrict__ xsum, int64_t n4)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n4; i += (int64_t)gridDim.x * blockDim.x) {
        const float4 x = __ldcs(reinterpret_cast<const float4*>(Xhalf) + i);
        double2 a = reinterpret_cast<double2*>(xsum)[2 * i], b = reinterpret_cast<double2*>(xsum)[2 * i + 1];
        a.x += (double)x.x; a.y += (double)x.y; b.x += (double)x.z; b.y += (double)x.w;
        reinterpret_cast<double2*>(xsum)[2 * i] = a;
        reinterpret_cast<double2*>(xsum)[2 * i + 1] = b;
    }
}

cudaError_t launch_average(const PlanDev& p, const float* Xhalf, double* xsum, cudaStream_t s)
{
    const int64_t n4 = p.padded_elems / 4;
    const unsigned blocks = (unsigned)((n4 + 255) / 256 < kSms * 16 ? (n4 + 255) / 256 + 1 : kSms * 16);
    average_kernel<<<blocks, 256, 0, s>>>(Xhalf, xsum, n4);
    return cudaGetLastError();
}

cudaError_t launch_decode(const PlanDev& p, const uint32_t* packed, const float* norms,
                          const float* levels, const float* X1, float* Y, float* Xhalf, float* X,
                          float* gbar, int mode, const uint8_t* masks, cudaStream_t s)
{
    if (p.num_tiles == 0) return cudaSuccess;
    DecodeArgs a{masks, packed, norms, levels, X1, Y, Xhalf, X, gbar, rates_in_decoder(p), false, 0};
    a.vec = reinterpret_cast<uintptr_t>(packed) % 16 == 0 && (!p.bucket_norm || reinterpret_cast<uintptr_t>(norms) % 16 == 0);
    // room for the widest layer's tables (narrower layers' need less), plus what aligning 2 KB tables may skip
    const int tables = std::min(p.bucket_norm ? 1 : p.num_workers, (int)(kTableBytes >> (p.most_bits + 3)));
    a.table_bytes = ((uint32_t)tables << (p.most_bits + 3)) + (p.most_bits == 8 ? 1024u : 0u);
    a.table_bytes = (a.table_bytes + 127u) & ~127u;
    const bool split = p.dec_blocks == 1;
    const unsigned grid = (unsigned)p.num_tiles << p.dec_shift;
    const size_t smem = a.table_bytes + 128 + kDecWarps * (2 * (kUnitBytes + (p.bucket_norm ? 32 * 16 : 0)) + (mode ? kStateBytes : 0));
    using Kernel = void (*)(PlanDev, DecodeArgs);
    static const Kernel kernels[3][2][2] = {
        {{decode_kernel<0, false, false>, decode_kernel<0, false, true>}, {decode_kernel<0, true, false>, decode_kernel<0, true, true>}},
        {{decode_kernel<1, false, false>, decode_kernel<1, false, true>}, {decode_kernel<1, true, false>, decode_kernel<1, true, true>}},
        {{decode_kernel<2, false, false>, decode_kernel<2, false, true>}, {decode_kernel<2, true, false>, decode_kernel<2, true, true>}}};
    static std::atomic<uint64_t> configured{0};
    const cudaError_t e = opt_in_shared_memory(
        configured, 100 * 1024, kernels[0][0][0], kernels[0][0][1], kernels[0][1][0], kernels[0][1][1], kernels[1][0][0], kernels[1][0][1],
        kernels[1][1][0], kernels[1][1][1], kernels[2][0][0], kernels[2][0][1], kernels[2][1][0], kernels[2][1][1]);
    if (e != cudaSuccess) return e;
    return launch(kernels[mode][p.bucket_norm ? 1 : 0][split ? 1 : 0], grid, kDecThreads, smem, s, p, a);
}

cudaError_t launch_alt_scalars(const PlanDev& p, double qhat, cudaStream_t s)
{
    return launch(alt_scalars_kernel, 1, 32, 0, s, p, qhat);
}

cudaError_t launch_alt_finalize(const PlanDev& p, cudaStream_t s)
{
    if (p.num_tiles == 0) return cudaSuccess;
    return launch(alt_finalize_kernel, 1, 256, 0, s, p);
}

cudaError_t launch_qoda_scalars(const PlanDev& p, cudaStream_t s)
{
    return launch(qoda_scalars_kernel, 1, kThreads, 0, s, p);
}

cudaError_t launch_qoda_init(const PlanDev& p, const float* X1, float* Y, float* Xhalf, cudaStream_t s)
{
    const int64_t n4 = p.padded_elems / 4;
    const unsigned blocks = (unsigned)((n4 + 255) / 256 < kSms * 8 ? (n4 + 255) / 256 + 1 : kSms * 8);
    qoda_init_kernel<<<blocks, 256, 0, s>>>(p, X1, Y, Xhalf);
    return cudaGetLastError();
}

}  // namespace lq
