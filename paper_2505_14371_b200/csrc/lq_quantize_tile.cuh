// A CTA's share of one (layer, worker) in the layer and global norm scopes, with the CTA's tables in place: the blocks of
// a run of consecutive blocks of the layer, taken round-robin by the warps (lq_quantize.cu).
#pragma once

#include "lq_quantize_rows.cuh"

namespace lq {

// Everything a warp needs to walk its blocks of one (tile, worker).
struct WarpCtx {
    const float* g;              // first coordinate of the layer in this worker's row
    int64_t nfull;               // blocks below this index lie wholly inside the layer
    int lane;
};

// x of lane i, the same in every lane and known to be (a reduction's result is warp-uniform)
__device__ __forceinline__ uint32_t lane_value(uint32_t x, int i, int lane)
{
    return __reduce_or_sync(0xffffffffu, lane == i ? x : 0u);
}

// A warp's share of a tile: the whole blocks warp, warp + 8, ...  A block whose rows are all zero in this input
// and in the input behind the previous message is an all-zero piece of message that adds nothing to the
// statistic: its words are stored and nothing is read.  The other blocks are taken in order.
template <int B, int kSearch, bool kHist, bool kStat>
__device__ __forceinline__ double quantize_tile(const PlanDev& p, const PhiloxConsts& pc, const WarpCtx& c,
                                                const Tile& tile, uint32_t* __restrict__ out,
                                                const uint32_t* __restrict__ prev, const QuantEnv& ev,
                                                const uint8_t* rows_cur, const uint8_t* rows_prev, uint32_t ring_base)
{
    constexpr int C = B + 1;
    const int warp = threadIdx.x >> 5, lane = c.lane;
    double stat = 0.0;
    const int64_t nf = c.nfull - tile.block0;                 // whole blocks of this tile
    const int nfb = nf < tile.nblocks ? (int)nf : tile.nblocks;

    // lane i < 16 keeps the masks of the warp's i-th block (this input's rows in bits 0..7, the previous input's
    // in bits 8..15, bit 16: the block exists)
    uint32_t mymask = 0;
    {
        const int b = warp + kQWarps * lane;
        if (lane < kTileBlocks / kQWarps && b < nfb) mymask = (uint32_t)rows_cur[b] | ((uint32_t)rows_prev[b] << 8) | 0x10000u;
    }
    uint32_t zero = __ballot_sync(0xffffffffu, mymask == 0x10000u);
    uint32_t todo = __ballot_sync(0xffffffffu, (mymask & 0xffffu) != 0u);
    while (zero) {
        const int i = __ffs(zero) - 1;
        zero &= zero - 1;
        const int64_t blk = tile.block0 + warp + kQWarps * i;
        const int64_t woff = blk * (int64_t)C * 32 + lane;
#pragma unroll
        for (int w = 0; w < C; ++w) __stcs(out + woff + w * 32, 0u);
        if (kHist && lane == 0) atomicAdd(ev.hist, (uint32_t)kBlockCoords);     // its coordinates all have u = 0
    }
    if (todo == 0u) return stat;
    const SearchPar<kSearch> sp(ev);

    auto block_base = [&](int i) { return c.g + (tile.block0 + warp + kQWarps * i) * (int64_t)kBlockCoords; };
    int i = __ffs(todo) - 1;
    todo &= todo - 1;
    uint32_t m = lane_value(mymask, i, lane);
    const float* src = block_base(i) + 4 * lane;             // this lane's float4 of row 0
    // While a lane works on row j of a block, row j of the next block with content is already on its way into
    // the slot that row j has just left (one commit group per row slot, so waiting for all but the last 7
    // groups means the row is there).
    const uint32_t ring = ring_base + (uint32_t)(warp * 8 * 512 + lane * 16);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        if ((m >> j) & 1u) cp_async16(ring + 512u * j, src + 128 * j, 16);
        cp_async_commit();
    }
    for (;;) {
        const int64_t blk = tile.block0 + warp + kQWarps * i;
        const uint32_t rows = m & 0xffu, prows = (m >> 8) & 0xffu;
        // the next block with content: its rows follow this block's
        const int inext = todo ? __ffs(todo) - 1 : 0;
        const uint32_t mnext = todo ? lane_value(mymask, inext, lane) : 0u;
        const float* nsrc = block_base(inext) + 4 * lane;
        uint32_t pw[C];
#pragma unroll
        for (int w = 0; w < C; ++w)
            pw[w] = (kStat && prev && prows) ? __ldcg(prev + blk * (int64_t)C * 32 + lane + w * 32) : 0u;
        uint32_t cw[C];
        pack_begin<C>(cw, ev.ld);
        const uint32_t ctr0 = (uint32_t)(blk * 256) + (uint32_t)lane;     // index / 4 of this lane's row 0
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if ((rows >> j) & 1u) {
                float4 v;
                cp_async_wait<7>();
                asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                             : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(ring + 512u * j));
                if ((mnext >> j) & 1u) cp_async16(ring + 512u * j, nsrc + 128 * j, 16);
                cp_async_commit();
                uint32_t x[4];
                philox4x32_10_folded(ctr0 + 32 * j, pc, p, x);
                const float vv[4] = {v.x, v.y, v.z, v.w};
                float u[4];
                normalise4(v, ev.r, u);
                uint32_t t8[4];
                step_search4<B, kHist>(ev, sp, u, t8);
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    quantize_coord<B, kSearch, kHist, kStat, false>(ev, sp, vv[e], u[e], t8[e], x[e], 4 * j + e, cw, pw, stat, 0.f, 0.f, true);
            } else {
                if ((mnext >> j) & 1u) cp_async16(ring + 512u * j, nsrc + 128 * j, 16);
                cp_async_commit();
                pack_zero_row<C>(cw, j, ev.ld);
                if (kStat && ((prows >> j) & 1u)) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) stat_prev_only<C, false>(ev, pw, 4 * j + e, 0.f, stat);
                }
                if (kHist && lane == 0) atomicAdd(ev.hist, 128u);   // an all-zero row: its coordinates have u = 0
            }
        }
        const int64_t woff = blk * (int64_t)C * 32 + lane;
#pragma unroll
        for (int w = 0; w < C; ++w) __stcs(out + woff + w * 32, cw[w]);
        if (todo == 0u) break;
        i = inext;
        todo &= todo - 1;
        m = mnext;
    }
    cp_async_wait<0>();
    return stat;
}

// The step search out of line, which leaves the other searches of the widest code more registers: 201 M coordinates, uniform levels, step
// 736 -> 723 us (random levels, 33.5 M: encoder 89 -> 97).  Widths below gain nothing by it (7 bits, uniform 66 and 68, random 79 and 94), nor does the
// kernel of all widths (widths 2, 3, 4 and 8, 512 layers, step 2345 -> 2365).
template <int B, bool kHist, bool kStat>
__device__ __noinline__ double quantize_tile_steps(const PlanDev& p, const PhiloxConsts pc, const WarpCtx c, const Tile tile, uint32_t* out,
                                                   const uint32_t* prev, const QuantEnv ev, const uint8_t* rows_cur, const uint8_t* rows_prev,
                                                   uint32_t ring_base)
{
    return quantize_tile<B, kSearchStep, kHist, kStat>(p, pc, c, tile, out, prev, ev, rows_cur, rows_prev, ring_base);
}

// The whole blocks of a layer of width B.
template <int B, int kWidth, bool kHist, bool kStat>
__device__ __forceinline__ double quantize_width(const PlanDev& p, const PhiloxConsts& pc, const WarpCtx& c, const Tile& tile, int search,
                                                 uint32_t* __restrict__ out, const uint32_t* __restrict__ prev, const QuantEnv& ev,
                                                 const uint8_t* rows_cur, const uint8_t* rows_prev, uint32_t ring_base)
{
    if (ev.r == 0.0f) return zeroed_tile<B>(tile, c.lane, out, kStat ? prev : nullptr, ev.tprev);
    if (search == kSearchOctave)
        return quantize_tile<B, kSearchOctave, kHist, kStat>(p, pc, c, tile, out, prev, ev, rows_cur, rows_prev, ring_base);
    if constexpr (B >= kWindowBits)
        if (search == kSearchWindow)
            return quantize_tile<B, kSearchWindow, kHist, kStat>(p, pc, c, tile, out, prev, ev, rows_cur, rows_prev, ring_base);
    if constexpr (kWidth == LQ_MAX_BITS)
        return quantize_tile_steps<B, kHist, kStat>(p, pc, c, tile, out, prev, ev, rows_cur, rows_prev, ring_base);
    else
        return quantize_tile<B, kSearchStep, kHist, kStat>(p, pc, c, tile, out, prev, ev, rows_cur, rows_prev, ring_base);
}

// The CTA's whole blocks for the layer's code width (kWidth, or `bits` where kWidth is 0) and search; returns the thread's
// statistic term.
template <int kWidth, bool kHist, bool kStat>
__device__ __forceinline__ double quantize_blocks(const PlanDev& p, const PhiloxConsts& pc, const WarpCtx& c, const Tile& tile,
                                                  int bits, int search, uint32_t* __restrict__ out, const uint32_t* __restrict__ prev,
                                                  const QuantEnv& ev, const uint8_t* rows_cur, const uint8_t* rows_prev,
                                                  uint32_t ring_base)
{
    double stat = 0.0;
    if constexpr (kWidth != 0) {
        stat = quantize_width<kWidth, kWidth, kHist, kStat>(p, pc, c, tile, search, out, prev, ev, rows_cur, rows_prev, ring_base);
    } else {
        switch (bits) {
#define LQ_CASE(BB) case BB: stat = quantize_width<BB, 0, kHist, kStat>(p, pc, c, tile, search, out, prev, ev, rows_cur, rows_prev, ring_base); break;
            LQ_CASE(1) LQ_CASE(2) LQ_CASE(3) LQ_CASE(4) LQ_CASE(5) LQ_CASE(6) LQ_CASE(7) LQ_CASE(8)
#undef LQ_CASE
            default: break;
        }
    }
    return kStat ? stat : 0.0;
}

}  // namespace lq
