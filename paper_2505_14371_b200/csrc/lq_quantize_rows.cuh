// Blocks of a layer encoded a row of 128 coordinates a warp: all blocks of small plans (lq_quantize_small.cu), and the last, partial
// block of every layer in the general encoder (lq_quantize_tile.cuh).
#pragma once

#include "lq_quantize.cuh"

namespace lq {

// What the warps of a CTA share about their blocks.
struct RowsJob {
    const float* g;              // first coordinate of the layer in this worker's row
    const uint32_t* prev;        // the layer's words in the previous message, or NULL
    int64_t size;                // d_m
    int block0, nblocks;         // the CTA's blocks of the layer
    const uint32_t* rows;        // per block: bits 0..7 its rows that hold anything, bits 8..15 those of the previous input
    uint32_t words;              // shared-memory address of the blocks' words, zeroed
    bool counts;                 // histogram mode, and the layer is not sent as zeros
};

// Row j of all of the CTA's blocks (of a layer's partial block, too: coordinates behind the layer's end are zeros and turn into
// symbols 0), by warp j.  A row's four symbols a lane are 4 C bits of the lane's string: they are formed as the first four of a string,
// moved into place and ORed into the block's words, and so with the previous message's, so that all rows run the same code:
// fetching code that no warp has run yet is what takes longest here.  Steps of 8192 coordinates and 8 workers, and of a perceptron's
// 203 530 and 4: a warp a block, 8 rows of it unrolled, 16.7 and 26.8 us; a row a warp, code of its own for each, 13.5 and 24.8; the
// same code for all 12.0 and 20.5.  (Two blocks side by side: 0.6 us slower.)
template <int B, int kSearch, bool kHist, bool kStat>
__device__ __forceinline__ double quantize_rows(const PlanDev& p, const PhiloxConsts& pc, const RowsJob& job, const QuantEnv& ev, float4 first,
                                                int lane, int j)
{
    constexpr int C = B + 1;
    const SearchPar<kSearch> sp(ev);
    const int w0 = (4 * C * j) >> 5, shift = (4 * C * j) & 31;
    const bool two = shift + 4 * C > 32;                         // the row's bits reach into a second word
    double stat = 0.0;
    float4 next = first;
    uint32_t pnext0, pnext1;
    auto request_prev = [&](int b) {
        const uint32_t* from = job.prev + (int64_t)(job.block0 + b) * (C * 32) + lane + 32 * w0;
        pnext0 = kStat && job.prev ? __ldcg(from) : 0u;
        pnext1 = kStat && job.prev && two ? __ldcg(from + 32) : 0u;
    };
    request_prev(0);
#pragma unroll 1
    for (int b = 0; b < job.nblocks; ++b) {
        const float4 v = next;
        uint32_t pw[C], cw[C];
#pragma unroll
        for (int i = 0; i < C; ++i) { pw[i] = 0u; cw[i] = 0u; }
        pw[0] = __funnelshift_r(pnext0, pnext1, shift);
        pw[1] = pnext1 >> shift;
        if (b + 1 < job.nblocks) {
            next = row_values(job.g, job.block0 + b + 1, j, job.size, lane);
            request_prev(b + 1);
        }
        const uint32_t m = job.rows[b] >> j;
        const int64_t pos = (int64_t)(job.block0 + b) * kBlockCoords + 128 * j;          // of the row
        if (m & 1u) {
            uint32_t x[4];
            philox4x32_10_folded((uint32_t)((job.block0 + b) * 256 + 32 * j + lane), pc, p, x);
            const float vv[4] = {v.x, v.y, v.z, v.w};
            float u[4];
            normalise4(v, ev.r, u);
            uint32_t t8[4];
            step_search4<B, kHist>(ev, sp, u, t8);
            pack_first_row<C>(cw, ev.ld);
#pragma unroll
            for (int e = 0; e < 4; ++e)
                quantize_coord<B, kSearch, kHist, kStat, false>(ev, sp, vv[e], u[e], t8[e], x[e], e, cw, pw, stat, 0.f, 0.f, pos + 4 * lane + e < job.size);
            const uint32_t at = job.words + 4u * (uint32_t)(b * (C * 32) + lane + 32 * w0);
            asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(at), "r"(cw[0] << shift) : "memory");
            if (two) asm volatile("red.shared.or.b32 [%0+128], %1;" ::"r"(at), "r"(__funnelshift_l(cw[0], cw[1], shift)) : "memory");
        } else {
            if (kStat && ((m >> 8) & 1u)) {
#pragma unroll
                for (int e = 0; e < 4; ++e) stat_prev_only<C, false>(ev, pw, e, 0.f, stat);
            }
            if (kHist && job.counts && lane == 0 && pos < job.size)       // its coordinates have u = 0
                atomicAdd(ev.hist, (uint32_t)min((int64_t)128, job.size - pos));
        }
    }
    return stat;
}

template <int B, bool kHist, bool kStat>
__device__ __forceinline__ double quantize_rows_by(const PlanDev& p, const PhiloxConsts& pc, const RowsJob& job, const QuantEnv& ev, int search,
                                                   float4 first, int lane, int j)
{
    if (search == kSearchOctave) return quantize_rows<B, kSearchOctave, kHist, kStat>(p, pc, job, ev, first, lane, j);
    if constexpr (B >= kWindowBits)
        if (search == kSearchWindow) return quantize_rows<B, kSearchWindow, kHist, kStat>(p, pc, job, ev, first, lane, j);
    return quantize_rows<B, kSearchStep, kHist, kStat>(p, pc, job, ev, first, lane, j);
}

}  // namespace lq
