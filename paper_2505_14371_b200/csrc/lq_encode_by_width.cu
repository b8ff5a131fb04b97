// The entropy encoder of plans whose layers' code widths take turns: tiles in the order of their widths, so that the CTAs that run at a
// time run the same code, in three launches: the words of every tile, the places, the blocks.  In stream order, with one launch
// (lq_coding.cu), what bounds such plans is the fetching of both walks' code for all widths.
// The rule (entropy_by_width, lq_coding.cuh) follows from the plan's tiles.
#include <algorithm>

#include "lq_encode.cuh"

namespace lq {
namespace {

// The words of all tiles up to the end of every tile, from those of every tile: one CTA per worker.
__global__ void __launch_bounds__(1024) entropy_place_kernel(PlanDev p, uint64_t* __restrict__ states)
{
    constexpr int kEach = 8;
    __shared__ uint32_t part[32];
    uint64_t* state = states + (int64_t)blockIdx.x * p.num_tiles;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t before = 0;
    for (int t0 = 0; t0 < p.num_tiles; t0 += 1024 * kEach) {
        const int first = t0 + threadIdx.x * kEach;
        uint32_t v[kEach], sum = 0;
#pragma unroll
        for (int i = 0; i < kEach; ++i) { v[i] = first + i < p.num_tiles ? (uint32_t)state[first + i] : 0u; sum += v[i]; }
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += x;
        }
        __syncthreads();
        if (lane == 31) part[warp] = incl;
        __syncthreads();
        uint32_t w = part[lane], wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += x;
        }
        uint32_t at = before + __shfl_sync(0xffffffffu, wi - w, warp) + incl - sum;
        before += __shfl_sync(0xffffffffu, wi, 31);
#pragma unroll
        for (int i = 0; i < kEach; ++i) {
            at += v[i];
            if (first + i < p.num_tiles) state[first + i] = kTileEnd | at;
        }
    }
}

}  // namespace

cudaError_t launch_entropy_encode_by_width(const PlanDev& p, const uint32_t* packed, const uint32_t* enc_tables, uint32_t* offsets, uint32_t* out,
                                           int64_t capacity, uint16_t* run_offsets, EncodeScratch scratch, uint32_t* bad, cudaStream_t s)
{
    const uint32_t code_bytes = code_table_bytes(p);
    static std::atomic<uint64_t> configured{0};
    const cudaError_t e = opt_in_shared_memory(configured, kEncodeSmem, entropy_encode_kernel<kSizes>, entropy_encode_kernel<kPlaced>);
    if (e != cudaSuccess) return e;
    const unsigned grid = (unsigned)((int64_t)p.num_tiles * p.num_workers);
    uint64_t* states = scratch.states + 1;
    entropy_encode_kernel<kSizes><<<grid, kThreads, code_bytes, s>>>(p, packed, enc_tables, offsets, out, capacity, run_offsets, scratch.sized, states,
                                                                     nullptr, kMostLooks, bad, code_bytes);
    entropy_place_kernel<<<(unsigned)p.num_workers, 1024, 0, s>>>(p, states);
    entropy_encode_kernel<kPlaced><<<grid, kThreads, code_bytes + kCodeBufBytes, s>>>(p, packed, enc_tables, offsets, out, capacity, run_offsets,
                                                                                      scratch.sized, states, nullptr, kMostLooks, bad, code_bytes);
    return cudaGetLastError();
}

}  // namespace lq
