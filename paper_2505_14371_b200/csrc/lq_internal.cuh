// Internal declarations shared by the .cu files of liblq (not part of the public ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "lq.h"
#include "lq_small_rule.h"

namespace lq {

constexpr int kSms = 148;             // of a B200: what grids and waves are counted in
constexpr int kBlockCoords = 1024;    // coordinates per message block (32 lanes x 32 positions)
constexpr int kTileBlocks = 128;      // most blocks per tile (the encoder's unit: its per-CTA tables are amortised over a
                                      // tile); a plan takes the largest power of two that still gives several waves of
                                      // CTAs, down to 8 (one block per warp) when even a single wave is not reached
constexpr int kSubBlocks = 32;        // most blocks per sub-tile (the unit of the norm kernel and the symbol counts), and
                                      // of the decoder's CTAs; fewer in plans that would leave SMs idle
constexpr int kWarps = 8;
constexpr int kThreads = 256;
constexpr int kDecWarps = 4;          // of the decoder's CTAs
constexpr int kDecThreads = kDecWarps * 32;
constexpr int kLevelStride = 256;     // floats per layer in a level table
constexpr int kMaxLevels = 256;
constexpr int kCodeMaxLen = 12;       // longest code word of the entropy stage (LQ_CODE_MAX_LEN)
constexpr int kLutEntries = 2048;     // u32 entries per layer in the encoder's search table: one per value of the
                                      // top 13 bits of a non-negative float (16 bins per octave); 2033 are reachable

struct LayerDesc {
    int64_t elem_off;     // first element of the layer inside a worker's fp32 row
    int64_t word_off;     // first word of the layer inside a worker's message
    int64_t size;         // d_m
    int32_t bits;         // b_m
    int32_t nlevels;      // 2^b_m
    int32_t nblocks;      // ceil(d_m / 1024)
    int32_t first_tile;   // tiles of one layer are contiguous in the tile table
    int32_t ntiles;
    int32_t pad_;
    int64_t block_off;    // first block of the layer in a worker's row of the zero-row masks
};

struct Tile {
    int32_t layer;
    int32_t block0;       // first block of the tile inside its layer
    int32_t nblocks;      // 1..kTileBlocks
    int32_t pad_;
};

// What an encoder CTA needs to know about its tile, one record per CTA in launch order (read with one round trip
// instead of the chain launch order -> tile -> layer).
struct TileJob {
    int32_t tile;         // index in the tile table (the per-tile partials are kept by it)
    int32_t layer;
    int32_t block0;       // first block of the tile inside its layer
    int32_t nblocks;      // 1..kTileBlocks
    int32_t bits;         // b_m
    int32_t pad_;
    int64_t size;         // d_m
    int64_t elem_off;     // first coordinate of the layer inside a worker's row of `grads`
    int64_t word_off;     // first word of the layer inside a worker's message
    int64_t block_off;    // first block of the layer in a worker's row of the zero-row masks
    int64_t pad2_;
};
static_assert(sizeof(TileJob) == 64, "TileJob is read as four 16-byte words");

struct QodaScalars {
    double S;             // running sum of Eq. (general_stepsize)
    double last_delta;    // the term added by the last qoda_step
    long long t;          // index of the next iteration
    float eta;            // eta_t (= gamma_t under Eq. general_stepsize)
    float gamma;          // gamma_t (differs from eta_t only under Eq. Alt)
    double lambda;        // Eq. (Alt): running sum of ||gbar||^2
    double mu;            // Eq. (Alt): running sum of ||X_s - X_{s+1}||^2
    float eta_cur;        // Eq. (Alt): the eta that produced the current X_t (needed to recompute X_t from Y_t)
    float pad_;
};

// Device-side view of a plan, passed to kernels by value.
struct PlanDev {
    const LayerDesc* layers;
    const Tile* tiles;
    const TileJob* jobs;         // the encoder's tiles in the order in which its CTAs take them: all layers advance
                                 // together, so that layers of different character (dense, mostly zero rows) share the
                                 // SMs at any time
    int32_t num_layers;
    int32_t num_tiles;
    int32_t num_workers;
    int32_t q;            // 0 = infinity norm
    int32_t sub_tiles;    // sub-tiles per tile: the plan's tile size / sub_blocks, a power of two
    int32_t sub_shift;    // log2(sub_tiles)
    int32_t sub_blocks;   // blocks per sub-tile
    int16_t small_ranks;  // CTAs a (layer, worker) in the kernel of small plans, 0: the general path (small_plan_ranks) ...
    int16_t small_share;  // ... and the most blocks that one of them has
    int32_t most_bits;    // widest code of the plan
    int32_t least_bits;   // narrowest code of the plan
    int32_t dec_blocks;   // blocks per decoder CTA; 1: its warps share them
    int32_t dec_shift;    // log2(plan's tile size / dec_blocks)
    int32_t global_norm;  // 1: one norm per worker over all layers (Section 3.1), 0: one per layer
    int32_t bucket_norm;  // 1: one norm per bucket of 128 consecutive coordinates of a layer (Section 7.1)
    int32_t worker0;      // the encode-side kernels cover workers worker0 .. worker0 + worker_count - 1 (grid.y =
    int32_t worker_count; // worker_count); `grads` holds only those rows, every other buffer all K rows
    int64_t padded_elems; // D_pad
    int64_t packed_words; // W
    uint32_t seed_lo, seed_hi;
    uint32_t rk0[8], rk1[8];  // Philox keys of rounds 2..9 (seed words plus multiples of the Weyl constants): kernels
                              // read them straight from the parameter bank
    double* norm_partial; // [K][num_tiles * sub_tiles]
    double* stat_partial; // [K][num_tiles]
    double* sq_diff;      // [K][L]
    float* rnorm;         // [K][L]   1/N, or 0 for a zeroed layer
    uint32_t* status;     // [K][L]
    double* layer_total;  // [K][L]  per-layer sums (or maxima) before the root, for the global norm
    double* alt_partial;  // [2][num_tiles << dec_shift]  per-CTA terms of lambda and mu (Eq. Alt)
    uint8_t* row_mask;    // [K][total_blocks]  bit j of a block's byte: row j (128 values) holds a nonzero value
    const uint8_t* row_mask_prev;   // the same for the input behind the previous message, or NULL when unknown
    int64_t total_blocks; // blocks of 1024 values per worker, all layers
    double* energy_partial;   // [K][num_tiles]  bucket scope: per-tile sums of squared bucket norms
    uint32_t* flag_partial;   // [K][num_tiles]  bucket scope: bit 0 a non-finite bucket, bit 1 a nonzero bucket
    float* layer_weight;      // [K][L]          bucket scope: sqrt of a layer's summed squared bucket norms
    QodaScalars* scalars;     // [2]  the live values, and their copy as the last lq_quantize_pack found them: a decoder
                              // whose CTAs each form the step's rates reads the copy while one of them writes the first
};

// Stores a printf-style reason for lq_last_error() (calling thread) and returns `code`.
int lq_set_error(int code, const char* fmt, ...);

// Whether the decoder's CTAs form the step's rates themselves from sq_diff (Eq. general_stepsize) instead of a kernel of
// its own, which with the gap before it takes 2 to 4 us: two sums per thread, four where the CTAs fit at once (4 per SM).
// The step with 8 workers, by the decoder and by the kernel: 32 small layers 48.9 and 50.4 us, 64 of them 67.6 and 68.8; but 64
// layers of 245 blocks 373 and 370, 128 small ones 119.6 and 117.7.
inline bool rates_in_decoder(const PlanDev& p)
{
    const int64_t sums = (int64_t)p.num_workers * p.num_layers, ctas = (int64_t)p.num_tiles << p.dec_shift;
    return p.num_tiles > 0 && (sums <= 2 * kDecThreads || (sums <= 4 * kDecThreads && ctas <= 4 * kSms));
}

// Launches `kernel` so that it may start while the kernel before it on the stream is still finishing (programmatic
// dependent launch).  Every kernel of the library waits for its predecessor's memory (pdl_wait) before it touches anything
// a kernel may have written, so only the launch itself and the reading of the plan's constant tables overlap: an
// iteration of a small plan is a chain of kernels of a few us each, and what lies between two of them shrinks from 1.7 us
// to well below 1 us.  Grids of many waves are launched the plain way: with the attribute every CTA starts about 3 us
// late, not just the first ones (norm pass of 37 000 CTAs 690 -> 850 us, decoder of 4 700 CTAs 451 -> 486 us).  The line: up to 24 CTAs per
// SM no case got slower (with 8: WGAN step 174 -> 170 us, in bucket scope 175 -> 167, low-rank factors 336 -> 328).
constexpr int64_t kDependentCtas = kSms * 24;
// `cluster`: CTAs per cluster along x.  A launch that fails leaves no error behind for the next call to find.
template <typename... Params, typename... Args>
cudaError_t launch_as(bool dependent, void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, unsigned cluster, cudaStream_t s,
                      Args... args)
{
    cudaLaunchAttribute at[2];
    unsigned n = 0;
    if (dependent) {
        at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        at[n].id = cudaLaunchAttributeClusterDimension;
        at[n].val.clusterDim.x = cluster; at[n].val.clusterDim.y = 1; at[n++].val.clusterDim.z = 1;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s;
    cfg.attrs = at; cfg.numAttrs = n;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
    if (e != cudaSuccess) cudaGetLastError();
    return e;
}
template <typename... Params, typename... Args>
cudaError_t launch_cluster(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, unsigned cluster, cudaStream_t s,
                           Args... args)
{
    return launch_as((int64_t)grid.x * grid.y * grid.z <= kDependentCtas, kernel, grid, block, smem, cluster, s, args...);
}
template <typename... Params, typename... Args>
cudaError_t launch(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args... args)
{
    return launch_cluster(kernel, grid, block, smem, 1, s, args...);
}

// More than 48 KB of dynamic shared memory: every kernel opts in once per device (`configured`: bit d = device d is done).
template <typename... Kernels>
cudaError_t opt_in_shared_memory(std::atomic<uint64_t>& configured, int bytes, Kernels... kernels)
{
    int dev = 0;
    cudaGetDevice(&dev);
    const bool known = dev >= 0 && dev < 64;
    if (known && ((configured.load(std::memory_order_relaxed) >> dev) & 1u)) return cudaSuccess;
    cudaError_t e = cudaSuccess;
    ((e = e == cudaSuccess ? cudaFuncSetAttribute(kernels, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) : e), ...);
    if (e == cudaSuccess && known) configured.fetch_or(1ull << dev, std::memory_order_relaxed);
    return e;
}

// Clusters of up to 16 CTAs: likewise.
template <typename... Kernels>
cudaError_t allow_clusters(std::atomic<uint64_t>& configured, Kernels... kernels)
{
    int dev = 0;
    cudaGetDevice(&dev);
    const bool known = dev >= 0 && dev < 64;
    if (known && ((configured.load(std::memory_order_relaxed) >> dev) & 1u)) return cudaSuccess;
    cudaError_t e = cudaSuccess;
    ((e = e == cudaSuccess ? cudaFuncSetAttribute(kernels, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) : e), ...);
    if (e == cudaSuccess && known) configured.fetch_or(1ull << dev, std::memory_order_relaxed);
    return e;
}

// ---- launchers (each enqueues on `s` and returns the launch status) ----
// `write_mask`: also record the zero-row masks of `grads` in p.row_mask
cudaError_t launch_norm_partial(const PlanDev& p, const float* grads, bool write_mask, cudaStream_t s);
cudaError_t launch_norm_finalize(const PlanDev& p, float* norms, cudaStream_t s);
// Encode-side tables derived from one level table (rebuilt whenever the levels change).
struct SearchTables {
    uint32_t* lut;     // [L][kLutEntries] per bin: what added to a value's pattern gives tau << 19 (build_search_kernel)
    float2* ld;        // [L][kMaxLevels]  {l_tau, l_{tau+1} - l_tau}
    int2* how;         // [L]              which search a layer takes and its parameters
};
// how.x & 3:
//   kSearchOctave  bins of 1/16 octave over the whole fp32 range, at most one level in each
//   kSearchWindow  bins of 2^s patterns, s = how.x >> 2, from the pattern how.y on (bin 0: everything below, too), at most one
//                  level in each: level sets too dense for 16 bins per octave whose range from the first level to 1 fits
//                  2048 bins that are fine enough (uniform 8-bit levels)
//   kSearchStep    byte table over the top 15 bits in lut's place, and at most how.x >> 2 levels per bin: the rest
constexpr int kSearchOctave = 1, kSearchStep = 2, kSearchWindow = 3;
constexpr int kWindowBits = 5;      // narrowest codes with a window search: fewer levels are hardly ever that dense, and every search
                                    // more in a kernel costs the others registers
cudaError_t launch_build_search(const PlanDev& p, const float* levels, float* kept, SearchTables t, cudaStream_t s);
cudaError_t launch_quantize(const PlanDev& p, const float* grads, uint32_t step, uint32_t* packed,
                            const float* norms, uint32_t* hist, const uint32_t* prev_packed,
                            const float* prev_norms, const float* levels_cur,
                            const float* levels_prev, SearchTables t, bool need_stat, cudaStream_t s);
// layer scope, plans whose layers are all small: norms, messages and statistic in one kernel
inline bool use_small(const PlanDev& p) { return p.small_ranks > 0 && !p.global_norm && !p.bucket_norm; }
ClusterRoom small_cluster_room();      // of the current device
cudaError_t launch_layer_norms_small(const PlanDev& p, const float* grads, float* norms, cudaStream_t s);
cudaError_t launch_quantize_small(const PlanDev& p, const float* grads, uint32_t step, uint32_t* packed, float* norms,
                                  uint32_t* hist, const uint32_t* prev_packed, const float* prev_norms,
                                  const float* levels_cur, const float* levels_prev, SearchTables t, bool need_stat, cudaStream_t s);
// bucket scope: `bucket_norms` [K][8 * total_blocks] is written, `prev_norms` has the same shape
cudaError_t launch_quantize_bucketed(const PlanDev& p, const float* grads, uint32_t step, uint32_t* packed,
                                     float* bucket_norms, uint32_t* hist, const uint32_t* prev_packed,
                                     const float* prev_norms, const float* levels_cur,
                                     const float* levels_prev, SearchTables t, cudaStream_t s);
cudaError_t launch_bucket_finalize(const PlanDev& p, cudaStream_t s);
cudaError_t launch_stat_finalize(const PlanDev& p, cudaStream_t s);
// mode 0: decode + aggregate only; 1: + QODA update, Eq. (general_stepsize); 2: + QODA update, Eq. (Alt)
// masks: the zero-row masks of exactly this message's input, [K][total_blocks] with K <= 32 (a worker's all-zero
// blocks are then not read), or nullptr
cudaError_t launch_decode(const PlanDev& p, const uint32_t* packed, const float* norms,
                          const float* levels, const float* X1, float* Y, float* Xhalf, float* X,
                          float* gbar, int mode, const uint8_t* masks, cudaStream_t s);
cudaError_t launch_level_probabilities(const PlanDev& p, const uint32_t* hist, const float* norms, int num_samples,
                                       const float* levels, double* probs, cudaStream_t s);
cudaError_t launch_symbol_counts(const PlanDev& p, const uint32_t* packed, uint32_t* counts, cudaStream_t s);
cudaError_t launch_alt_scalars(const PlanDev& p, double qhat, cudaStream_t s);
cudaError_t launch_alt_finalize(const PlanDev& p, cudaStream_t s);
cudaError_t launch_qoda_scalars(const PlanDev& p, cudaStream_t s);
cudaError_t launch_average(const PlanDev& p, const float* Xhalf, double* xsum, cudaStream_t s);
cudaError_t launch_qoda_init(const PlanDev& p, const float* X1, float* Y, float* Xhalf,
                             cudaStream_t s);
cudaError_t launch_fit(const PlanDev& p, const uint32_t* hist, const float* norms, int num_samples,
                       float* levels_stage, cudaStream_t s);
cudaError_t launch_fit_shared(const PlanDev& p, const uint32_t* hist, const float* norms, int num_samples,
                              float* levels_stage, const int32_t* member_off, const int32_t* member_layer,
                              int num_types, cudaStream_t s);

// ---- device helpers ----
#ifdef __CUDACC__

// First statements of every kernel: the next kernel of the stream may be launched from now on (its CTAs take slots as
// this kernel's last ones leave them), and nothing written by the kernels before this one is read until they are done.
__device__ __forceinline__ void pdl_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// What a kernel that may overlap its predecessor reads after pdl_wait, and an earlier kernel of the stream may have written,
// must neither be read early nor through the read-only path, which takes memory as constant while the kernel runs: the
// compiler moves such loads (__ldg, const __restrict__ parameters, and the load intrinsics, which it takes for pure functions
// of the address) above the wait.  So: ordinary loads, the volatile ones below, or intrinsics on a pointer from fresh().
// All go to L2.
template <typename T>
__device__ __forceinline__ T* fresh(T* p) { asm volatile("" : "+l"(p) :: "memory"); return p; }
__device__ __forceinline__ float load_f32(const float* p)
{
    float v;
    asm volatile("ld.global.cg.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ float2 load_f32x2(const float2* p)
{
    float2 v;
    asm volatile("ld.global.cg.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t load_u8(const uint8_t* p)
{
    uint32_t v;
    asm volatile("ld.global.cg.u8 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int2 load_i32x2(const int2* p)
{
    int2 v;
    asm volatile("ld.global.cg.v2.s32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint4 load_u32x4(const uint4* p)
{
    uint4 v;
    asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}

// Philox4x32-10 (Salmon et al., SC'11): 10 rounds of two 32x32->64 multiplies and xors,
// the key bumped by the Weyl constants between rounds.
__device__ __forceinline__ void philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                              uint32_t k0, uint32_t k1, uint32_t (&out)[4])
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t p0 = (uint64_t)0xD2511F53u * c0;
        const uint64_t p1 = (uint64_t)0xCD9E8D57u * c2;
        const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c1 ^ k0;
        const uint32_t n2 = (uint32_t)(p0 >> 32) ^ c3 ^ k1;
        c1 = (uint32_t)p1;
        c3 = (uint32_t)p0;
        c0 = n0;
        c2 = n2;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    out[0] = c0; out[1] = c1; out[2] = c2; out[3] = c3;
}

// ---- shared-memory loads by absolute 32-bit address (volatile pins their place after the barrier or wait that
// ---- precedes them)
__device__ __forceinline__ uint32_t lds_u32(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ uint32_t lds_u8(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ float lds_f32(uint32_t a)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
    return v;
}
template <int kOff>
__device__ __forceinline__ float lds_f32_at(uint32_t a)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1+%2];" : "=f"(v) : "r"(a), "n"(kOff));
    return v;
}
__device__ __forceinline__ float2 lds_f32x2(uint32_t a)
{
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
    return v;
}

__device__ __forceinline__ float4 lds_f32x4(uint32_t a)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
    return v;
}

// a0 += b0 and a1 += b1, each rounded as a plain addition, in one instruction
__device__ __forceinline__ void add_f32x2(float& a0, float& a1, float b0, float b1)
{
    asm("{\n\t.reg .b64 a, b;\n\tmov.b64 a, {%0, %1};\n\tmov.b64 b, {%2, %3};\n\tadd.rn.f32x2 a, a, b;\n\tmov.b64 {%0, %1}, a;\n\t}"
        : "+f"(a0), "+f"(a1) : "f"(b0), "f"(b1));
}

// 16-byte asynchronous copies global -> shared (completion by commit / wait groups of the issuing thread)
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, int bytes)
{
    // copies `bytes` (0..16) bytes and fills the rest of the 16 with zeros
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const void* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ double warp_max(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Sum over the CTA in a fixed order (xor tree inside a warp, warps added in index order).
// The result is valid in thread 0.  `scratch` holds one double per warp.
template <bool kMax>
__device__ __forceinline__ double block_reduce(double v, double* scratch)
{
    v = kMax ? warp_max(v) : warp_sum(v);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) scratch[warp] = v;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        r = scratch[0];
        for (int w = 1; w < nw; ++w) r = kMax ? fmax(r, scratch[w]) : r + scratch[w];
    }
    return r;
}

// One value's term of a layer's L^q norm (Section 2.2), accumulated in fp64 (the maximum as an integer pattern).
// mode 0: max |v|   1: sum |v|   2: sum v^2   3: sum |v|^q (integer q >= 3)
template <int kMode>
__device__ __forceinline__ void accumulate(double& acc, uint32_t& maxbits, float v, int q)
{
    if (kMode == 0) {
        // |v| as an unsigned integer orders like the float; NaN and Inf have the largest patterns
        const uint32_t b = __float_as_uint(v) & 0x7fffffffu;
        maxbits = max(maxbits, b);
    } else if (kMode == 1) {
        acc += (double)fabsf(v);
    } else if (kMode == 2) {
        const double a = (double)v;
        acc = fma(a, a, acc);            // the product of two floats is exact in fp64
    } else {
        const double a = fabs((double)v);
        double p = a;
        for (int r = 1; r < q; ++r) p = __dmul_rn(p, a);
        acc += p;
    }
}

// This lane's four values of row j of block blk (fresh() pointer), zeros behind the layer's end.
__device__ __forceinline__ float4 row_values(const float* g, int64_t blk, int j, int64_t size, int lane)
{
    const int64_t pos = blk * kBlockCoords + 128 * j + 4 * lane;
    if (pos + 4 <= size) return __ldcg(reinterpret_cast<const float4*>(g + pos));
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (pos < size) v.x = __ldcg(g + pos);
    if (pos + 1 < size) v.y = __ldcg(g + pos + 1);
    if (pos + 2 < size) v.z = __ldcg(g + pos + 2);
    return v;
}

// One block of 1024 values of a fresh() pointer (a lane takes the float4 at 128 j + 4 lane of row j): adds its terms to the lane's
// accumulators and returns, in every lane, the byte whose bit j says whether row j holds anything but zeros.  A partial block's rows are
// loaded like a whole one's, all at once: value by value its loads were a chain of 8 waits, and the second copy of the sums
// cost the whole blocks registers (norm pass of the Transformer-XL shapes 688 -> 666 us; step of 1 365 blocks in 40 layers
// 53.9 -> 50.9).
template <int kMode>
__device__ __forceinline__ uint32_t norm_block(const float* __restrict__ g, int64_t blk, int64_t size, int lane, int q,
                                               double& acc, uint32_t& maxbits)
{
    const int64_t blk0 = blk * kBlockCoords, base = blk0 + 4 * lane;
    float4 v[8];
    if (blk0 + kBlockCoords <= size) {
#pragma unroll
        for (int j = 0; j < 8; ++j)
            v[j] = __ldcg(reinterpret_cast<const float4*>(g + base + 128 * j));
    } else {                                 // (zeros behind the layer's end add nothing)
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = row_values(g, blk, j, size, lane);
    }
    uint32_t rows = 0;                       // bit j: this lane's part of row j holds a value that is not +-0 (NaN counts)
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        accumulate<kMode>(acc, maxbits, v[j].x, q);
        accumulate<kMode>(acc, maxbits, v[j].y, q);
        accumulate<kMode>(acc, maxbits, v[j].z, q);
        accumulate<kMode>(acc, maxbits, v[j].w, q);
        const float mag = (fabsf(v[j].x) + fabsf(v[j].y)) + (fabsf(v[j].z) + fabsf(v[j].w));
        rows |= (mag != 0.0f ? 1u : 0u) << j;
    }
    return __reduce_or_sync(0xffffffffu, rows);      // a row is live if any lane's part of it is
}

// The CTA's total of the lanes' accumulators, valid in thread 0; NaN when a value was not finite.
template <int kMode>
__device__ __forceinline__ double norm_cta_total(double acc, uint32_t maxbits, double* scratch)
{
    if (kMode == 0) {
        // fmax drops NaNs: reduce a "bad" flag next to the maximum
        const unsigned bad = __syncthreads_or(maxbits >= 0x7f800000u);
        const double r = block_reduce<true>((double)__uint_as_float(maxbits), scratch);
        return bad ? __longlong_as_double(0x7ff8000000000000LL) : r;
    }
    return block_reduce<false>(acc, scratch);
}

// A layer's norm from the norm pass's partials, in a fixed order: thread i < 128 takes partials i, i + 128, ...,
// then the CTA tree; the root, the rounding to fp32, the flags and the fp32 reciprocal.  Every thread of the CTA
// calls it (128 threads or more); the result is valid in thread 0.  `scratch`: one double per warp.
struct LayerNorm {
    double total;        // the sum (or maximum) before the root
    float norm, rnorm;   // fp32(||v||_q) and 1 / norm, both 0 when flagged
    uint32_t status;
    bool bad;            // a partial was NaN or Inf
};
__device__ __forceinline__ LayerNorm layer_norm_of_total(double total, bool bad, int q)
{
    LayerNorm r;
    r.total = total;
    r.bad = bad;
    double n64;
    if (q == 0 || q == 1) n64 = total;
    else if (q == 2)      n64 = sqrt(total);
    else                  n64 = pow(total, 1.0 / (double)q);
    float nf = (float)n64;
    r.status = 0;
    if (bad || !(fabs(n64) <= 1.7976931348623157e308) || !(fabsf(nf) <= 3.402823466e38f))
        r.status = LQ_STATUS_NONFINITE;
    else if (nf < 1.17549435e-38f)
        r.status = LQ_STATUS_ZERO_NORM;
    r.norm = r.status ? 0.0f : nf;
    r.rnorm = r.status ? 0.0f : __fdiv_rn(1.0f, nf);
    return r;
}
__device__ __forceinline__ LayerNorm layer_norm_from_partials(const double* part, int n, int q, double* scratch)
{
    double acc = 0.0;
    int bad = 0;
    if (threadIdx.x < 128)
        for (int i = threadIdx.x; i < n; i += 128) {
            const double v = __ldcg(part + i);
            if (!(fabs(v) <= 1.7976931348623157e308)) bad = 1;
            if (q == 0) acc = fmax(acc, v); else acc += v;
        }
    bad = __syncthreads_or(bad);
    const double total = q == 0 ? block_reduce<true>(acc, scratch) : block_reduce<false>(acc, scratch);
    return layer_norm_of_total(total, bad != 0, q);
}

#endif  // __CUDACC__

}  // namespace lq
