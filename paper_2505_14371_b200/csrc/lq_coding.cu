// Entropy stage on top of the fixed-width message (appendix on the coding framework: with the level
// frequencies known or estimated, a Huffman code on the level symbols; one sign bit per non-zero entry).
//
// A layer's code is a set of word lengths (1..12 bits) for its 2^b level indices; the words are the
// canonical ones (symbols ordered by length, then index; first word all zeros, each next word the
// previous plus one, shifted left when the length grows), written most significant bit first.
//
// Stream format of one worker: the blocks of 1024 coordinates of the fixed-width layout, layer after
// layer, each block starting on a 32-bit word.  Inside a block the coordinates come in the order
// s = 32 * lane + p (lane = 0..31, p = 0..31), i.e. coordinate 128 * (p / 4) + 4 * lane + p % 4 of the block;
// padding coordinates past the layer's end are left out.  Each coordinate contributes its level's word and,
// when the level index is not 0, its sign bit.  Stream bit t of a block is bit t % 32 of its word t / 32.
// block_offsets[k][i] is the first word of block i in worker k's stream, block_offsets[k][blocks] its length.
#include <algorithm>
#include <vector>

#include "lq_encode.cuh"

namespace lq {

// ---- host: Huffman lengths and canonical tables ------------------------------------------------

// Lengths of a Huffman code for n symbols (two-queue construction on the sorted weights), every symbol
// with a word; weights below a floor are raised to it, and the floor doubles until no word is longer
// than max_len.
bool huffman_lengths_host(const double* w, int n, int max_len, uint8_t* len)
{
    if (n == 1) { len[0] = 1; return true; }
    double total = 0.0;
    for (int i = 0; i < n; ++i) { if (!(w[i] >= 0.0)) return false; total += w[i]; }
    if (!(total > 0.0)) total = 1.0;
    double floor_w = total * 9.094947017729282e-13;            // 2^-40 of the total
    std::vector<int> order(n), parent(2 * n), depth(2 * n);
    std::vector<double> wt(2 * n);
    for (;;) {
        for (int i = 0; i < n; ++i) { wt[i] = std::max(w[i], floor_w); order[i] = i; }
        std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return wt[a] < wt[b]; });
        // leaves are taken from `order`, merged trees from a second queue that is born sorted
        int leaf = 0, tree = n, made = n;
        auto take = [&]() {
            if (leaf < n && (tree >= made || wt[order[leaf]] <= wt[tree])) return order[leaf++];
            return tree++;
        };
        for (int m = 0; m < n - 1; ++m) {
            const int a = take(), b = take();
            wt[made] = wt[a] + wt[b];
            parent[a] = made; parent[b] = made;
            ++made;
        }
        parent[made - 1] = -1;
        depth[made - 1] = 0;
        for (int v = made - 2; v >= 0; --v) depth[v] = depth[parent[v]] + 1;
        int longest = 0;
        for (int i = 0; i < n; ++i) { len[i] = (uint8_t)depth[i]; longest = std::max(longest, depth[i]); }
        if (longest <= max_len) return true;
        floor_w *= 2.0;
    }
}

// Canonical words of the lengths; returns false unless the lengths describe a prefix code (Kraft sum <= 1).
bool canonical_codes_host(const uint8_t* len, int n, int max_len, uint32_t* code)
{
    uint64_t kraft = 0;                                        // in units of 2^-max_len
    for (int i = 0; i < n; ++i) {
        if (len[i] < 1 || len[i] > max_len) return false;
        kraft += (uint64_t)1 << (max_len - len[i]);
    }
    if (kraft > ((uint64_t)1 << max_len)) return false;
    uint32_t next = 0; int prev = 0;
    for (int l = 1; l <= max_len; ++l)
        for (int i = 0; i < n; ++i)
            if (len[i] == l) { next <<= (l - prev); code[i] = next; next += 1; prev = l; }
    return true;
}

static uint32_t reverse_bits(uint32_t v, int l)
{
    uint32_t r = 0;
    for (int j = 0; j < l; ++j) r |= ((v >> j) & 1u) << (l - 1 - j);
    return r;
}

// enc[level] = word with its first bit in bit 0 | length << 16 (the decode table is made from these on the device).
void build_code_table_host(const uint8_t* len, const uint32_t* code, int n, uint32_t* enc)
{
    for (int i = 0; i < kMaxLevels; ++i) enc[i] = i < n ? reverse_bits(code[i], len[i]) | ((uint32_t)len[i] << 16) : 0u;
}

// ---- device ------------------------------------------------------------------------------------
namespace {

// The decode tables (lq_coding.cuh) of layers layer0, layer0 + 1, ... from their encode entries, a CTA per layer.  A code may
// be renewed as often as the levels: on the host the 8192 entries and their pairs took 21 us a layer.
__global__ void __launch_bounds__(1024) build_decode_tables_kernel(PlanDev p, int layer0, const uint32_t* enc_tables, uint16_t* dec_tables)
{
    __shared__ uint16_t one[kDecEntries];                       // a single coordinate per entry
    const int layer = layer0 + blockIdx.x, n = p.layers[layer].nlevels, C = p.layers[layer].bits + 1;
    const uint32_t* enc = enc_tables + (int64_t)layer * kMaxLevels;
    uint16_t* dec = dec_tables + (int64_t)layer * kDecEntries;
    for (int i = threadIdx.x; i < kDecEntries; i += blockDim.x) one[i] = (uint16_t)(kDecInvalid | (1u << kDecLenShift));
    __syncthreads();
    for (int s = threadIdx.x >> 5; s < n; s += (int)(blockDim.x >> 5)) {
        const uint32_t e = enc[s], rev = e & 0xffffu, l = e >> 16;
        for (uint32_t hi = threadIdx.x & 31; hi < 1u << (kDecBits - l); hi += 32) {
            const uint32_t sign = s != 0 ? (hi & 1u) : 0u;             // the bit right after the word
            one[rev | (hi << l)] = (uint16_t)((2u * (uint32_t)s + sign) | ((l + (s != 0 ? 1u : 0u)) << kDecLenShift));
        }
    }
    __syncthreads();
    for (uint32_t w = threadIdx.x; w < (uint32_t)kDecEntries; w += blockDim.x) {
        const uint32_t e = one[w], l = e >> kDecLenShift;
        uint32_t out = e;
        if (C <= kDecPairBits) {
            const uint32_t e1 = one[w >> l], l1 = e1 >> kDecLenShift;  // what follows a window's first coordinate
            if (e & kDecInvalid) out = kDecPairInvalid | kDecSingle | (1u << kDecLenShift);
            else if (!(e1 & kDecInvalid) && l + l1 <= (uint32_t)kDecBits) out = (e & 0x1ffu) | ((e1 & 0x1ffu) << C) | ((l + l1) << kDecLenShift);
            else out = (e & 0x1ffu) | (l << kDecLenShift) | kDecSingle;
        }
        dec[w] = (uint16_t)out;
    }
}

// One coordinate from the next 13 stream bits: its symbol, the bits it takes and whether no word matched.
struct OneCoord { uint32_t sym, bits; bool invalid; };
__device__ __forceinline__ OneCoord decode_one(uint32_t e, int C, const uint32_t* enc)
{
    if (C > kDecPairBits) return OneCoord{e & 0x1ffu, e >> kDecLenShift, (e & kDecInvalid) != 0u};
    OneCoord r{e & ((1u << C) - 1u), e >> kDecLenShift, (e & kDecPairInvalid) != 0u};
    if (!(e & kDecSingle)) r.bits = (enc[r.sym >> 1] >> 16) + (r.sym > 1u ? 1u : 0u);      // the first one's share of the pair's
    return r;
}

// One thread per (block, worker): walks the block's stream and rebuilds the fixed-width words, two coordinates per look-up
// where the table holds pairs.  Its chain of dependent look-ups bounds it: 300 000 coordinates at 4 bits, 4 workers, 344 us
// one by one, 416 with a second look-up (the first one's share of a pair's bits) for each, 203 by pairs.
__global__ void __launch_bounds__(128) entropy_decode_kernel(PlanDev p, const uint32_t* __restrict__ in, int64_t capacity,
                                                             const uint32_t* __restrict__ offsets,
                                                             const uint32_t* __restrict__ enc_tables,
                                                             const uint16_t* __restrict__ dec_tables,
                                                             uint32_t* __restrict__ packed, uint32_t* __restrict__ bad)
{
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int k = blockIdx.y;
    if (g >= p.total_blocks) return;
    // the layer that owns global block g (layers are few: a linear search over their block ranges)
    int layer = 0;
    while (layer + 1 < p.num_layers && p.layers[layer + 1].block_off <= g) ++layer;
    while (p.layers[layer].nblocks == 0 && layer + 1 < p.num_layers) ++layer;
    const LayerDesc L = p.layers[layer];
    const int64_t blk = g - L.block_off;
    const int C = L.bits + 1;
    const uint16_t* dec = dec_tables + (int64_t)layer * kDecEntries;
    const uint32_t* enc = enc_tables + (int64_t)layer * kMaxLevels;
    const uint32_t* off_k = offsets + (int64_t)k * (p.total_blocks + 1);
    const int64_t first = off_k[g], last = min((int64_t)off_k[g + 1], capacity);
    const uint32_t* src = in + (int64_t)k * capacity;
    uint32_t* dst = packed + (int64_t)k * p.packed_words + L.word_off + blk * (int64_t)C * 32;
    const int rest = (int)min((int64_t)kBlockCoords, L.size - blk * kBlockCoords);
    int64_t wi = first;                                       // next word to load
    uint64_t window = 0; int have = 0;                        // `have` valid bits in the low end of `window`
    bool broken = false;
    uint32_t pos = 0, last_at = 0, last_pair = 0;             // bits taken; where the last look-up was made; its entry if a pair's
    for (int lane = 0; lane < 32; ++lane) {
        uint32_t cw[LQ_MAX_BITS + 2];
        for (int i = 0; i <= C; ++i) cw[i] = 0u;
        const int real = real_positions(rest, lane);
        for (int pp = 0; pp < real; pp += 2) {
            while (have <= 32) { const uint32_t x = wi < last ? src[wi] : 0u; ++wi; window |= (uint64_t)x << have; have += 32; }
            const uint32_t e = dec[window & (uint32_t)(kDecEntries - 1)];
            uint32_t two, bits;                               // the symbols of coordinates pp and pp + 1 (a pattern without a word: 0)
            last_at = pos; last_pair = 0;
            if (C <= kDecPairBits && pp + 1 < real && !(e & kDecSingle)) {
                two = e & ((1u << (2 * C)) - 1u);
                bits = e >> kDecLenShift;
                last_pair = e;
            } else {
                const OneCoord c = decode_one(e, C, enc);
                two = c.sym; bits = c.bits;
                broken |= c.invalid;
                if (pp + 1 < real) {
                    const OneCoord c1 = decode_one(dec[(window >> bits) & (uint32_t)(kDecEntries - 1)], C, enc);
                    last_at = pos + bits;
                    two |= c1.sym << C; bits += c1.bits;
                    broken |= c1.invalid;
                }
            }
            window >>= bits; have -= (int)bits; pos += bits;
            const int off = pp * C, i = off >> 5, s = off & 31;
            cw[i] |= two << s;
            if (s + 2 * C > 32) cw[i + 1] |= two >> (32 - s);
        }
        for (int i = 0; i < C; ++i) dst[i * 32 + lane] = cw[i];
    }
    if (last_pair) last_at += decode_one(last_pair, C, enc).bits;
    // no valid word, or a last coordinate that starts past the word behind the block's end
    if (broken || first + (int64_t)(last_at >> 5) > last) atomicOr(bad, LQ_CODE_BROKEN);
}

// Decoder on the run offsets.  A run is four lanes (128 coordinates) of a block; one CTA takes a tile (up to 128 blocks of
// one layer = 1024 runs) with the layer's decode table in shared memory.  First every thread looks at some runs: a
// run of 128 zero bits where "0" is the word of level 0 (what untouched rows turn into) is written as zeros at once;
// the other runs are collected in a list, so that the walk below is done by full warps and not by the few lanes of
// every warp whose run happens to hold values.  Then the warps take 32 runs of the list at a time and a thread walks one
// run from its recorded bit offset: the next 13 stream bits come from a funnel shift over two of three words kept in
// registers, one table lookup gives two coordinates (one, where symbols are wider than 5 bits or two do not fit 13 bits),
// A run that meets no valid word, that would read past the block's end, or
// that does not end where the next run starts reports a broken stream; nothing is read or written out of bounds.
//
// What bounds the walk is its instructions (per two coordinates about 16, and 10 more when one lane's pair does not fit) and,
// before, its loads: a thread that read its run word by word from global memory touched 16 lines a load and waited for
// every second one, so a run's words are brought to shared memory at once.  Mostly zero tiles were walked by one or two warps
// of a CTA while it took a CTA per 32 blocks, and each had its table to fetch first.
struct RunRef {
    const uint32_t* src;     // first word of the block's stream
    int nwords;              // words of the block that may be read
    uint32_t start_bit, end_bit;
    bool check_end;          // the run is followed by another run of the block (end_bit is known)
};

__device__ __forceinline__ uint32_t stream_word(const RunRef& r, int i) { return i < r.nwords ? __ldg(r.src + i) : 0u; }

// Shared memory of a CTA: decode table, list of runs, word lengths, then room for the stream words of every thread's run, an
// odd number of 16-byte pieces; a broken run can read up to 13 * 128 bits on from its first word.
constexpr int kRunsPerTile = kTileBlocks * LQ_CODE_RUNS;
__host__ __device__ constexpr int run_pieces(int C) { return (C + 2) | 1; }
constexpr int kRunList = kDecEntries * 2, kRunLen = kRunList + kRunsPerTile * 2, kRunTaken = kRunLen + 64;
constexpr int kRunSmem(int bits, int walkers) { return kRunTaken + walkers * 16 * run_pieces(bits + 1) + 256; }
extern __shared__ __align__(16) unsigned char run_smem[];

__device__ __forceinline__ uint32_t run_entry(uint32_t bits)
{
    return *reinterpret_cast<const uint16_t*>(run_smem + ((bits << 1) & (2u * kDecEntries - 2u)));
}

// A run of a whole (kFull) or partial block, words in shared memory: `at` is the address of the run's first word.  `len`: bits of every symbol's word and
// sign (pair tables).  Word i of lane l4 of the run goes to dst[32 i + l4].
// A lane of a partial block holds the first `real` of its 32 positions: rows before the layer's end, and its share of the last.
template <int C, bool kFull>
__device__ __forceinline__ bool walk_run(const RunRef& r, uint32_t at, const uint8_t* len, int64_t blk, int run, int64_t size, uint32_t* dst)
{
    const int rest = kFull ? 0 : (int)(size - blk * kBlockCoords);
    constexpr bool kPair = C <= kDecPairBits;
    const uint32_t at0 = at;
    uint32_t lo = lds_u32(at), hi = lds_u32(at + 4u), nx = lds_u32(at + 8u);       // `lo` is the word at `at`
    uint32_t sh = r.start_bit & 31u, flags = 0;
#pragma unroll 1
    for (int l4 = 0; l4 < 4; ++l4) {
        uint32_t cw[C + 1];
#pragma unroll
        for (int i = 0; i <= C; ++i) cw[i] = 0u;
        const int real = kFull ? 32 : real_positions(rest, 4 * run + l4);
#pragma unroll
        for (int pp = 0; pp < 32; pp += 2) {
            if (!kFull && pp >= real) break;
            // with sh < 32 the 32 bits from the current position lie inside {lo, hi}; two coordinates take at most 26
            asm volatile("{\n\t.reg .pred p;\n\tsetp.ge.u32 p, %3, 32;\n\t@p mov.u32 %0, %1;\n\t@p mov.u32 %1, %2;\n\t"
                         "@p ld.shared.u32 %2, [%4+12];\n\t@p add.u32 %4, %4, 4;\n\tand.b32 %3, %3, 31;\n\t}"
                         : "+r"(lo), "+r"(hi), "+r"(nx), "+r"(sh), "+r"(at));
            const uint32_t win = __funnelshift_r(lo, hi, sh);
            const uint32_t e = run_entry(win);
            uint32_t sy, bits = e >> kDecLenShift;
            if (kPair) {
                sy = e & ((1u << (2 * C)) - 1u);
                if (!kFull && pp + 1 == real) {
                    sy = e & ((1u << C) - 1u);
                    flags |= (e & kDecSingle) ? e : 0u;
                    if (!(e & kDecSingle)) bits = len[sy];             // the first one's share of the pair's
                } else if (e & kDecSingle) {
                    const uint32_t e1 = run_entry(win >> bits), s1 = e1 & ((1u << C) - 1u);
                    flags |= e | e1;
                    sy |= s1 << C;
                    bits += (e1 & kDecSingle) ? e1 >> kDecLenShift : (uint32_t)len[s1];
                }
            } else {
                flags |= e;
                sy = e & 0x1ffu;
                if (kFull || pp + 1 < real) {
                    const uint32_t e1 = run_entry(win >> bits);
                    flags |= e1;
                    sy |= (e1 & 0x1ffu) << C;
                    bits += e1 >> kDecLenShift;
                }
            }
            sh += bits;
            const int off = pp * C, i = off >> 5, s = off & 31;
            cw[i] += sy << s;                                // the fields do not overlap: a multiply-add
            if (s + 2 * C > 32) cw[i + 1] |= sy >> (32 - s);
        }
#pragma unroll
        for (int i = 0; i < C; ++i) __stcs(dst + 32 * i + l4, cw[i]);
    }
    const uint32_t used = (r.start_bit & ~31u) + 8u * (at - at0) + sh;
    return (flags & (kPair ? kDecPairInvalid : kDecInvalid)) != 0u || (r.check_end ? used != r.end_bit : used > 32u * (uint32_t)r.nwords);
}

// Runs of more words than there is room for, and broken ones: coordinate by coordinate, from global memory, a word ahead of
// the 64 bits being read.  What a broken run decodes to is thereby the stream's doing alone: the walk goes on over the
// block's other words, and zeros past its end.
static __device__ __noinline__ bool walk_run_plain(const RunRef r, int C, const uint8_t* len, int64_t blk, int run, int64_t size,
                                                   uint32_t* dst)
{
    int i = (int)(r.start_bit >> 5);
    uint64_t window = stream_word(r, i) >> (r.start_bit & 31u);
    int have = 32 - (int)(r.start_bit & 31u);
    uint32_t next = stream_word(r, ++i), pos = r.start_bit;
    bool invalid = false;
    const bool pairs = C <= kDecPairBits;
#pragma unroll 1
    for (int l4 = 0; l4 < 4; ++l4) {
        uint64_t acc = 0;
        int fill = 0, word = 0;
#pragma unroll 4
        for (int pp = 0; pp < 32; ++pp) {
            uint32_t sym = 0;
            if (real_coord(blk, 4 * run + l4, pp, size)) {
                if (have < kDecBits) {
                    window |= (uint64_t)next << have;
                    have += 32;
                    next = stream_word(r, ++i);
                }
                const uint32_t e = run_entry((uint32_t)window);
                uint32_t bits = e >> kDecLenShift;
                if (pairs) {
                    sym = e & ((1u << C) - 1u);
                    invalid |= (e & kDecPairInvalid) != 0u;
                    if (!(e & kDecSingle)) bits = len[sym];            // the first one's share of the pair's
                } else {
                    sym = e & 0x1ffu;
                    invalid |= (e & kDecInvalid) != 0u;
                }
                pos += bits; window >>= bits; have -= (int)bits;
            }
            acc |= (uint64_t)sym << fill;
            fill += C;
            if (fill >= 32) { dst[32 * word++ + l4] = (uint32_t)acc; acc >>= 32; fill -= 32; }
        }
    }
    return invalid || (r.check_end ? pos != r.end_bit : pos > 32u * (uint32_t)r.nwords);
}

// The C words of each of a run's four lanes, which are neighbours: 16 bytes per plane where the message allows it.
__device__ __forceinline__ void store_zero_lanes(uint32_t* dst, bool vec)
{
    if (vec) { __stcs(reinterpret_cast<uint4*>(dst), make_uint4(0u, 0u, 0u, 0u)); return; }
    dst[0] = 0u; dst[1] = 0u; dst[2] = 0u; dst[3] = 0u;
}

__global__ void __launch_bounds__(kThreads, 4) entropy_decode_runs_kernel(PlanDev p, const uint32_t* __restrict__ in, int64_t capacity,
                                                                       const uint32_t* __restrict__ offsets,
                                                                       const uint16_t* __restrict__ run_offsets,
                                                                       const uint32_t* __restrict__ enc_tables,
                                                                       const uint16_t* __restrict__ dec_tables,
                                                                       uint32_t* __restrict__ packed, uint32_t* __restrict__ bad, bool vec, int walkers)
{
    __shared__ int ntodo;
    uint16_t* dec = reinterpret_cast<uint16_t*>(run_smem);
    uint16_t* todo = reinterpret_cast<uint16_t*>(run_smem + kRunList);
    uint8_t* len = run_smem + kRunLen;
    const TileJob T = p.jobs[blockIdx.x];
    const int layer = T.layer, k = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int C = T.bits + 1;
    {
        const uint4* src = reinterpret_cast<const uint4*>(dec_tables + (int64_t)layer * kDecEntries);
        uint4* dst = reinterpret_cast<uint4*>(dec);
#pragma unroll
        for (int i = 0; i < kDecEntries / 8 / kThreads; ++i) dst[i * kThreads + threadIdx.x] = __ldg(src + i * kThreads + threadIdx.x);
        if (C <= kDecPairBits && threadIdx.x < 1 << C)
            len[threadIdx.x] = (uint8_t)((enc_tables[(int64_t)layer * kMaxLevels + (threadIdx.x >> 1)] >> 16) + (threadIdx.x > 1 ? 1 : 0));
    }
    if (threadIdx.x == 0) ntodo = 0;
    const uint32_t* off_k = offsets + (int64_t)k * (p.total_blocks + 1);
    const uint32_t* stream = in + (int64_t)k * capacity;
    uint32_t* msg = packed + (int64_t)k * p.packed_words + T.word_off;
    // the run with index t of this tile: block t / 8, run t % 8
    auto run_ref = [&](int t, int64_t& blk) {
        blk = T.block0 + (t >> 3);
        const int64_t g = T.block_off + blk;
        const int64_t first = off_k[g], last = min((int64_t)off_k[g + 1], capacity);
        const uint16_t* ro = run_offsets + ((int64_t)k * p.total_blocks + g) * LQ_CODE_RUNS;
        const int run = t & 7;
        RunRef r;
        r.src = stream + first;
        r.nwords = (int)max((int64_t)0, last - first);
        r.start_bit = ro[run];
        r.check_end = run + 1 < LQ_CODE_RUNS;
        r.end_bit = r.check_end ? (uint32_t)ro[run + 1] : 0u;
        return r;
    };
    __syncthreads();
    const bool zero_bit = dec[0] == (uint16_t)zero_bit_entry(C);

    bool broken = false;
    for (int t0 = 0; t0 < T.nblocks * LQ_CODE_RUNS; t0 += kThreads) {
        const int t = t0 + threadIdx.x;
        bool walk = false;
        if (t < T.nblocks * LQ_CODE_RUNS) {
            int64_t blk;
            const RunRef r = run_ref(t, blk);
            uint32_t* dst = msg + blk * (int64_t)C * 32 + 4 * (t & 7);
            walk = true;
            if ((int64_t)(r.start_bit >> 5) > (int64_t)r.nwords) {            // an offset that points past the block's end:
                broken = true; walk = false;                                 // the run's words are still written (zeros)
            } else if (zero_bit && (blk + 1) * kBlockCoords <= T.size) {
                // 128 coordinates of level 0 are 128 zero bits; the last run of a block is followed by zero padding
                // up to the block's last word
                const uint32_t nbits = r.check_end ? r.end_bit - r.start_bit : 32u * (uint32_t)r.nwords - r.start_bit;
                if (r.check_end ? nbits == 128u : (nbits >= 128u && nbits < 160u)) {
                    const uint32_t end = r.start_bit + nbits;
                    const int w0 = (int)(r.start_bit >> 5), w1 = (int)(end >> 5);
                    uint32_t any = stream_word(r, w0) >> (r.start_bit & 31u);
#pragma unroll
                    for (int i = 1; i < 6; ++i) {
                        const uint32_t x = stream_word(r, w0 + i);
                        if (w0 + i < w1) any |= x;
                        else if (w0 + i == w1 && (end & 31u)) any |= x << (32u - (end & 31u));
                    }
                    walk = any != 0u;
                }
            }
            if (!walk)
                for (int i = 0; i < C; ++i) store_zero_lanes(dst + i * 32, vec);
        }
        const uint32_t m = __ballot_sync(0xffffffffu, walk);
        int at = 0;
        if (lane == 0 && m) at = atomicAdd(&ntodo, __popc(m));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (walk) todo[at + __popc(m & ((1u << lane) - 1u))] = (uint16_t)t;
    }
    __syncthreads();
    const int n = ntodo;
    const int pieces = run_pieces(C);
    const uint32_t taken = (uint32_t)__cvta_generic_to_shared(run_smem + kRunTaken) + threadIdx.x * pieces * 16;
    const bool in_vec = reinterpret_cast<uintptr_t>(in) % 16 == 0;
    for (int i0 = warp * 32 < walkers ? warp * 32 : n; i0 < n; i0 += walkers) {
        if (i0 + lane >= n) continue;
        const int t = todo[i0 + lane];
        int64_t blk;
        const RunRef r = run_ref(t, blk);
        uint32_t* dst = msg + blk * (int64_t)C * 32 + 4 * (t & 7);
        const int w0 = (int)(r.start_bit >> 5), w1 = r.check_end ? min((int)((r.end_bit + 31u) >> 5), r.nwords) : r.nwords;
        const uintptr_t at = reinterpret_cast<uintptr_t>(r.src + w0), to = reinterpret_cast<uintptr_t>(r.src + w1);
        const uintptr_t from = at & ~(uintptr_t)15;
        bool again = w1 <= w0 || to - from > (uintptr_t)(16 * pieces);
        if (!again) {
            if (in_vec) {
                for (uintptr_t f = from; f < to; f += 16)
                    cp_async16(taken + (uint32_t)(f - from), reinterpret_cast<const void*>(f), (int)min((uintptr_t)16, to - f));
            } else {
                for (uintptr_t f = at; f < to; f += 4) cp_async4(taken + (uint32_t)(f - from), reinterpret_cast<const void*>(f));
            }
            cp_async_commit();
            cp_async_wait<0>();
            const uint32_t first = taken + (uint32_t)(at - from);
            switch ((blk + 1) * kBlockCoords <= T.size ? C : -C) {
#define LQ_CASE(CC) case CC:  again = walk_run<CC, true>(r, first, len, blk, t & 7, T.size, dst); break;  \
                    case -CC: again = walk_run<CC, false>(r, first, len, blk, t & 7, T.size, dst); break;
                LQ_CASE(2) LQ_CASE(3) LQ_CASE(4) LQ_CASE(5) LQ_CASE(6) LQ_CASE(7) LQ_CASE(8) LQ_CASE(9)
#undef LQ_CASE
                default: break;
            }
        }
        // a broken run has read on past its own words into other threads': its words are formed again, from the block's
        if (again) broken |= walk_run_plain(r, C, len, blk, t & 7, T.size, dst);
    }
    if (broken) atomicOr(bad, LQ_CODE_BROKEN);
}

}  // namespace

cudaError_t launch_build_decode_tables(const PlanDev& p, int layer0, int layers, const uint32_t* enc_tables, uint16_t* dec_tables,
                                       cudaStream_t s)
{
    if (layers == 0) return cudaSuccess;
    return launch_as(false, build_decode_tables_kernel, (unsigned)layers, 1024, 0, 1, s, p, layer0, enc_tables, dec_tables);
}

cudaError_t launch_entropy_encode(const PlanDev& p, const uint32_t* packed, const uint32_t* enc_tables,
                                  uint32_t* offsets, uint32_t* out, int64_t capacity, uint16_t* run_offsets,
                                  EncodeScratch scratch, uint32_t* bad, cudaStream_t s)
{
    if (p.num_tiles == 0) return cudaSuccess;
    if (scratch.by_width) return launch_entropy_encode_by_width(p, packed, enc_tables, offsets, out, capacity, run_offsets, scratch, bad, s);
    cudaError_t e = cudaMemsetAsync(scratch.states, 0, scratch.bytes, s);
    if (e != cudaSuccess) return e;
    const uint32_t code_bytes = code_table_bytes(p);
    static std::atomic<uint64_t> configured{0};
    e = opt_in_shared_memory(configured, kEncodeSmem, entropy_encode_kernel<kByTicket>);
    if (e != cudaSuccess) return e;
    entropy_encode_kernel<kByTicket><<<(unsigned)((int64_t)p.num_tiles * p.num_workers), kThreads, code_bytes + kCodeBufBytes, s>>>(
        p, packed, enc_tables, offsets, out, capacity, run_offsets, scratch.sized, scratch.states + 1, reinterpret_cast<uint32_t*>(scratch.states),
        scratch.looks, bad, code_bytes);
    return cudaGetLastError();
}

cudaError_t launch_entropy_decode(const PlanDev& p, const uint32_t* in, int64_t capacity, const uint32_t* offsets,
                                  const uint16_t* run_offsets, const uint32_t* enc_tables, const uint16_t* dec_tables,
                                  uint32_t* packed, uint32_t* bad, cudaStream_t s)
{
    if (p.total_blocks == 0) return cudaSuccess;
    if (run_offsets) {
        static std::atomic<uint64_t> configured{0};
        const cudaError_t e = opt_in_shared_memory(configured, kRunSmem(LQ_MAX_BITS, kThreads), entropy_decode_runs_kernel);
        if (e != cudaSuccess) return e;
        const dim3 grid_r((unsigned)p.num_tiles, (unsigned)p.num_workers);
        // where tiles have few runs (layers of a few blocks) half of the threads do the walking, and the shared memory of the
        // others' runs makes room for a CTA more (of more than fit at once): 306 layers, 2 800 blocks, 12 workers at 8 bits, 88.0 us with
        // 256 walkers and 73.9 with 128
        const int walkers = LQ_CODE_RUNS * p.total_blocks <= (kThreads / 2) * (int64_t)p.num_tiles &&
                                    (int64_t)p.num_tiles * p.num_workers > 3 * kSms ? kThreads / 2 : kThreads;
        entropy_decode_runs_kernel<<<grid_r, kThreads, kRunSmem(p.most_bits, walkers), s>>>(
            p, in, capacity, offsets, run_offsets, enc_tables, dec_tables, packed, bad, reinterpret_cast<uintptr_t>(packed) % 16 == 0,
            walkers);
        return cudaGetLastError();
    }
    const dim3 grid((unsigned)((p.total_blocks + 127) / 128), (unsigned)p.num_workers);
    entropy_decode_kernel<<<grid, 128, 0, s>>>(p, in, capacity, offsets, enc_tables, dec_tables, packed, bad);
    return cudaGetLastError();
}

}  // namespace lq
