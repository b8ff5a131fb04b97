// The entropy encoder's kernel: of plans of one code width (lq_coding.cu) and of several side by side (lq_encode_by_width.cu), each
// with its own copy of the functions below: shared by the kernels of both, they cost the first ones 2 % (Transformer-XL message 571 -> 581 us).
#pragma once

#include <algorithm>

#include "lq_coding.cuh"

namespace lq {
namespace {

// Number of real coordinates among the 32 of this lane in block `blk`: coordinate of position p is
// blk * 1024 + 128 * (p / 4) + 4 * lane + p % 4.
__device__ __forceinline__ bool real_coord(int64_t blk, int lane, int p, int64_t size)
{
    return blk * kBlockCoords + 128 * (p >> 2) + 4 * lane + (p & 3) < size;
}

// Coordinates of lane `lane` inside a layer's last block, which holds `rest` of them: the first of its 32 positions (whole
// rows, then its share of the row that the layer ends in).
__device__ __forceinline__ int real_positions(int rest, int lane) { return 4 * (rest >> 7) + max(0, min(4, (rest & 127) - 4 * lane)); }

// symbol p of a lane's string of 32 symbols of C bits held in C words
template <int C>
__device__ __forceinline__ uint32_t symbol_at(const uint32_t (&w)[C + 1], int p)
{
    const int off = p * C, i = off >> 5, s = off & 31;
    const uint32_t v = s + C <= 32 ? w[i] >> s : __funnelshift_r(w[i], w[i + 1], s);
    return v & ((1u << C) - 1u);
}

// The encoder takes two coordinates at a time.  Entry of a pair of symbols: their stream bits (word, then the sign bit of a
// non-zero level; first bit in bit 0; at most 26 bits) in bits 0..26, the number of bits in bits 27..31.  Symbols of up to
// kPairBits bits have a table of pairs in shared memory, wider ones join the entries of two single symbols.
constexpr int kPairBits = 6;
constexpr int kLenShift = 27;
constexpr uint32_t kCodeMask = (1u << kLenShift) - 1u;

__device__ __forceinline__ uint32_t join_entries(uint32_t e0, uint32_t e1)
{
    const uint32_t l0 = e0 >> kLenShift;
    return ((e0 & kCodeMask) | ((e1 & kCodeMask) << l0)) | ((l0 + (e1 >> kLenShift)) << kLenShift);
}

// Where a string of bits moves on from bit o to bit o1 (their low six bits count, and o1 - o < 32), its last 32 bits before being
// r and the new ones the low bits of e: if a word is complete, it goes to shared memory at `out`, which moves on.  Predicated
// instructions and no branch: at nearly every step it is some lanes' turn.
__device__ __forceinline__ void sts_u32(uint32_t a, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
__device__ __forceinline__ void put_word(uint32_t& out, uint32_t r, uint32_t e, uint32_t o, uint32_t o1)
{
    asm volatile("{\n\t.reg .pred p;\n\t.reg .u32 t;\n\txor.b32 t, %3, %4;\n\tand.b32 t, t, 32;\n\tsetp.ne.u32 p, t, 0;\n\t"
                 "@p shf.l.wrap.b32 t, %1, %2, %3;\n\t@p st.shared.u32 [%0], t;\n\t@p add.u32 %0, %0, 4;\n\t}"
                 : "+r"(out) : "r"(r), "r"(e), "r"(o), "r"(o1) : "memory");
}

// The address of the table entry whose number times 4 is v.  Tables start at a multiple of their size; the largest ones, of pairs of
// 6-bit symbols, would lose a CTA of five to that.
template <int C>
__device__ __forceinline__ uint32_t entry_at(uint32_t code, uint32_t v) { return C == kPairBits ? v + code : v | code; }

// Entry of the coordinates pp, pp + 1 (pp even) of a lane's string.  `code`: shared-memory address of the layer's table.
template <int C>
__device__ __forceinline__ uint32_t pair_entry(uint32_t code, const uint32_t (&w)[C + 1], int pp)
{
    if constexpr (C <= kPairBits) {
        const int off = pp * C, i = off >> 5, s = off & 31;
        uint32_t v;                                              // 4 * (the pair's 2 C bits)
        if (s + 2 * C <= 32) v = s >= 2 ? (w[i] >> (s - 2)) : (w[i] << (2 - s));
        else                 v = __funnelshift_r(w[i], w[i + 1], s - 2);
        return lds_u32(entry_at<C>(code, v & (((1u << (2 * C)) - 1u) << 2)));
    } else {
        return join_entries(lds_u32(entry_at<C>(code, 4u * symbol_at<C>(w, pp))), lds_u32(entry_at<C>(code, 4u * symbol_at<C>(w, pp + 1))));
    }
}

// Entry of the single coordinate pp (table of pairs: its pair with symbol 0, without that one's bits).
template <int C>
__device__ __forceinline__ uint32_t single_entry(uint32_t code, const uint32_t (&w)[C + 1], int pp)
{
    const uint32_t e = lds_u32(entry_at<C>(code, 4u * symbol_at<C>(w, pp)));
    if constexpr (C <= kPairBits) {
        const uint32_t l = (e >> kLenShift) - (lds_u32(code) >> (kLenShift + 1));       // (entry 0: symbol 0 twice)
        return (e & ((1u << l) - 1u)) | (l << kLenShift);
    } else {
        return e;
    }
}

// In a partial block: the entry of coordinate pp and, where a table of pairs exists, of the one behind it, if it is real.
// (Joining two entries there as well cost the wide codes' functions registers in their whole blocks: 2 900 blocks, 12 workers
// at 8 bits 67.6 -> 71.0 us.)
template <int C>
constexpr int kPartialStep = C <= kPairBits ? 2 : 1;
template <int C>
__device__ __forceinline__ uint32_t partial_entry(uint32_t code, const uint32_t (&w)[C + 1], int pp, int real)
{
    if constexpr (C <= kPairBits)
        if (pp + 1 < real) return pair_entry<C>(code, w, pp);
    return single_entry<C>(code, w, pp);
}

// The rows of 128 coordinates of a block that hold anything but symbols 0, from the words of all lanes: bit j for row j (its four
// symbols sit in bits 4 C j .. 4 C (j + 1) of every lane's string).
template <int C>
__device__ __forceinline__ uint32_t rows_of(const uint32_t (&w)[C + 1])
{
    uint32_t any[C], rows = 0;
#pragma unroll
    for (int i = 0; i < C; ++i) any[i] = __reduce_or_sync(0xffffffffu, w[i]);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        uint32_t x = 0;
#pragma unroll
        for (int i = 0; i < C; ++i) {
            const int lo = 4 * C * j - 32 * i, hi = lo + 4 * C;         // the row's bits of word i
            if (lo < 32 && hi > 0) {
                const uint32_t below = hi >= 32 ? 0xffffffffu : (1u << (hi & 31)) - 1u;
                x |= any[i] & (lo <= 0 ? below : below & ~((1u << (lo & 31)) - 1u));
            }
        }
        rows |= (x != 0u ? 1u : 0u) << j;
    }
    return rows;
}

// Bits that a lane's 32 coordinates take in the stream; of a whole block's, rows of symbols 0 take 4 zero_bits.
template <int C>
__device__ __forceinline__ uint32_t lane_bits(uint32_t code, const uint32_t (&w)[C + 1], uint32_t rows, uint32_t zero_bits)
{
    uint32_t bits = 0;
    if (rows == 0xffu) {
#pragma unroll
        for (int pp = 0; pp < 32; pp += 2) bits += pair_entry<C>(code, w, pp) >> kLenShift;
    } else {
        bits = 4u * zero_bits * (8u - (uint32_t)__popc(rows));
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if ((rows >> j) & 1u) bits += (pair_entry<C>(code, w, 4 * j) >> kLenShift) + (pair_entry<C>(code, w, 4 * j + 2) >> kLenShift);
    }
    return bits;
}
// The same for a layer's last, partial block.
template <int C>
__device__ __forceinline__ uint32_t lane_bits_partial(uint32_t code, const uint32_t (&w)[C + 1], int real)
{
    uint32_t bits = 0;
#pragma unroll
    for (int pp = 0; pp < 32; pp += kPartialStep<C>)
        if (pp < real) bits += partial_entry<C>(code, w, pp, real) >> kLenShift;
    return bits;
}

// Stream bits on their way into a block's buffer: `r` holds the last 32 of them, `f` counts them from the block's first word on
// (its low six bits are what is looked at), and whenever a word is complete it is stored at the shared-memory address `dst`.
struct Emitter {
    uint32_t r, f, dst;
    // takes the low len < 32 bits of e
    __device__ __forceinline__ void push(uint32_t e, uint32_t len)
    {
        const uint32_t f1 = f + len;
        put_word(dst, r, e, f, f1);
        r = __funnelshift_r(r, e, len);
        f = f1;
    }
};

// Writes a whole block's lane into the block's buffer (shared-memory address) from bit `pos` on.  Every lane has 32 bits or more,
// so it completes the word it starts in, which at most the lane before it shares: completed words are stored plainly (zeros in
// the place of the lane before), and after all lanes have done so each ORs the bits it has left over into the word that the
// next lane has stored (the last lane stores them).  Four entries are looked up before they are pushed: a look-up cannot be
// moved above a store.  A row of symbols 0 is one run of zero bits where level 0's word is one of up to 7 zero bits.
template <int C>
__device__ __forceinline__ void emit_full(uint32_t code, const uint32_t (&w)[C + 1], int lane, uint32_t pos, uint32_t buf,
                                          uint32_t rows, uint32_t zero_bits, uint32_t zero_code)
{
    Emitter em{0u, pos, buf + ((pos >> 5) << 2)};
    if (rows == 0xffu) {
#pragma unroll
        for (int p8 = 0; p8 < 32; p8 += 8) {
            uint32_t e[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) e[i] = pair_entry<C>(code, w, p8 + 2 * i);
#pragma unroll
            for (int i = 0; i < 4; ++i) em.push(e[i], e[i] >> kLenShift);
        }
    } else {
        const bool quick = zero_code == 0u && zero_bits <= 7u;
        const uint32_t zero2 = (zero_code | (zero_code << zero_bits));           // two words of level 0
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if ((rows >> j) & 1u) {
                const uint32_t e0 = pair_entry<C>(code, w, 4 * j), e1 = pair_entry<C>(code, w, 4 * j + 2);
                em.push(e0, e0 >> kLenShift);
                em.push(e1, e1 >> kLenShift);
            } else if (quick) {
                em.push(0u, 4u * zero_bits);
            } else {
                em.push(zero2, 2u * zero_bits);
                em.push(zero2, 2u * zero_bits);
            }
        }
    }
    const uint32_t left = __funnelshift_l(em.r, 0u, em.f);
    __syncwarp();
    if (em.f & 31u) {
        if (lane == 31) sts_u32(em.dst, left);
        else asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(em.dst), "r"(left) : "memory");
    }
}

// The same for a layer's last, partial block, into a zeroed buffer.  (Layers of a few thousand values hardly have other
// blocks: walked coordinate by coordinate, the sizing pass over 17 of them took 4.4 us instead of 3.1.)
template <int C>
__device__ __forceinline__ void emit_partial(uint32_t code, const uint32_t (&w)[C + 1], int real, uint32_t pos, uint32_t buf)
{
#pragma unroll
    for (int pp = 0; pp < 32; pp += kPartialStep<C>) {
        if (pp >= real) continue;
        const uint32_t e = partial_entry<C>(code, w, pp, real);
        const uint64_t c = (uint64_t)(e & kCodeMask) << (pos & 31u);
        const uint32_t at = buf + ((pos >> 5) << 2);
        asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(at), "r"((uint32_t)c) : "memory");
        if (c >> 32) asm volatile("red.shared.or.b32 [%0+4], %1;" ::"r"(at), "r"((uint32_t)(c >> 32)) : "memory");
        pos += e >> kLenShift;
    }
}

constexpr int kCodeBufWords = kBlockCoords * (kCodeMaxLen + 1) / 32;      // longest block: every coordinate 13 bits

// What the warps of an encoder CTA share about their tile.
struct EncodeJob {
    const uint32_t* msg;         // the tile's words in this worker's message
    uint32_t* out;               // this worker's stream, at the tile's first word (second walk)
    uint16_t* runs;              // this worker's run offsets at the tile's first block, or NULL
    uint16_t* lane_bits;         // bits per lane and block of the tile (shared memory); not of blocks without rows
    uint32_t* words;             // words of every block of the tile, then where they start in the tile's (shared memory)
    uint8_t* rows;               // the blocks' rows that hold anything, kPartialRows for a partial block (shared memory)
    int64_t room;                // words of the stream buffer from `out` on
    int nblocks, rest;           // the tile's blocks; coordinates of its last one
    const uint32_t* enc;         // the layer's words
    uint32_t code, single, buf;  // shared-memory addresses: the layer's table, that of its single symbols, this warp's buffer
};
constexpr uint32_t kPartialRows = 0xfeu;       // (a partial block is looked at as a whole)

// The layer's table, by all warps of the CTA: per symbol (2 * level + sign) the level's word, the sign bit behind it unless the level is
// 0, and their length; per pair of symbols of up to kPairBits bits the same of both.
__device__ __forceinline__ void make_code_table(const EncodeJob& J, int C)
{
    const uint32_t one = C <= kPairBits ? J.single : J.code, nsym = 1u << C;
    for (uint32_t sym = threadIdx.x; sym < nsym; sym += kThreads) {
        const uint32_t e = J.enc[sym >> 1], l = e >> 16;
        sts_u32(one + 4u * sym, (sym >> 1) ? ((e & 0xffffu) | ((sym & 1u) << l) | ((l + 1u) << kLenShift)) : ((e & 0xffffu) | (l << kLenShift)));
    }
    __syncthreads();
    if (C <= kPairBits) {
        for (uint32_t i = threadIdx.x; i < nsym * nsym; i += kThreads)
            sts_u32(J.code + 4u * i, join_entries(lds_u32(one + 4u * (i & (nsym - 1u))), lds_u32(one + 4u * (i >> C))));
        __syncthreads();
    }
}

// A warp's blocks of a tile for one symbol width (its own function per width, so that each is compiled with
// its own register budget).  kWrite = false: every lane's bits, the block's words and its rows.  true: the blocks are written,
// those without rows without a look at the message.
// The next block's words are requested before the current one is worked on.  (The job by value: as
// a reference it lives in local memory, 763 -> 645 us for the whole encode; two or three blocks ahead: no faster.)
template <int C, bool kWrite>
__device__ __noinline__ void encode_blocks(const EncodeJob J)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int partial = J.rest < kBlockCoords ? J.nblocks - 1 : -1;
    uint32_t next[C];
    auto request = [&](int b) {
        if (b >= J.nblocks) return;
        const uint32_t* from = J.msg + b * (C * 32) + lane;
#pragma unroll
        for (int i = 0; i < C; ++i) next[i] = kWrite ? __ldcs(from + i * 32) : __ldcg(from + i * 32);
    };
    if (!kWrite) { request(warp); make_code_table(J, C); }
    const uint32_t zero = lds_u32(C <= kPairBits ? J.single : J.code), zero_bits = zero >> kLenShift, zero_code = zero & kCodeMask;    // the word of level 0
    if (!kWrite) {
        for (int b = warp; b < J.nblocks; b += kWarps) {
            uint32_t w[C + 1], any = 0;
#pragma unroll
            for (int i = 0; i < C; ++i) { w[i] = next[i]; any |= w[i]; }
            w[C] = 0u;
            request(b + kWarps);
            uint32_t rows = 0, total = 32u * zero_bits * 32u;
            if (b == partial || __any_sync(0xffffffffu, any != 0u)) {
                uint32_t bits;
                if (b != partial) {
                    rows = rows_of<C>(w);
                    bits = lane_bits<C>(J.code, w, rows, zero_bits);
                } else {
                    rows = kPartialRows;
                    bits = lane_bits_partial<C>(J.code, w, real_positions(J.rest, lane));
                }
                J.lane_bits[b * 32 + lane] = (uint16_t)bits;
                total = __reduce_add_sync(0xffffffffu, bits);
            }
            if (lane == 0) { J.words[b] = (total + 31u) >> 5; J.rows[b] = (uint8_t)rows; }
        }
        return;
    }
    const bool quick_zero = zero_code == 0u;
    // blocks without rows, where level 0's word is all zeros (untouched rows), are so many zero words
    auto loaded = [&](int b) { return b < J.nblocks && !(quick_zero && J.rows[b] == 0u); };
    if (loaded(warp)) request(warp);
    for (int b = warp; b < J.nblocks; b += kWarps) {
        const uint32_t first = J.words[b], rows = J.rows[b];
        uint32_t w[C + 1];
#pragma unroll
        for (int i = 0; i < C; ++i) w[i] = next[i];
        w[C] = 0u;
        if (loaded(b + kWarps)) request(b + kWarps);
        uint32_t* out = J.out + first + lane;
        if (rows == 0u && quick_zero) {
            if (J.runs && (lane & 3) == 0) J.runs[b * LQ_CODE_RUNS + (lane >> 2)] = (uint16_t)(32u * zero_bits * lane);
            if ((int64_t)first + 32 * zero_bits <= J.room)       // a stream buffer that is too small is never overrun
                for (uint32_t i = 0; i < zero_bits; ++i) __stcs(out + 32 * i, 0u);
            continue;
        }
        const uint32_t bits = rows == 0u ? 32u * zero_bits : (uint32_t)J.lane_bits[b * 32 + lane];
        uint32_t incl = bits;                                // inclusive prefix sum over the lanes
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        const uint32_t nwords = (__reduce_add_sync(0xffffffffu, bits) + 31u) >> 5;
        const uint32_t pos = incl - bits;
        // where the runs of four lanes (128 coordinates) start inside the block's stream: lets a decoder work on
        // eight runs of a block at once
        if (J.runs && (lane & 3) == 0) J.runs[b * LQ_CODE_RUNS + (lane >> 2)] = (uint16_t)pos;
        if (b != partial) {
            emit_full<C>(J.code, w, lane, pos, J.buf, rows, zero_bits, zero_code);
        } else {
            for (uint32_t i = lane; i < nwords; i += 32) sts_u32(J.buf + 4u * i, 0u);
            __syncwarp();
            emit_partial<C>(J.code, w, real_positions(J.rest, lane), pos, J.buf);
        }
        __syncwarp();
        if ((int64_t)first + nwords <= J.room) {
#pragma unroll 4
            for (uint32_t i = 0; i < nwords; i += 32)
                if (i + lane < nwords) __stcs(out + i, lds_u32(J.buf + 4u * (i + lane)));
        }
        __syncwarp();
    }
}

// What a tile tells the tiles behind it in the same worker's stream, one 64-bit word: its words (kTileSum) or all words up to
// its end (kTileEnd) in the low half, or that it does not know where it starts (kTileLost).  Written and read whole, and nothing
// else is passed on by it.
constexpr uint64_t kTileSum = 1ull << 32, kTileEnd = 2ull << 32, kTileLost = 3ull << 32;
__device__ __forceinline__ void put_state(uint64_t* a, uint64_t v) { asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(a), "l"(v) : "memory"); }
__device__ __forceinline__ uint64_t get_state(const uint64_t* a)
{
    uint64_t v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(a) : "memory");
    return v;
}

// The words of all tiles before tile t (one warp; state: this worker's words, one per tile): looks back 32 tiles at a time until
// one knows everything before it.  `failed`: a tile before it has told nothing in `looks` looks, or gave up itself.
__device__ __forceinline__ uint32_t words_before(const uint64_t* state, int t, int lane, int looks, bool& failed)
{
    uint32_t before = 0;
    for (int last = t - 1; last >= 0; last -= 32) {
        const int i = last - lane;
        uint64_t v = i >= 0 ? 0ull : kTileEnd;
        for (int look = 0;; ++look) {
            if (look >= looks) { failed = true; return 0u; }
            if ((v >> 32) == 0ull) v = get_state(state + i);
            if (__all_sync(0xffffffffu, (v >> 32) != 0ull)) break;
            if (look > 8) __nanosleep(100);
        }
        const uint32_t ends = __ballot_sync(0xffffffffu, (v & kTileEnd) != 0ull);
        const int upto = ends ? __ffs(ends) - 1 : 31;
        if (__any_sync(0xffffffffu, lane == upto && (v >> 32) == (kTileLost >> 32))) { failed = true; return 0u; }
        before += __reduce_add_sync(0xffffffffu, lane <= upto ? (uint32_t)v : 0u);
        if (ends) break;
    }
    return before;
}

// kByTicket: tiles in stream order, each of which finds out where it starts.  kSizes: the words of each tile, and what the first walk
// learned of its blocks, kept; kPlaced: the blocks written, their places known (both with tiles in the order of their widths).
constexpr int kByTicket = 0, kSizes = 1, kPlaced = 2;

// One warp per block, one CTA per tile (up to 128 blocks of one layer; on 32 the CTA's tables took longer than its blocks): the
// blocks are sized, the tile tells its words to the tiles behind it and learns where it starts itself, and the blocks are written.
// The tile's words are read a second time for that, from L2: the 740 CTAs that run at a time hold 80 KB each at 4 bits, 59 of its
// 126 MB, and 144 KB at 8, 107.  Tiles are taken from a counter in stream order, so that a tile only waits for tiles that run already.
// What bounds it is instructions (59 % of the issue slots are used) and, at the CTA's barriers, the warps that wait for each other (the
// largest stall, 2.9 per issue).  Against a sizing pass, a scan and a writing pass, each over the whole message: Transformer-XL message (755 MB
// in, 291 MB out, 8 workers) 598 -> 568 us, 67 M coordinates at 3 bits 65.6 -> 57.3 us and at 8 bits 99.5 -> 91.5, 120 000 coordinates 18.5
// -> 9.9 us (two launches instead of four).  The table of codes is made by the width's own code, behind the request of the first block:
// 400 layers of up to 8 blocks, 64 workers 209 -> 196 us.
// 5 CTAs per SM: with 6 (40 registers) 60.5 and 98.8 us at 3 and 8 bits, the same on the large message (by width, 512 layers of widths 1 to 8
// in turn, 114 and 117).  Blocks dealt out as warps come for them, against the waiting: 618 us, as the requests then follow a shared
// counter's answer.  A record per tile in stream order in place of tile and layer: 571 -> 585 us.
template <int kMode>
__global__ void __launch_bounds__(kThreads, 5) entropy_encode_kernel(PlanDev p, const uint32_t* __restrict__ packed,
                                                                     const uint32_t* __restrict__ enc_tables,
                                                                     uint32_t* __restrict__ offsets,
                                                                     uint32_t* __restrict__ out, int64_t capacity,
                                                                     uint16_t* __restrict__ run_offsets, SizedBlocks sized, uint64_t* states,
                                                                     uint32_t* ticket, int looks, uint32_t* bad, uint32_t code_bytes)
{
    // tables of pairs of symbols, or of the single ones of wide codes, at a multiple of their size; a buffer for every warp's block
    extern __shared__ __align__(16) unsigned char enc_smem[];
    __shared__ uint32_t single[2 * kMaxLevels];
    __shared__ __align__(16) uint16_t lane_bits[kTileBlocks * 32];
    __shared__ uint32_t words[kTileBlocks];
    __shared__ uint8_t rows[kTileBlocks];
    __shared__ uint32_t slot_s, before_s, total_s;
    uint32_t slot = blockIdx.x;
    if constexpr (kMode == kByTicket) {
        if (threadIdx.x == 0) slot_s = atomicAdd(ticket, 1u);
        __syncthreads();
        // Overlapping encodes of one plan, which the caller has to order, clear the counter under each other: more numbers are drawn
        // then than there are tiles.  What they write is wrong, but lies in the call's buffers.
        slot = slot_s;
        if (slot >= gridDim.x) return;
    }
    int t = (int)(slot / (uint32_t)p.num_workers);
    const int k = (int)(slot - (uint32_t)t * (uint32_t)p.num_workers), lane = threadIdx.x & 31;
    if constexpr (kMode != kByTicket) t = p.jobs[t].tile;
    const Tile T = p.tiles[t];
    const int layer = T.layer;
    const LayerDesc L = p.layers[layer];
    const int C = L.bits + 1;
    const uint32_t entries = C <= kPairBits ? 1u << (2 * C) : 1u << C;
    const uint32_t align = C == kPairBits ? 16u : 4u * entries;
    const uint32_t smem = (uint32_t)__cvta_generic_to_shared(enc_smem), code_at = (smem + align - 1u) & ~(align - 1u);
    EncodeJob J;
    J.msg = packed + (int64_t)k * p.packed_words + L.word_off + T.block0 * (int64_t)C * 32;
    J.runs = run_offsets ? run_offsets + ((int64_t)k * p.total_blocks + L.block_off + T.block0) * LQ_CODE_RUNS : nullptr;
    J.lane_bits = lane_bits; J.words = words; J.rows = rows;
    J.nblocks = T.nblocks;
    J.rest = (int)min((int64_t)kBlockCoords, L.size - (T.block0 + T.nblocks - 1) * (int64_t)kBlockCoords);
    J.out = nullptr; J.room = 0;
    J.enc = enc_tables + (int64_t)layer * kMaxLevels;
    J.code = code_at; J.single = (uint32_t)__cvta_generic_to_shared(single); J.buf = smem + code_bytes + (threadIdx.x >> 5) * (kCodeBufWords * 4);
#define LQ_BLOCKS(WRITE)                                                                                                  \
    switch (C) {                                                                                                          \
        case 2: encode_blocks<2, WRITE>(J); break; case 3: encode_blocks<3, WRITE>(J); break;                             \
        case 4: encode_blocks<4, WRITE>(J); break; case 5: encode_blocks<5, WRITE>(J); break;                             \
        case 6: encode_blocks<6, WRITE>(J); break; case 7: encode_blocks<7, WRITE>(J); break;                             \
        case 8: encode_blocks<8, WRITE>(J); break; case 9: encode_blocks<9, WRITE>(J); break;                             \
        default: break;                                                                                                   \
    }
    const int64_t block = (int64_t)k * p.total_blocks + L.block_off + T.block0;
    if constexpr (kMode == kSizes) { J.lane_bits = sized.lane_bits + block * 32; J.rows = sized.rows + block; J.words = offsets + block + k; }
    if constexpr (kMode == kPlaced) {
        if (threadIdx.x < T.nblocks) { words[threadIdx.x] = offsets[block + k + threadIdx.x]; rows[threadIdx.x] = sized.rows[block + threadIdx.x]; }
        const uint4* from = reinterpret_cast<const uint4*>(sized.lane_bits + block * 32);
        for (int i = threadIdx.x; i < T.nblocks * 4; i += kThreads) reinterpret_cast<uint4*>(lane_bits)[i] = from[i];
        make_code_table(J, C);
    } else {
        LQ_BLOCKS(false)
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        // where the tile's blocks start in it: four blocks a lane
        uint32_t v[kTileBlocks / 32], sum = 0;
#pragma unroll
        for (int i = 0; i < kTileBlocks / 32; ++i) {
            const int b = lane * (kTileBlocks / 32) + i;
            v[i] = b < T.nblocks ? (kMode == kSizes ? J.words[b] : words[b]) : 0u;
            sum += v[i];
        }
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += x;
        }
        const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
        uint64_t* state = states + (int64_t)k * p.num_tiles;
        if (kMode != kPlaced && lane == 0) put_state(state + t, (t == 0 ? kTileEnd : kTileSum) | total);
        if (kMode == kSizes) return;
        uint32_t at = incl - sum;
#pragma unroll
        for (int i = 0; i < kTileBlocks / 32; ++i) { words[lane * (kTileBlocks / 32) + i] = at; at += v[i]; }
        bool failed = false;
        const uint32_t before = words_before(state, t, lane, looks, failed);
        if (lane == 0) {
            if (kMode == kByTicket && t > 0) put_state(state + t, failed ? kTileLost : kTileEnd | (uint32_t)(before + total));
            if (failed) atomicOr(bad, LQ_CODE_GAVE_UP);
            before_s = before; total_s = failed ? 0xffffffffu : total;
        }
    }
    if (kMode == kSizes) return;
    __syncthreads();
    const uint32_t before = before_s;
    uint32_t* off = offsets + (int64_t)k * (p.total_blocks + 1) + L.block_off + T.block0;
    if (total_s == 0xffffffffu) {            // gave up: offsets that no stream has, and that a decoder refuses
        if (threadIdx.x < T.nblocks) off[threadIdx.x] = 0xffffffffu;
        if (threadIdx.x == 0 && t == p.num_tiles - 1) off[T.nblocks] = 0xffffffffu;
        return;
    }
    if (threadIdx.x < T.nblocks) off[threadIdx.x] = before + words[threadIdx.x];
    if (threadIdx.x == 0 && t == p.num_tiles - 1) off[T.nblocks] = before + total_s;
    J.out = out + (int64_t)k * capacity + before;
    J.room = capacity - (int64_t)before;
    LQ_BLOCKS(true)
#undef LQ_BLOCKS
}

// Shared memory of a warp's buffers, and of the largest table with them.
constexpr uint32_t kCodeBufBytes = kWarps * kCodeBufWords * 4;
constexpr int kEncodeSmem = (4 << (2 * kPairBits)) + (int)kCodeBufBytes;

// The room that any of the plan's widths asks for: its table, of pairs of symbols of up to kPairBits bits, and what aligning it may skip.
inline uint32_t code_table_bytes(const PlanDev& p)
{
    uint32_t bytes = 0;
    for (int C = p.least_bits + 1; C <= p.most_bits + 1; ++C) {
        const uint32_t table = C <= kPairBits ? 4u << (2 * C) : 4u << C;
        bytes = std::max(bytes, C == kPairBits ? table : 2u * table - 16u);
    }
    return bytes;
}

}  // namespace
}  // namespace lq
