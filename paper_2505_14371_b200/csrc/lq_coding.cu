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

#include "lq_coding.cuh"

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

// One warp per block, one CTA per tile (up to 128 blocks of one layer; on 32 the CTA's tables took longer than its blocks): the
// blocks are sized, the tile tells its words to the tiles behind it and learns where it starts itself, and the blocks are written.
// The tile's words are read a second time for that, from L2: 888 CTAs hold 80 KB each at 4 bits, 71 of its 126 MB.  Tiles are
// taken from a counter in stream order, so that a tile only waits for tiles that run already.
// What bounds it is instructions and, at the CTA's barriers, the warps that wait for each other (62 % of the issue slots are used).  Against a sizing pass, a scan and a writing
// pass, each over the whole message: Transformer-XL message (755 MB in, 291 MB out, 8 workers) 598 -> 568 us, 67 M coordinates at
// 3 bits 65.6 -> 57.3 us and at 8 bits 99.5 -> 91.5, 120 000 coordinates 18.5 -> 9.9 us (two launches instead of four).
// 5 CTAs per SM: with 6 (40 registers) 60.5 and 98.8 us at 3 and 8 bits, the same on the large message.  Blocks dealt out as warps
// come for them, against the waiting: 618 us, as the requests then follow a shared counter's answer.
__global__ void __launch_bounds__(kThreads, 5) entropy_encode_kernel(PlanDev p, const uint32_t* __restrict__ packed,
                                                                     const uint32_t* __restrict__ enc_tables,
                                                                     uint32_t* __restrict__ offsets,
                                                                     uint32_t* __restrict__ out, int64_t capacity,
                                                                     uint16_t* __restrict__ run_offsets, uint64_t* states,
                                                                     uint32_t* ticket, int looks, uint32_t* bad, uint32_t code_bytes)
{
    // tables of pairs of symbols, or of the single ones of wide codes, at a multiple of their size; a buffer for every warp's block
    extern __shared__ __align__(16) unsigned char enc_smem[];
    __shared__ uint32_t single[2 * kMaxLevels];
    __shared__ uint16_t lane_bits[kTileBlocks * 32];
    __shared__ uint32_t words[kTileBlocks];
    __shared__ uint8_t rows[kTileBlocks];
    __shared__ uint32_t slot_s, before_s, total_s;
    if (threadIdx.x == 0) slot_s = atomicAdd(ticket, 1u);
    __syncthreads();
    // Overlapping encodes of one plan, which the caller has to order, clear the counter under each other: more numbers are drawn
    // then than there are tiles.  What they write is wrong, but lies in the call's buffers.
    if (slot_s >= gridDim.x) return;
    const int t = (int)(slot_s / (uint32_t)p.num_workers), k = (int)(slot_s - (uint32_t)t * (uint32_t)p.num_workers);
    const Tile T = p.tiles[t];
    const int layer = T.layer, lane = threadIdx.x & 31;
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
    LQ_BLOCKS(false)
    __syncthreads();
    if (threadIdx.x < 32) {
        // where the tile's blocks start in it: four blocks a lane
        uint32_t v[kTileBlocks / 32], sum = 0;
#pragma unroll
        for (int i = 0; i < kTileBlocks / 32; ++i) {
            const int b = lane * (kTileBlocks / 32) + i;
            v[i] = b < T.nblocks ? words[b] : 0u;
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
        if (lane == 0) put_state(state + t, (t == 0 ? kTileEnd : kTileSum) | total);
        uint32_t at = incl - sum;
#pragma unroll
        for (int i = 0; i < kTileBlocks / 32; ++i) { words[lane * (kTileBlocks / 32) + i] = at; at += v[i]; }
        bool failed = false;
        const uint32_t before = words_before(state, t, lane, looks, failed);
        if (lane == 0) {
            if (t > 0) put_state(state + t, failed ? kTileLost : kTileEnd | (uint32_t)(before + total));
            if (failed) atomicOr(bad, LQ_CODE_GAVE_UP);
            before_s = before; total_s = failed ? 0xffffffffu : total;
        }
    }
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
    cudaError_t e = cudaMemsetAsync(scratch.states, 0, scratch.bytes, s);
    if (e != cudaSuccess) return e;
    // the room that any of the plan's widths asks for: its table, of pairs of symbols of up to kPairBits bits, and what aligning it may skip
    uint32_t code_bytes = 0;
    for (int C = p.least_bits + 1; C <= p.most_bits + 1; ++C) {
        const uint32_t table = C <= kPairBits ? 4u << (2 * C) : 4u << C;
        code_bytes = std::max(code_bytes, C == kPairBits ? table : 2u * table - 16u);
    }
    const uint32_t smem = code_bytes + kWarps * kCodeBufWords * 4;
    static std::atomic<uint64_t> configured{0};
    e = opt_in_shared_memory(configured, (4 << (2 * kPairBits)) + kWarps * kCodeBufWords * 4, entropy_encode_kernel);
    if (e != cudaSuccess) return e;
    entropy_encode_kernel<<<(unsigned)((int64_t)p.num_tiles * p.num_workers), kThreads, smem, s>>>(
        p, packed, enc_tables, offsets, out, capacity, run_offsets, scratch.states + 1, reinterpret_cast<uint32_t*>(scratch.states),
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
