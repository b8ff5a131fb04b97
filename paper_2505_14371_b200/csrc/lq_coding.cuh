// Decode table of the entropy stage (shared by the kernel that builds it and the ones that read it).
// One entry per value of the next kDecBits = 13 stream bits (first bit in bit 0): a code word is at most
// kCodeMaxLen = 12 bits and a non-zero level is followed by its sign bit, so 13 bits always hold one whole
// coordinate.  Symbol = 2 * level index + sign, of C = b + 1 bits.
//   C <= kDecPairBits: the symbols of two coordinates (bits 0..4 and C up) and the bits that both take << kDecLenShift; where
//     13 bits do not hold the second one, the first symbol, its bits and kDecSingle; no word matches (incomplete codes):
//     kDecSingle, kDecPairInvalid and 1 bit.
//   wider: symbol (bits 0..8) | bits taken (word + sign, 1..13) << kDecLenShift; no match: kDecInvalid | 1 bit.
// The invalid flags are sticky when entries are OR-ed together, and a walker still advances.
#pragma once
#include "lq_internal.cuh"

namespace lq {

constexpr int kDecBits = kCodeMaxLen + 1;
constexpr int kDecEntries = 1 << kDecBits;
constexpr uint32_t kDecInvalid = 1u << 9;
constexpr int kDecLenShift = 12;
constexpr int kDecPairBits = 5;
constexpr uint32_t kDecSingle = 1u << 10;
constexpr uint32_t kDecPairInvalid = 1u << 11;
// entry 0 when level 0 is the word "0": symbol 0 in one bit, or two of them in two
__host__ __device__ constexpr uint32_t zero_bit_entry(int C) { return (C <= kDecPairBits ? 2u : 1u) << kDecLenShift; }

// ---- host side of the stage (lq_coding.cu) ----
bool huffman_lengths_host(const double* w, int n, int max_len, uint8_t* len);
bool canonical_codes_host(const uint8_t* len, int n, int max_len, uint32_t* code);
void build_code_table_host(const uint8_t* len, const uint32_t* code, int n, uint32_t* enc);

// Scratch of the encoder, owned by the plan: a counter from which its CTAs take their tiles, then what every (worker, tile)
// tells the tiles behind it; cleared before each encode.
// Whether an encode takes the tiles in the order of their widths.  ctas: tiles x workers; blocks: of all workers; widths: how many there
// are; runs: stretches of tiles of one width in the stream.  us by width and in stream order:
//   512 layers of 64 to 400 000 values, 4 workers (4484 CTAs): widths 1 to 8 in turn 114 and 218, 2, 3, 4 and 8 in turn 108 and 153, 3 and 4 in turn
//   96 and 101, 2 and 8 in turn 118 and 139, 8 layers of each width after the other (70 CTAs a run) 116 and 186, all layers of a width together 113 and 115;
//   184 layers up to 300 000, 2 workers (1098 CTAs): 1 to 8 in turn 37 and 42, the four 34.4 and 34.9, 3 and 4 in turn 31 and 28; 8 workers (2416
//   CTAs): 68 and 116, 65 and 88, 58 and 55; 16 layers of 4 and of 8 bits in turn (201 CTAs a run) 68 and 74;
//   300 layers up to 9000 (2 blocks a CTA), 4 workers (1212 CTAs): 35 and 41, 31 and 32, 27 and 25; 16 workers (4800 CTAs): 66 and 122, 62 and 80,
//   61 and 55; all layers of a width together (600 CTAs a run) 65 and 54;
//   60 layers, 2 workers (590 CTAs): 24 and 20; 128 layers up to 4 M (7176 CTAs of 30 blocks): 216 and 219, 195 and 191, 174 and 156.
inline bool entropy_by_width(int64_t ctas, int64_t blocks, int widths, int64_t runs)
{
    return widths >= 2 && widths * ctas >= 8500 && ctas <= 150 * runs && blocks < 24 * ctas && (widths > 2 || blocks >= 8 * ctas);
}

struct SizedBlocks {
    uint16_t* lane_bits;     // [K][total_blocks][32] the bits of every lane of every block
    uint8_t* rows;           // [K][total_blocks]
};
constexpr int kMostLooks = 1 << 22;      // some seconds
struct EncodeScratch {
    uint64_t* states;        // [1 + K * num_tiles]
    size_t bytes;
    int looks;               // at the words before a tile, until the tile gives up
    bool by_width;           // entropy_by_width
    SizedBlocks sized;       // by_width only: what the first of its launches tells the last
};
cudaError_t launch_build_decode_tables(const PlanDev& p, int layer0, int layers, const uint32_t* enc_tables, uint16_t* dec_tables,
                                       cudaStream_t s);
cudaError_t launch_entropy_encode(const PlanDev& p, const uint32_t* packed, const uint32_t* enc_tables,
                                  uint32_t* offsets, uint32_t* out, int64_t capacity, uint16_t* run_offsets,
                                  EncodeScratch scratch, uint32_t* bad, cudaStream_t s);
cudaError_t launch_entropy_encode_by_width(const PlanDev& p, const uint32_t* packed, const uint32_t* enc_tables, uint32_t* offsets, uint32_t* out,
                                           int64_t capacity, uint16_t* run_offsets, EncodeScratch scratch, uint32_t* bad, cudaStream_t s);
cudaError_t launch_entropy_decode(const PlanDev& p, const uint32_t* in, int64_t capacity, const uint32_t* offsets,
                                  const uint16_t* run_offsets, const uint32_t* enc_tables, const uint16_t* dec_tables, uint32_t* packed, uint32_t* bad,
                                  cudaStream_t s);

}  // namespace lq
