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
constexpr int kMostLooks = 1 << 22;      // some seconds
struct EncodeScratch {
    uint64_t* states;        // [1 + K * num_tiles]
    size_t bytes;
    int looks;               // at the words before a tile, until the tile gives up
};
cudaError_t launch_build_decode_tables(const PlanDev& p, int layer0, int layers, const uint32_t* enc_tables, uint16_t* dec_tables,
                                       cudaStream_t s);
cudaError_t launch_entropy_encode(const PlanDev& p, const uint32_t* packed, const uint32_t* enc_tables,
                                  uint32_t* offsets, uint32_t* out, int64_t capacity, uint16_t* run_offsets,
                                  EncodeScratch scratch, uint32_t* bad, cudaStream_t s);
cudaError_t launch_entropy_decode(const PlanDev& p, const uint32_t* in, int64_t capacity, const uint32_t* offsets,
                                  const uint16_t* run_offsets, const uint32_t* enc_tables, const uint16_t* dec_tables, uint32_t* packed, uint32_t* bad,
                                  cudaStream_t s);

}  // namespace lq
