// Layout of the prepared-codebook block shared by prepare.cu and the kernels
// that read it.
#pragma once

#include "common.cuh"

namespace rvq {

constexpr uint32_t kPreparedMagic = 0x52565133u;
constexpr int kSlotCodewords = 128;                       // codewords per operand slot
// Operand slot of 128 codewords: thirteen cells of 16 bytes per codeword -- remainders as halves (4 cells), norm (1),
// heads (4), corrections in 8 bits (4).  An encoder copies nine of them: the first nine (remainders, norm, heads) or
// the last nine (norm, heads, corrections).
constexpr int kCellBytes = kSlotCodewords * 16;           // 2048
constexpr int kSlotStride = 13 * kCellBytes;              // 26624
constexpr int kSlotBytes = 9 * kCellBytes;                // 18432, as copied
constexpr int kSlotTail = 4 * kCellBytes;                 // where the last nine cells begin
constexpr size_t kPreparedParamsOffset = 256;             // StageParams[16]
constexpr size_t kPreparedMaximaOffset = 512;             // StageMaxima[16]
constexpr size_t kPreparedPartialsOffset = 768;           // StagePartial[16 stages][kPrepareParts], scratch of the prepare step
constexpr int kPrepareParts = 16;
constexpr size_t kPreparedImageOffset = 768 + 16 * 16 * 24;   // operand image, [R][slots][kSlotStride]

struct PreparedHeader {
    uint32_t magic, R, K, gd, slots;
    uint32_t decode_offset;   // byte offset of the decoder section, 0 if absent
    uint32_t even;            // 1: the codebooks suit the 8-bit corrections (kEvenKurtosis, kMostInverse); 2: packed scores as well (kPackedInverse)
};
// A stage's codewords count as even when the fourth moment of their entries is at most this many times the square of the
// second (3 for a normal distribution); the block does when at least half of its stages do and its codewords are not
// too small for the steps of the 8-bit operands.  The throughput encoder takes the 8-bit corrections by it (encode_tensor.cu).
constexpr float kEvenKurtosis = 6.0f;
// The 8-bit operands have a smallest step, so a row's window has a part that does not shrink with the row (window8): of
// the rows, whose norms follow the codewords', some 0.5 % + 5 % / norm have several candidates, the norm in the operands'
// scale (the largest of a stage is 45 ... 90), and each of them costs the more the smaller it is.  So a codeword counts by
// what 1 / norm has over kInverseFree, and the block by the mean.  (A fourth moment does not see it: with one group of
// four 1000 times smaller than the others it is 4.1.)  us with seven steps -> with five, by the mean; 194176 vectors on
// contiguous groups, 2048 codes unless said:
//   all groups alike 0: 1831 -> 1596; one of four 10 times smaller 0.04: 1843 -> 1652, 30 times 0.16: 1850 -> 1779, 100
//   times 0.57: 1852 -> 2361, 300 times 1.8: 1898 -> 5163, 1000 times 4: 1973 -> 41109;
//   outlier channels in one stage of eight, x200 0.08: 1815 -> 1734 (1024 codes 997 -> 1010), x1000 0.56: 1805 -> 10447;
//   in two, x60 0.09: 1821 -> 1684, x200 with 1024 codes 0.13: 992 -> 1044;
//   in four, x20 0.08: 1841 -> 1691 (1024 codes 0.05: 1012 -> 1027), x60 0.15: 1819 -> 1874, x1000 2.2: 1818 -> 36012.
// Back to back, under the power cap, five steps take 3-9 % less than that beside seven.
// Packed scores have a unit that does not shrink with the row either, 2^-16 of the range of a row against the largest
// codeword, and twice to four times the window.  65536 vectors, 2048 codes, us as they are / packed and share of the rows and stages
// with several candidates, one of four groups smaller than the others: alike 543 / 485, 1.0 %; 3 times 587 / 526, 1.7 %; 5 times
// (mean 0.009) 593 / 534, 2.2 %; 10 times (0.04) 570 / 691, 4.0 %.
constexpr float kMostInverse = 0.1f, kPackedInverse = 0.015f, kInverseFree = 0.0625f, kInverseCap = 16.0f;

// Decoder section (group_dim 32, R <= 8, K <= kDecodeMaxK): per stage an affine
// map value = lo_r + q * scale_r * base with q a 16-bit level, scale_r an integer in
// 1..255 and base common to all stages, so that the sum over the stages is
// sum lo_r + base * (sum q_r scale_r) with the second sum exact in 32-bit integers
// (at most 8 * 65535 * 255); then channel slices of the codebooks as levels:
// table[slice][code][stage 0..7][CH channels] uint16.  A slice is CH = 8
// channels wide (four slices) while K <= kDecodeWideK and 4 channels (eight
// slices) above, so that one slice of all codes fits the shared memory of a CTA.
struct DecodeParams {
    float step[8];     // value of one level, scale_r * base, per stage; 0 for absent stages
    float bias;        // sum over stages of the stage minimum lo_r
    float err;         // bound on |sum of table values - sum of float32 values| per channel
    float base;
    float pad[5];
    uint32_t scale[8]; // integer scale of a stage's levels (0 for absent stages)
    // Second set of tables ("summed levels"): the stages of one parity (even r, odd r) share a unit
    // fine enough that the levels of all four of them add up to at most 65535, so a decoder adds
    // table words as they are (two 16-bit fields per 32-bit word, no carry between them) and scales
    // once per parity.  Coarser than the tables above by a factor of about four.
    float pstep[2];      // value of one summed level, pscale * pbase, for even / odd stages; 0 if unused
    float perr;          // bound on |sum of summed-table values - sum of float32 values| per channel
    float pbase;         // common base of the two parities' units
    uint32_t pscale[2];  // integer scales (1..255) of the two parities
};
constexpr int kDecodeWideK = 1536;                        // 128 bytes per code per slice in shared memory
constexpr int kDecodeMaxK = 3072;                         // 64 bytes per code per slice
__host__ __device__ inline int decode_slice_channels(int K) { return K <= kDecodeWideK ? 8 : 4; }
__host__ __device__ inline size_t decode_table_bytes(int K) { return (size_t)K * 512; }   // 32 channels x 8 stages x 2 bytes
// the prepared block holds two such tables: levels scaled per stage, then levels summed per stage parity;
// the section: DecodeParams in 256 bytes, then the tables
__host__ __device__ inline size_t decode_section_bytes(int K) { return 256 + 2 * decode_table_bytes(K); }
static_assert(sizeof(DecodeParams) <= 256, "the decoder's parameters have 256 bytes");
constexpr int kDecodeExactWideK = 1792;                   // float32 tables: 128 bytes per code per 4-channel slice
constexpr int kDecodeExactK = 3584;                       // ... 64 bytes per code per 2-channel slice
// Which tables a shape can be decoded through (group_dim 32, a power-of-two number of groups up to 32, depth <= 8; of
// these, four groups and more take their codewords from L2 instead where decode_direct_wanted says so; everything
// else gathers from global memory):
//   - float32 table slices (exact sums, any output type) fit shared memory up to kDecodeExactK codes
//     (4 channels per slice up to kDecodeExactWideK, 2 beyond);
//   - 16-bit level tables (16-bit outputs only: their own rounding, 2^-9 or 2^-12 relative, dwarfs the
//     tables') fit up to kDecodeMaxK codes and are the faster ones while the deviations are moderate;
//   - where both fit (16-bit outputs, up to kDecodeMaxK codes) a sample of the deviations decides on the
//     device: four groups at depth 8 with up to kDecodeWideK codes in one launch that holds all three kinds of table, other
//     shapes as two launches of which the one not called for returns at once.
__host__ __device__ inline bool decode_exact_tables(const Shape &s)
{
    return s.gd == 32 && s.G <= 32 && (s.G & (s.G - 1)) == 0 && s.R <= 8 && s.K <= kDecodeExactK;
}
__host__ __device__ inline int decode_exact_channels(int K) { return K <= kDecodeExactWideK ? 4 : 2; }
__host__ __device__ inline bool decode_levels_prepared(const Shape &s)    // the prepared block holds level tables
{
    return s.gd == 32 && s.G <= 32 && (s.G & (s.G - 1)) == 0 && s.R <= 8 && s.K <= kDecodeMaxK;
}
__host__ __device__ inline bool decode_levels_supported(const Shape &s)
{
    return decode_levels_prepared(s) && s.dtype != RVQ_F32;
}
__host__ __device__ inline bool decode_sliced_supported(const Shape &s)
{
    return decode_exact_tables(s) || decode_levels_supported(s);
}
// Float32 section (group_dim 32, R <= kFloatMaxStages, K <= kFloatMaxK), after the decoder section: the
// codebooks as float32 with the pieces of a codeword apart, [R][blocks of 128 codewords][8 pieces][128][4], so
// that a block is one copy and neighbouring threads read neighbouring 16 bytes of it.  Padding codewords are
// infinite (never the nearest).
constexpr int kFloatMaxStages = 8;
constexpr int kFloatMaxK = 2048;
constexpr int kFloatBlockBytes = 128 * 128;
__host__ __device__ inline bool float_blocks_prepared(const Shape &s)
{
    return s.gd == 32 && s.R <= kFloatMaxStages && s.K <= kFloatMaxK;
}
__host__ __device__ inline size_t encode_image_bytes(const Shape &s)
{
    return s.gd == 32 ? (size_t)s.R * ((s.K + kSlotCodewords - 1) / kSlotCodewords) * kSlotStride : 0;
}

__host__ __device__ inline size_t decode_section_offset(const Shape &s)
{
    return (kPreparedImageOffset + encode_image_bytes(s) + 255) / 256 * 256;
}
__host__ __device__ inline size_t float_blocks_offset(const Shape &s)
{
    return decode_section_offset(s) + (decode_levels_prepared(s) ? decode_section_bytes(s.K) : 0);
}
__host__ __device__ inline size_t float_blocks_bytes(const Shape &s)
{
    return float_blocks_prepared(s) ? (size_t)s.R * ((s.K + 127) / 128) * kFloatBlockBytes : 0;
}

struct StageParams {
    float scale;    // 2^k applied to residuals and codewords of this stage
    float a, b;     // |score error| <= a * ||Z|| + b
    float unsafe;   // non-zero: the scaled codebook left the half-precision range
};

struct StagePartial {
    double max_norm2;   // largest squared norm among this part's codewords
    float sum2, sum4;   // sums of the entries' squares and fourth powers
    float lo, hi;       // smallest and largest entry
};

struct StageMaxima {
    uint32_t emax, eerr;                 // float bit patterns (non-negative), filled with atomicMax
    uint32_t inverse;                    // the codewords' sum of what 1 / norm has over kInverseFree, in units of 2^-11
    uint32_t elomax;                     // as emax
};

#ifdef __CUDACC__
// A row's eight (STEPS 4: four) codes as halves of words, stage by stage, into the order in which a lane visits its stages: at
// step k stage rot ^ k, so that the eight lanes of a quarter warp, whose rot are 0 ... 7, read eight different bank groups.
// (A rotation, stage rot + k, takes eight operations more.)
template <int STEPS>
__device__ __forceinline__ void exchange_codes(uint32_t rot, uint32_t &c0, uint32_t &c1, uint32_t &c2, uint32_t &c3)
{
    auto swap_if = [](bool yes, uint32_t &a, uint32_t &b) { const uint32_t t = yes ? b : a; b = yes ? a : b; a = t; };
    const uint32_t halves = (rot & 1u) ? 0x1032u : 0x3210u;
    swap_if(rot & 2u, c0, c1);
    c0 = __byte_perm(c0, 0u, halves); c1 = __byte_perm(c1, 0u, halves);
    if (STEPS == 8) {
        swap_if(rot & 2u, c2, c3);
        c2 = __byte_perm(c2, 0u, halves); c3 = __byte_perm(c3, 0u, halves);
        swap_if(rot & 4u, c0, c2);
        swap_if(rot & 4u, c1, c3);
    }
}
#endif

__host__ __device__ inline int slots_per_stage(int K) { return (K + kSlotCodewords - 1) / kSlotCodewords; }

}  // namespace rvq
