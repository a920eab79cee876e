// Walking a sub-block of a prefix-coded stream, two symbols per look-up (qgx_decode.cu).
#pragma once

#include "qgx_common.cuh"

namespace qgx {

// A symbol as the fused kernels keep it: its level, plus nlev for a negative coordinate; 2 nlev where no codeword starts like
// the bits.  So a byte is an index into a table of signed values (see fill_signed_values).
__host__ __device__ constexpr uint32_t bad_symbol(int nlev) { return 2u * (uint32_t)nlev; }
constexpr int kSignedValues = 2 * QGX_MAX_LEVELS + 1;

// signed level values by symbol; NaN for the symbol that is none, so that it shows in the sums
__device__ __forceinline__ void fill_signed_values(float* val, const LevelTable& lt) {
  for (int i = threadIdx.x; i < kSignedValues; i += blockDim.x)
    val[i] = i < lt.nlev ? lt.lev[i] : (i < 2 * lt.nlev ? -lt.lev[i - lt.nlev] : __int_as_float(0x7fc00000));
}

// The decoder's tables of a configuration, built on the device when it is first used (k_build_decode_tables).
//  pair:   index = the next pair_bits stream bits.  Bits 0..4 the bits that the next two symbols take, 8..12 those of the first
//          alone, 16..23 and 24..31 the symbols.  Where two symbols do not fit the index: bit 15 set, and the first symbol only.
//  single: index = the next maxlen + 1 bits; symbol | bits taken << 8.
constexpr int kPairBitsMax = 13;         // at least the longest symbol: a codeword of QGX_MAX_CODE_LEN and its sign
constexpr uint32_t kPairEscape = 0x8000u;
struct DecodeTables {
  uint32_t pair[1 << kPairBitsMax];
  uint16_t single[2 << QGX_MAX_CODE_LEN];
};
__host__ __device__ constexpr int pair_bits(int maxlen) { return 2 * (maxlen + 1) < kPairBitsMax ? 2 * (maxlen + 1) : kPairBitsMax; }

}  // namespace qgx
