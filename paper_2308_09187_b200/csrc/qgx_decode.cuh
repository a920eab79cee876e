// The fused exchange's decode pass (qgx_decode.cu).
#pragma once

#include "qgx_walk.cuh"

namespace qgx {

struct DecodeArgs {
  const uint32_t* stream;       // [K][cap_words]
  size_t cap_words;
  const uint32_t* bucket_bits;  // [K][nb]
  const uint32_t* offsets;      // [K][nb]
  size_t d;
  int bucket;
  int K;
  size_t nb;
  const DecodeTables* tables;
  float* mean;                  // [d]
  // optional fused state update (the two axpy of Eq. Q-GenX)
  int update;                   // 0 none, 1: xout = xin - gamma * mean, 2: xout = xin - mean
  const float* xin;
  float* xout;
  const double* scalars;        // scalars[1] = gamma_t
  bool vec_out;                 // mean, xin and xout 16-byte aligned: 128-bit stores
  // optional: keep the decoded symbols, worker k's coordinate i at byte k * sym_ld + i ...
  uint8_t* sym_out;             // [K][sym_ld] or null
  // ... or compare with the symbols and norms kept by the other exchange of the iteration:
  // *sum_sq += sum_k ||vhat_k of that exchange - vhat_k of this one||^2 (fp32 differences, fp64 sum)
  const uint8_t* sym_prev;      // [K][sym_ld] or null
  size_t sym_ld;                // a multiple of 4, at least d
  const float* norms_prev;      // [K][nb]
  double* sum_sq;
  // what the encode pass summed up, [K], or null; cleared here, as its scan's words are, for the next exchange
  unsigned long long* sums;
  unsigned long long* total_bits;   // [K], where the sums go, and the caller's copy of them or null
  unsigned long long* total_out;
  int total_add;                // added to what is there
  unsigned long long* scan;
  size_t scan_words;
  DevStatus* st;
};

// sym_mode, a set of bits: 1 keeps the decoded symbols; 2 adds the squared differences between the vectors kept by an
// earlier exchange (whose level table is `lt_kept`) and the ones decoded now to *sum_sq; 4 adds the squared decoded values
// themselves (an earlier vector of zero).  1 | 2 compares first and then overwrites the kept symbols in place.  early: see
// launch_next.
qgx_status launch_exchange_decode(qgx_ctx* c, const DecodeArgs& da, const CodeTable& ct, const LevelTable& lt, const LevelTable& lt_kept,
                                  int sym_mode, bool early);
void launch_build_decode_tables(const CodeTable& ct, DecodeTables* out, cudaStream_t stream);

}  // namespace qgx
