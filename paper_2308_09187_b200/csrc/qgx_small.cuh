// The one-launch exchange of small vectors (qgx_exchange_small.cu).
#pragma once

#include "qgx_encode.cuh"
#include "qgx_walk.cuh"

namespace qgx {

constexpr int kSmallMaxWorkers = 16;     // the largest cluster (more than 8 where the device allows it)

struct SmallArgs {
  const DecodeTables* tables;
  float* mean;
  int update;                            // as DecodeArgs
  const float* xin;
  float* xout;
  const double* scalars;
  uint8_t* sym_out;
  const uint8_t* sym_prev;
  size_t sym_ld;
  const float* norms_prev;
  double* sum_sq;
  int square;                            // add the squared values themselves
  unsigned long long* total_out;         // the caller's copy of the totals, or null
  int total_add;                         // added to what is there
  uint32_t img_words, off_img, off_sym, off_tab;
};

bool small_exchange_size(const qgx_ctx* c, int K, size_t nb, int bucket);   // necessary, without the tables
bool small_exchange_fits(const qgx_ctx* c, int K, size_t nb, int bucket, const CodeTable& ct, const RoundTable& rt, bool octets, bool steps);
// After small_exchange_fits.  ea.status [K][nb] and ea.ticket [2] are zero before the launch and again after it.
qgx_status launch_exchange_small(qgx_ctx* c, const EncodeArgs& ea, SmallArgs r, const LevelTable& lt, const LevelTable& lt_kept,
                                 const CodeTable& ct, const PhiloxKey& key, const RoundTable& rt, bool early);

}  // namespace qgx
