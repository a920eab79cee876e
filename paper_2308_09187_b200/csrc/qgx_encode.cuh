// What the encode kernels of the fused exchange share: their arguments and the tables of a configuration.
#pragma once

#include "qgx_bucket.cuh"
#include "qgx_chunk.cuh"
#include "qgx_codec.cuh"

namespace qgx {

struct EncodeArgs {
  DualSource src;
  size_t d;
  int bucket;
  int K;
  size_t nb;
  int norm_type;
  uint32_t xid;
  uint64_t quad_base;           // (index of the vector's first coordinate in the generator's counter space) / 4
  bool vec_ok;
  bool v_vec, a_vec;            // the workers' rows / the shared vector are 16-byte aligned (whatever d is)
  uint32_t* stream;
  size_t cap_words;
  uint32_t* bucket_bits;        // [K][nb]
  uint32_t* offsets;            // [K][nb] word offset of each bucket
  unsigned long long* total_bits;   // [K], zero before the launch
  float* norms;                 // [K][nb] (kept for the caller; the streams carry them too)
  unsigned long long* status;   // [K][nb], zero before the launch
  unsigned int* ticket;         // zero before the launch
  const struct EncodeTables* tables;   // the shared-memory tables of the configuration, built once
  DevStatus* st;
  size_t b_first;               // first bucket of every worker to encode (0 but for the diagnostic)
  int spin_limit;               // polls of a wait for another bucket's count before it gives up
};

// The encoder's shared-memory tables as one block of global memory: built by one CTA when a configuration is first
// used and copied by every encode CTA after that (building them costs a CTA of a small bucket more than the bucket).
struct EncodeTables {
  float4 bin[kBinEntries];
  uint32_t pair[kPairLutSize];
  EncLut lut;
  float4 bin_fix[kBinEntries];             // the fixed-point rounding map of k_encode_pipeline
  uint32_t pair_fix[kPairLutSize];         // its pair table, (2 nlev)^2 entries: first + 2 nlev * second, a symbol being its level,
                                           // plus nlev for a negative coordinate
};
static_assert(sizeof(EncodeTables) % 16 == 0, "copied in 16-byte pieces");

struct PipePlan;
qgx_status launch_encode_pipeline(qgx_ctx* c, const EncodeArgs& ea, const LevelTable& lt, const CodeTable& ct, const PhiloxKey& key,
                                  const RoundTable& rt, const PipePlan& plan, bool early);

// The cut of a launch's work (see the kernel): chunks of kChunk coordinates, `unit` of them per unit of work, `units` units
// per worker; a unit has one status word, `status_ld` per worker of which the first `status_first` are never published
// (the diagnostic that leaves buckets out).
constexpr int kChunk = 1024;
struct PipePlan {
  int unit;
  size_t units, status_ld, status_first;
};
PipePlan plan_encode_pipeline(const qgx_ctx* c, int bucket, size_t nb, size_t b_first, int K);

}  // namespace qgx
