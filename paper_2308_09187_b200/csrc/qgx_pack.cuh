// qgx_encode in one pass (qgx_codec.cu, qgx_pack.cu).
#pragma once

#include "qgx_codec.cuh"

namespace qgx {

// The status word of a bucket in the look-back carries two sums at once: words in bits 0..32, unused bits at the ends of
// the buckets' last words in bits 33..61 -- so the last bucket of a worker knows the stream's bits, too.
constexpr int kPadShift = 33;

struct PackArgs {
  const float* norms;
  const uint8_t* sym;
  size_t d;
  int bucket, K;
  size_t nb;
  int load;                              // bytes per symbol load: 16 (k_pack_chunks), 8 (k_pack), 4 or 1
  uint32_t* stream;
  size_t cap_words;
  uint32_t* bucket_bits;
  uint64_t* total_bits;
  unsigned long long* status;            // [K][nb], zeroed before the launch
  unsigned int* ticket;                  // zeroed before the launch
  unsigned int first_ticket;             // K times the first bucket of every worker to encode (0 but for the diagnostic)
  int spin_limit;                        // polls of a wait for another bucket's words before it gives up
  DevStatus* st;
};

// Buckets of 1024 2^j coordinates, where there is enough of them.
bool pack_chunks_fits(int K, size_t nb, int bucket);
// status: K (nb + 1) words.  b_first: the first bucket of every worker to encode, less than nb.
qgx_status launch_pack_chunks(qgx_ctx* c, PackArgs a, size_t b_first, const CodeTable& ct);

}  // namespace qgx
