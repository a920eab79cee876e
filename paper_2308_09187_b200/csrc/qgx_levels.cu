// Sufficient statistics of the level refit (Sec. 3.3): the histogram of normalized magnitudes,
// each coordinate weighted by its bucket's squared norm (the weights lambda_j of Eq. QAda), and
// qgx_update_levels, which feeds it to the host-side fit and code builders.
#include "qgx_bucket.cuh"

#include <algorithm>
#include <cstring>

namespace qgx {

constexpr int kMaxBins = 4096;

// Bin of one coordinate: floor(fl(fl(|x| / norm) * nbins)), clamped to the last bin -- the definition, in IEEE
// operations.
__device__ __forceinline__ int bin_exact(float x, float norm, float nbf, int nbins) {
  float u = (norm > 0.0f) ? __fdiv_rn(fabsf(x), norm) : 0.0f;
  u = fminf(u, 1.0f);
  return min((int)floorf(__fmul_rn(u, nbf)), nbins - 1);
}

// floor(t) of t = |x| * c, c = fl(nbins / norm), read from the mantissa of t + (2^23 - 1/2) -- one exact rounding to the
// nearest integer of t - 1/2 (which is -1/2 while t < 1/4 and reads as bin -1, an entry that is folded into bin 0) --
// and whether it may not be the bin of x: t differs from the defining product T by less than 4.0001 * 2^-24 * T <
// 2^-21.9 * t (four roundings), so floor(t) = floor(T) whenever t keeps a distance of 2^-21 * t from the integers.  With c
// a normal number and |x| <= norm (1 + 2^-24), t stays below nbins + 1/2: bins -1 .. nbins, the ones outside never vouched
// for but for bin -1 (t near nbins rounds to nbins - 1 or nbins, at a distance of 1/2).
struct FastBin { uint32_t pattern; bool unsafe; };
constexpr uint32_t kBinZero = 0x4B000000u;                            // pattern of 2^23: bin 0
__device__ __forceinline__ FastBin fast_bin(float x, float c) {
  const float kMagic = 8388607.5f;                                    // 2^23 - 1/2
  const float tt = __fmul_rn(fabsf(x), c);
  const float m = __fadd_rn(tt, kMagic);
  FastBin f;
  f.pattern = __float_as_uint(m);
  const float dist = __fsub_rn(tt, __fsub_rn(m, kMagic));             // t - (floor(t) + 1/2)
  f.unsafe = fabsf(dist) > __fmaf_rn(tt, -4.76837158203125e-07f, 0.5f);
  return f;
}

// Persistent CTAs: bucket t of the launch (b = t / K, k = t % K, so that CTAs working side by side share the
// operator's bucket in L2) belongs to CTA t mod gridDim.x.  Counts per bin of one bucket in shared memory, folded
// after each bucket into the CTA's own fp64 histogram (count * weight); one fp64 atomic per occupied bin and CTA at
// the end.
//
// Lanes of a warp that meet in a bin add up in one pass, lanes that meet in a bank only follow one another: a bucket whose
// magnitudes spread over the bins (L-infinity norm) costs half as much again as one that crowds into the lowest.  (Several
// counters per bin, one for every second, fourth or eighth lane, made both slower.)  A coordinate counts for the bin that
// fast_bin gives it; where that may be wrong (a few in a million for bins of small index) the thread's coordinates are read
// again afterwards and the count moved to the bin of the defining operations, so that the common path has neither a select
// nor a clamp.  A CTA works on its bucket phase by phase (load, norm, count, fold, a barrier between them), so the SM is kept
// busy by its other CTAs: the fewer threads a bucket has -- the more coordinates each -- the more of them there are.  Fetching
// the next bucket into registers early bought less than the CTAs it cost.  8 workers of 2^24 coordinates, 1024 bins, L2 and
// L-infinity: buckets of 16384 with eight quads per thread 145 and 216 us; 8192 with four, fetched early, 177 and 262, with eight
// 143 and 218; 4096 177 and 265, 142 and 234; 2048 with two 238 and 324, with four 166 and 269; 1024 with two 246 and 361, with
// four 199 (L2), with two and not early 351; 512 with one 360 and 534, with two 295 and 495.  DRAM alone would take 82.
template <int V4>
__global__ void __launch_bounds__(512, 2) k_histogram(DualSource src, size_t d, int bucket, size_t nb, int K, int norm_type,
                                                      int nbins, int weighted, bool vec_ok, double* __restrict__ hist,
                                                      DevStatus* st) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  double* s_hist = reinterpret_cast<double*>(s_raw);                 // [nbins], then 4 words, then the counters
  uint32_t* s_cnt = reinterpret_cast<uint32_t*>(s_hist + ((nbins + 1) & ~1)) + 4;   // [-1 .. nbins]
  __shared__ double s_red[34];
  for (int i = threadIdx.x; i < nbins; i += blockDim.x) s_hist[i] = 0.0;
  const int words = (nbins + 1 + 3) & ~3;                            // from bin 0 on
  for (int i = (int)threadIdx.x - 4; i < words; i += blockDim.x) s_cnt[i] = 0u;
  const float nbf = (float)nbins;
  const uint32_t cnt_base = smem_addr(s_cnt) - 4u * kBinZero;         // a bin: base + 4 * pattern, modulo 2^32
  const unsigned long long total = (unsigned long long)nb * (unsigned long long)K;
  BucketRegs<V4> r;
  for (unsigned long long t = blockIdx.x; t < total; t += gridDim.x) {
    const size_t b = (size_t)(t / (unsigned long long)K), k = (size_t)(t % (unsigned long long)K);
    const size_t lo = b * (size_t)bucket;
    const int len = (int)min((size_t)bucket, d - lo);
    load_bucket<V4>(r, src, k, d, lo, len, vec_ok);
    const float norm = V4 == 1 ? bucket_norm<V4>(r, norm_type, s_red) : bucket_norm_all<V4>(r, norm_type, s_red);
    const bool finite = (norm - norm) == 0.0f;
    if (!finite) {
      if (threadIdx.x == 0) latch_error(st, QGX_ERR_NONFINITE);
    } else {
      const float c = (norm > 0.0f) ? __fdiv_rn(nbf, norm) : 0.0f;
      if (len == (int)blockDim.x * V4 * kQuad && (c == 0.0f || (c >= 1.17549435e-38f && c <= 3.0e38f))) {
        // every thread's quads lie inside the bucket
        bool redo = false;                                         // one of this thread's coordinates is not safe
#pragma unroll
        for (int j = 0; j < V4; ++j) {
          const float x[kQuad] = {r.x[j].x, r.x[j].y, r.x[j].z, r.x[j].w};
#pragma unroll
          for (int q = 0; q < kQuad; ++q) {
            const FastBin f = fast_bin(x[q], c);
            redo = redo || f.unsafe;
            asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(cnt_base + 4u * f.pattern) : "memory");
          }
        }
        if (redo) {                                                // rare: the thread's coordinates are read again
          for (int j = 0; j < V4; ++j) {
            const size_t e = lo + (size_t)(j * (int)blockDim.x + (int)threadIdx.x) * kQuad;
            for (int q = 0; q < kQuad; ++q) {
              const float xq = dual_value(src, k, d, e + q);
              const FastBin f = fast_bin(xq, c);
              if (!f.unsafe) continue;
              asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(cnt_base + 4u * f.pattern), "r"(0xffffffffu) : "memory");
              atomicAdd(&s_cnt[bin_exact(xq, norm, nbf, nbins)], 1u);
            }
          }
        }
      } else {                                                     // a short last bucket: the defining operations
#pragma unroll
        for (int j = 0; j < V4; ++j) {
          const int e = (j * (int)blockDim.x + (int)threadIdx.x) * kQuad;
          const float x[kQuad] = {r.x[j].x, r.x[j].y, r.x[j].z, r.x[j].w};
#pragma unroll
          for (int q = 0; q < kQuad; ++q)
            if (e + q < len) atomicAdd(&s_cnt[bin_exact(x[q], norm, nbf, nbins)], 1u);
        }
      }
    }
    __syncthreads();
    if (finite) {
      const double wgt = weighted ? (double)norm * (double)norm : 1.0;
      uint4* s_four = reinterpret_cast<uint4*>(s_cnt);
      for (int i = threadIdx.x; i * 4 < nbins; i += blockDim.x) {   // four bins at a time
        uint4 n = s_four[i];
        if (i == 0) { n.x += s_cnt[-1]; s_cnt[-1] = 0u; }
        if ((n.x | n.y | n.z | n.w) == 0u) continue;
        if (n.x) s_hist[i * 4] += (double)n.x * wgt;
        if (n.y) s_hist[i * 4 + 1] += (double)n.y * wgt;           // (never past the last bin: nothing stays counted there)
        if (n.z) s_hist[i * 4 + 2] += (double)n.z * wgt;
        if (n.w) s_hist[i * 4 + 3] += (double)n.w * wgt;
        s_four[i] = make_uint4(0u, 0u, 0u, 0u);
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nbins; i += blockDim.x) {
    const double h = s_hist[i];
    if (h != 0.0) atomicAdd(&hist[i], h);
  }
}

qgx_status launch_histogram(qgx_ctx* c, DualSource src, int K, size_t d, int bucket, int norm_type, int nbins, int weighted,
                            double* hist) {
  if (!c || !hist || K < 1 || K > 65535 || d < 1 || bucket < kQuad || bucket > QGX_MAX_BUCKET || bucket % kQuad != 0 ||
      nbins < 1 || nbins > kMaxBins || (norm_type != QGX_NORM_L2 && norm_type != QGX_NORM_LINF))
    return QGX_ERR_INVALID_ARG;
  if (cudaSetDevice(c->device) != cudaSuccess) return QGX_ERR_CUDA;
  if (cudaMemsetAsync(hist, 0, sizeof(double) * (size_t)nbins, c->stream) != cudaSuccess) return QGX_ERR_CUDA;
  const size_t nb = (d + (size_t)bucket - 1) / (size_t)bucket;
  const bool vec_ok = (d % kQuad == 0) && ((reinterpret_cast<uintptr_t>(src.v) & 15u) == 0) &&
                      ((reinterpret_cast<uintptr_t>(src.a) & 15u) == 0);
  const int v4 = bucket <= 256 ? 1 : (bucket <= 512 ? 2 : (bucket <= 1024 ? (norm_type == QGX_NORM_L2 ? 4 : 2) : (bucket <= 2048 ? 4 : 8)));
  const int threads = bucket_threads(bucket, v4);
  const size_t smem = sizeof(double) * (size_t)((nbins + 1) & ~1) + sizeof(uint32_t) * (4 + (((size_t)nbins + 1 + 3) & ~(size_t)3));
  const unsigned long long total = (unsigned long long)nb * (unsigned long long)K;
  ScopedKernelTimer timer(c, QGX_KERNEL_HISTOGRAM);
#define QGX_LAUNCH_H(V)                                                                                              \
  do {                                                                                                               \
    int per_sm = 1;                                                                                                  \
    if (smem > 40u * 1024u) cudaFuncSetAttribute(k_histogram<V>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem); \
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_histogram<V>, threads, smem);                        \
    const unsigned grid = (unsigned)std::min<unsigned long long>(total, (unsigned long long)c->num_sms * (unsigned long long)std::max(per_sm, 1)); \
    k_histogram<V><<<grid, threads, smem, c->stream>>>(src, d, bucket, nb, K, norm_type, nbins, weighted, vec_ok, hist, c->dstatus); \
  } while (0)
  switch (v4) {
    case 1: QGX_LAUNCH_H(1); break;
    case 2: QGX_LAUNCH_H(2); break;
    case 4: QGX_LAUNCH_H(4); break;
    default: QGX_LAUNCH_H(8); break;
  }
#undef QGX_LAUNCH_H
  count_launch(c);
  return cuda_status(cudaGetLastError());
}

// histogram -> host; levels refit; code rebuilt.  Synchronizes the stream.
qgx_status refit_from_source(qgx_ctx* c, DualSource src, int K, size_t d, qgx_quant_cfg* cfg, int refit, double* hist,
                             double* hist_host) {
  if (!cfg || refit == QGX_REFIT_NONE) return QGX_ERR_INVALID_ARG;
  if (cfg->nlev < 2 || cfg->nlev > QGX_MAX_LEVELS) return QGX_ERR_BAD_LEVELS;
  qgx_status rc = launch_histogram(c, src, K, d, cfg->bucket, cfg->norm_type, cfg->nbins, 1, hist);
  if (rc != QGX_OK) return rc;
  if (!c->hist_pinned && cudaMallocHost(&c->hist_pinned, sizeof(double) * kMaxBins) != cudaSuccess) return QGX_ERR_CUDA;
  const double* h = c->hist_pinned;                                    // pinned: the copy needs no staging
  if (cudaMemcpyAsync(c->hist_pinned, hist, sizeof(double) * (size_t)cfg->nbins, cudaMemcpyDeviceToHost, c->stream) != cudaSuccess ||
      cudaStreamSynchronize(c->stream) != cudaSuccess)
    return QGX_ERR_CUDA;
  rc = qgx_fit_levels(h, cfg->nbins, cfg->levels, cfg->nlev, refit == QGX_REFIT_FIRST ? 1 : 0);
  if (rc != QGX_OK) return rc;
  const int sub = cfg->cb.subblock;
  if (cfg->code_type == QGX_CODE_HUFFMAN) {
    double p[QGX_MAX_LEVELS];
    rc = qgx_symbol_pmf(h, cfg->nbins, cfg->levels, cfg->nlev, p);
    if (rc != QGX_OK) return rc;
    rc = qgx_build_codebook_huffman(p, cfg->nlev, sub, &cfg->cb);
  } else if (cfg->code_type == QGX_CODE_ELIAS) {
    rc = qgx_build_codebook_elias(cfg->nlev, sub, &cfg->cb);
  } else {
    rc = qgx_build_codebook_fixed(cfg->nlev, sub, &cfg->cb);
  }
  if (hist_host)
    std::memcpy(hist_host, h, sizeof(double) * (size_t)cfg->nbins);
  return rc;
}

}  // namespace qgx

using namespace qgx;

extern "C" {

qgx_status qgx_histogram(qgx_ctx* c, const float* v, int K, size_t d, int bucket, int norm_type, int nbins, int weighted,
                         double* hist) {
  if (!v) return QGX_ERR_INVALID_ARG;
  DualSource src{v, nullptr, 0, 0};
  return launch_histogram(c, src, K, d, bucket, norm_type, nbins, weighted, hist);
}

qgx_status qgx_update_levels(qgx_ctx* c, const float* v, int K, size_t d, qgx_quant_cfg* cfg, int refit, double* hist,
                             double* hist_host) {
  if (!v) return QGX_ERR_INVALID_ARG;
  DualSource src{v, nullptr, 0, 0};
  return refit_from_source(c, src, K, d, cfg, refit, hist, hist_host);
}

}  // extern "C"
