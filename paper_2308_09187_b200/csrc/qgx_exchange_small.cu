// A small exchange in one launch: quantize, encode, decode and average with one cluster of K CTAs per bucket, one CTA per
// worker.  A CTA rounds and packs its worker's bucket into an image in shared memory, decodes that image -- header lengths,
// codewords, signs, as any receiver would -- and the CTAs of the cluster then read one another's symbols through distributed
// shared memory to form the ordered sums, each for its share of the coordinates.  The image goes to its place in the stream
// meanwhile.
// What bounds it: latency.  The large kernels' way is five operations in a row (clearing the scan's words, encode, decode,
// sums, the copy of the totals), each a few microseconds of launch and of dependent loads whatever the size; here the
// chain is one load of the bucket, two barriers, a walk of one sub-block and one exchange between the CTAs.
#include "qgx_encode.cuh"
#include "qgx_small.cuh"

#include <algorithm>
#include <cooperative_groups.h>
#include <cstring>
#include <mutex>
#include <vector>

namespace cg = cooperative_groups;

namespace qgx {

// Fixed-point decision variable of a coordinate (see round_fixed) from a table with one copy per bin.
__device__ __forceinline__ uint32_t round_fixed_one(float x, uint32_t w, float rn, uint32_t shift, uint32_t base) {
  const float u2 = fmaf(fabsf(x), rn, kRoundShift);
  const float4 e = lds_table128(((__float_as_uint(u2) >> shift) & ~15u) + base);
  float z = fmaf(u2, e.y, e.x);
  z = fmaf(__saturatef(__fsub_rn(u2, e.z)), e.w, z);
  return __float_as_uint(z) - (w >> 16);
}

constexpr int kPadShift = 33;            // status words carry the words (low) and the unused bits (high) of the buckets so far

// Q quads per thread; G coordinates per sub-block.
template <int Q, int G>
__global__ void __launch_bounds__(Q == 4 ? 1024 : 512)
k_exchange_small(const __grid_constant__ EncodeArgs a, const __grid_constant__ SmallArgs r, const __grid_constant__ LevelTable lt,
                 const __grid_constant__ LevelTable lt_kept, const __grid_constant__ CodeTable ct, const __grid_constant__ PhiloxKey key,
                 const __grid_constant__ RoundTable rt) {
  extern __shared__ __align__(128) unsigned char s_raw[];
  __shared__ EncLut s_lut;
  __shared__ float s_lev[QGX_MAX_LEVELS], s_lev_kept[QGX_MAX_LEVELS];
  __shared__ double s_red[32];
  __shared__ uint32_t s_wtot[32];
  __shared__ unsigned int s_bucket;
  __shared__ float s_norm, s_norms[kSmallMaxWorkers], s_norms_kept[kSmallMaxWorkers];
  __shared__ unsigned long long s_prefix;
  __shared__ int s_skip;
  cg::cluster_group cluster = cg::this_cluster();
  const unsigned k = cluster.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
  const int K = a.K;
  float4* s_bin = reinterpret_cast<float4*>(s_raw);
  uint32_t* s_img = reinterpret_cast<uint32_t*>(s_raw + r.off_img);
  uint32_t* s_sym = reinterpret_cast<uint32_t*>(s_raw + r.off_sym);    // the decoded symbols, four per word
  uint16_t* s_tab = reinterpret_cast<uint16_t*>(s_raw + r.off_tab);    // the next maxlen + 1 bits -> symbol byte | bits << 8

  // which bucket: a ticket per cluster, so that the buckets a bucket looks back at are already under way
  unsigned ticket = 0;
  if (k == 0 && tid == 0) ticket = atomicAdd(a.ticket, 1u);
  asm volatile("barrier.cluster.arrive.aligned;" ::: "memory");
  const int rep = rt.key_shift - kKeyShiftMin, nbins = (int)((kKeyTop - kKeyBase) >> rt.key_shift) + 1;
  for (int i = tid; i < nbins; i += blockDim.x) s_bin[i] = __ldg(a.tables->bin_fix + (i << rep));
  for (int i = tid; i < (2 << ct.maxlen); i += blockDim.x) {
    const uint32_t e = __ldg(r.lut_len + 2 * i);                       // bits 0..4 bits consumed, 8..15 the symbol byte
    s_tab[i] = (uint16_t)(((e & 31u) << 8) | ((e >> 8) & 0xffu));
  }
  if (tid < 2 * QGX_MAX_LEVELS) s_lut.e[tid] = __ldg(a.tables->lut.e + tid);
  if (blockDim.x == kWarp) s_lut.e[QGX_MAX_LEVELS + tid] = __ldg(a.tables->lut.e + QGX_MAX_LEVELS + tid);   // a bucket of 128 has one warp
  if (tid < QGX_MAX_LEVELS) {
    s_lev[tid] = tid < lt.nlev ? lt.lev[tid] : 1.0f;
    s_lev_kept[tid] = tid < lt_kept.nlev ? lt_kept.lev[tid] : 0.0f;
  }
  for (uint32_t i = (uint32_t)tid; i < r.img_words; i += blockDim.x) s_img[i] = 0u;
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");          // the cluster's CTAs are there: their memory can be written
  if (k == 0 && tid == 0)
    for (int i = 0; i < K; ++i) *cluster.map_shared_rank(&s_bucket, i) = ticket;
  cluster.sync();
  const size_t b = a.b_first + s_bucket, lo = b * (size_t)a.bucket;
  const int len = (int)min((size_t)a.bucket, a.d - lo);

  // ---- load, norm ----
  BucketRegs<Q> x;
  const size_t ld = a.src.ld ? a.src.ld : a.d;
#pragma unroll
  for (int j = 0; j < Q; ++j) {
    const int e = ((warp * Q + j) * 32 + lane) * kQuad;
    float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
    if (a.vec_ok && e + kQuad <= len) {
      if (a.src.v) f = __ldg(reinterpret_cast<const float4*>(a.src.v + k * ld + lo + e));
      if (a.src.a) {
        const float4 av = __ldg(reinterpret_cast<const float4*>(a.src.a + lo + e));
        f = a.src.v ? dual_combine(av, f, a.src.mul) : av;
      }
    } else {
      if (e + 0 < len) f.x = dual_value(a.src, k, a.d, lo + e + 0);
      if (e + 1 < len) f.y = dual_value(a.src, k, a.d, lo + e + 1);
      if (e + 2 < len) f.z = dual_value(a.src, k, a.d, lo + e + 2);
      if (e + 3 < len) f.w = dual_value(a.src, k, a.d, lo + e + 3);
    }
    x.x[j] = f;
  }
  const float norm = bucket_norm_all<Q>(x, a.norm_type, s_red);
  const bool finite = (norm - norm) == 0.0f, live = finite && norm != 0.0f;
  const bool fast = rt.usable && norm > 7.9e-31f && norm < 1.2e30f;
  const float rn = fast ? __frcp_rn(norm) : 0.0f;
  const uint32_t thr = fast ? rt.thrfix : 0x10000u;
  if (tid == 0) {
    a.norms[(size_t)k * a.nb + b] = norm;
    if (!finite) latch_error(a.st, QGX_ERR_NONFINITE);
    s_img[0] = __float_as_uint(norm);
  }

  // ---- round and pack ----
  const uint32_t shift = (uint32_t)rt.key_shift - 4u, base = smem_addr(s_bin) - ((kKeyBase >> rt.key_shift) << 4);
  uint64_t qbits[Q];
  uint32_t qn[Q], qoff[Q];
#pragma unroll
  for (int j = 0; j < Q; ++j) {
    const int e = ((warp * Q + j) * 32 + lane) * kQuad;
    uint32_t sy = 0u;
    if (live && e < len) {
      const uint64_t ctr = a.quad_base + (uint64_t)((lo + (size_t)e) >> 2);
      const uint4 w4 = philox4x32_10((uint32_t)ctr, (uint32_t)(ctr >> 32), k, a.xid, key);
      const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
      const float v4[4] = {x.x[j].x, x.x[j].y, x.x[j].z, x.x[j].w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t dd = round_fixed_one(v4[i], w[i], rn, shift, base);
        uint32_t lv = (dd >> 16) & 0x1fu;
        if ((dd & 0xffffu) < thr) lv = level_exact_near(fabsf(v4[i]), norm, w[i] >> 8, (int)lv, smem_addr(s_lev), lt.nlev);
        sy |= symbol_of(v4[i], (int)lv) << (8 * i);
      }
    }
    pack_quad(sy, max(0, min(kQuad, len - e)), &s_lut, &qbits[j], &qn[j]);
  }
  const uint32_t nsub = (uint32_t)((len + G - 1) / G), hdr_bits = kNormBits + 16u * nsub;
  constexpr int kSeg = G / kQuad;                                      // lanes per sub-block: 8, 16 or 32
  uint32_t warp_bits = 0;
#pragma unroll
  for (int j = 0; j < Q; ++j) {
    const uint32_t incl = warp_incl_scan(qn[j], lane);
    const uint32_t before = __shfl_up_sync(0xffffffffu, incl, kSeg & 31);
    qoff[j] = warp_bits + incl - qn[j];
    warp_bits += __shfl_sync(0xffffffffu, incl, 31);
    if ((lane + 1) % kSeg == 0) {
      const uint32_t sb = (uint32_t)((warp * Q + j) * (32 / kSeg) + lane / kSeg);
      if (sb < nsub) reinterpret_cast<uint16_t*>(s_img)[2 + sb] = (uint16_t)(incl - (lane >= kSeg ? before : 0u));
    }
  }
  if (lane == 0) s_wtot[warp] = warp_bits;
  __syncthreads();
  const uint32_t wt = lane < nwarps ? s_wtot[lane] : 0u, wincl = warp_incl_scan(wt, lane);
  const uint32_t wbase = hdr_bits + __shfl_sync(0xffffffffu, wincl - wt, warp);
  const uint32_t nbits = hdr_bits + __shfl_sync(0xffffffffu, wincl, 31), nwords = (nbits + 31u) >> 5;
  const unsigned long long mine = (unsigned long long)nwords | ((unsigned long long)(32u * nwords - nbits) << kPadShift);
  unsigned long long* row = a.status + (size_t)k * a.nb;
  if (tid == 0) {
    st_status(row + b, kStAggregate | mine);
    a.bucket_bits[(size_t)k * a.nb + b] = nbits;
    s_norm = norm;
  }
#pragma unroll
  for (int j = 0; j < Q; ++j) put_bits(s_img, wbase + qoff[j], qbits[j], qn[j]);
  __syncthreads();                                                     // the image is complete

  // ---- decode (warps from the first on), the image's place in the stream (the last warp) ----
  bool bad = false;
  for (uint32_t s0 = (uint32_t)warp * 32u; s0 < nsub; s0 += (uint32_t)blockDim.x) {
    const uint32_t s = s0 + (uint32_t)lane;
    auto field = [&](uint32_t i) { return (uint32_t) reinterpret_cast<const uint16_t*>(s_img)[2 + i]; };
    uint32_t before = 0;
    for (uint32_t i = (uint32_t)lane; i < s0; i += 32u) before += field(i);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
    const uint32_t L = s < nsub ? field(s) : 0u;
    const uint32_t start = hdr_bits + before + warp_incl_scan(L, lane) - L;
    if (s < nsub) {
      const int first = (int)s * G, count = min(G, len - first);
      uint32_t next = start >> 5, left = L;
      uint64_t buf = (((uint64_t)s_img[next + 1] << 32) | s_img[next]) >> (start & 31u);
      int avail = 64 - (int)(start & 31u);
      next += 2;
      const uint32_t mask = (2u << ct.maxlen) - 1u;
      for (int i = 0; i < count; i += kQuad) {
        uint32_t word = 0;
#pragma unroll
        for (int q = 0; q < kQuad; ++q) {
          if ((q & 1) == 0 && avail <= 32) {                           // two symbols use at most 26 bits
            buf |= (uint64_t)s_img[min(next, r.img_words - 1u)] << avail;
            avail += 32;
            ++next;
          }
          if (i + q < count) {
            const uint32_t e = s_tab[(uint32_t)buf & mask], n = e >> 8;
            buf >>= n;
            avail -= (int)n;
            left -= n;
            bad = bad || (e & 0x40u) != 0u;                            // an index that no codeword starts like
            word |= (e & 0xffu) << (8 * q);
          }
        }
        s_sym[(first + i) >> 2] = word;
      }
      bad = bad || left != 0u;                                         // every sub-block uses exactly its length
    }
  }
  if (warp == nwarps - 1) {
    bool timed_out = false;
    const unsigned long long excl = lookback_prefix(row, (long long)b, lane, a.spin_limit, &timed_out);
    if (lane == 0) {
      const unsigned long long incl = excl + mine, words = incl & ((1ull << kPadShift) - 1ull), at = excl & ((1ull << kPadShift) - 1ull);
      st_status(row + b, kStPrefix | incl);
      const bool over = words > (unsigned long long)a.cap_words;
      if (timed_out) latch_error(a.st, QGX_ERR_TIMEOUT);
      else if (over) latch_error(a.st, QGX_ERR_CAPACITY);
      a.offsets[(size_t)k * a.nb + b] = (uint32_t)min(at, 0xffffffffull);
      if (b + 1 == a.nb) {
        const unsigned long long bits = 32ull * words - (incl >> kPadShift);
        a.total_bits[k] = bits;
        if (r.total_out) r.total_out[k] = bits;
      }
      s_prefix = at;
      s_skip = timed_out || over ? 1 : 0;
    }
  }
  cluster.sync();                                                      // every worker's symbols are there
  if (!s_skip) {
    uint32_t* dst = a.stream + (size_t)k * a.cap_words + s_prefix;
    for (uint32_t i = (uint32_t)tid; i < nwords; i += blockDim.x) dst[i] = s_img[i];
  }

  // ---- ordered sums of this CTA's share of the quads, kept symbols, squared differences, state update ----
  if (tid < K) {
    s_norms[tid] = *cluster.map_shared_rank(&s_norm, tid);
    s_norms_kept[tid] = r.norms_prev ? r.norms_prev[(size_t)tid * a.nb + b] : 0.0f;
  }
  __syncthreads();
  const float Kf = (float)K, gam = r.update == 1 ? (float)r.scalars[1] : 1.0f;
  const int quads = (len + kQuad - 1) / kQuad;
  const size_t spb = (size_t)a.bucket / G;
  double sq = 0.0;
  for (int q = (int)k * blockDim.x + tid; q < quads; q += K * (int)blockDim.x) {
    const int e = q * kQuad, nv = min(kQuad, len - e), i = e % G;
    const size_t gs = b * spb + (size_t)(e / G);
    const size_t sat = (gs >> 5) * (size_t)(32 * G) + (size_t)(i >> 2) * 128 + (size_t)(gs & 31) * 4;   // see DecodeArgs::sym_out
    float acc[kQuad] = {0.f, 0.f, 0.f, 0.f};
    for (int kk = 0; kk < K; ++kk) {
      const uint32_t word = *cluster.map_shared_rank(s_sym + q, kk);
      const float nrm = s_norms[kk];
      const uint32_t was = r.sym_prev ? *reinterpret_cast<const uint32_t*>(r.sym_prev + (size_t)kk * r.sym_ld + sat) : 0u;
#pragma unroll
      for (int c = 0; c < kQuad; ++c) {
        const float val = dequantize_symbol((word >> (8 * c)) & 0xffu, nrm, s_lev);
        acc[c] = __fadd_rn(acc[c], val);
        if (c < nv && r.sym_prev) {
          const float dlt = __fsub_rn(dequantize_symbol((was >> (8 * c)) & 0xffu, s_norms_kept[kk], s_lev_kept), val);
          sq = fma((double)dlt, (double)dlt, sq);
        } else if (c < nv && r.square) {
          sq = fma((double)val, (double)val, sq);
        }
      }
      if (r.sym_out) *reinterpret_cast<uint32_t*>(r.sym_out + (size_t)kk * r.sym_ld + sat) = word;
    }
#pragma unroll
    for (int c = 0; c < kQuad; ++c) {
      if (c < nv) {
        const size_t at = lo + (size_t)(e + c);
        const float m = __fdiv_rn(acc[c], Kf);
        bad = bad || m != m;
        r.mean[at] = m;
        if (r.update == 1) r.xout[at] = __fsub_rn(r.xin[at], __fmul_rn(gam, m));
        if (r.update == 2) r.xout[at] = __fsub_rn(r.xin[at], m);
      }
    }
  }
  if (r.sym_prev || r.square) {
    sq = warp_sum(sq);
    if (lane == 0 && sq != 0.0) atomicAdd(r.sum_sq, sq);
  }
  if (bad) latch_error(a.st, QGX_ERR_CORRUPT);
  cluster.sync();                                                      // nobody leaves while its symbols are being read

  // the last cluster leaves the scan's words as it found them: zero
  if (k == 0) {
    __shared__ bool s_last;
    if (tid == 0) {
      __threadfence();
      s_last = atomicAdd(a.ticket + 1, 1u) == (unsigned)(a.nb - a.b_first - 1);
    }
    __syncthreads();
    if (s_last) {
      for (size_t i = (size_t)tid; i < (size_t)K * a.nb; i += blockDim.x) a.status[i] = 0ull;
      if (tid == 0) { a.ticket[0] = 0u; a.ticket[1] = 0u; }
    }
  }
}

// Whether `workers` CTAs of this shape fit into a cluster (more than eight: not on every part), asked once per shape.
static bool cluster_fits(const void* fn, int device, int workers, int threads, size_t smem) {
  if (workers <= 8) return true;
  struct Seen { const void* fn; int device, workers, threads; size_t smem; bool fits; };
  static std::vector<Seen> seen;
  static std::mutex guard;
  std::lock_guard<std::mutex> lock(guard);
  for (const Seen& x : seen)
    if (x.fn == fn && x.device == device && x.workers == workers && x.threads == threads && x.smem == smem) return x.fits;
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)workers;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)workers);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int clusters = 0;
  const bool fits = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                    cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg) == cudaSuccess && clusters >= 4;
  if (!fits) cudaGetLastError();
  seen.push_back(Seen{fn, device, workers, threads, smem, fits});
  return fits;
}

// One bucket per CTA, so the launch takes ever more turns as the vector grows, while the large kernels' time hardly moves
// until theirs are full.  Measured (us, this way against the other): 4 x 10^4 coordinates of bucket 1024 12.3 : 28.7,
// 4 x 10^5 16.7 : 28.6, 8 x 10^5 22.1 : 31.8, 1.2 x 10^6 32.4 : 31.7; of bucket 4096 1.2 x 10^6 24.5 : 31.3, 2.4 x 10^6 38.5 : 38.8;
// of bucket 16384 1.6 x 10^6 24.6 : 34.9.
bool small_exchange_fits(const qgx_ctx* c, int K, size_t nb, int bucket) {
  if (K > kSmallMaxWorkers || bucket < 128 || bucket % 128 != 0 || nb > 65536) return false;
  return nb * (size_t)K * (size_t)bucket <= (size_t)c->all_sms * (bucket >= 4096 ? 12288 : 7168);
}

qgx_status launch_exchange_small(qgx_ctx* c, const EncodeArgs& ea, SmallArgs r, const LevelTable& lt, const LevelTable& lt_kept,
                                 const CodeTable& ct, const PhiloxKey& key, const RoundTable& rt) {
  const int Q = ea.bucket <= 2048 ? 1 : (ea.bucket <= 4096 ? 2 : 4);
  const int threads = ((ea.bucket / kQuad + Q - 1) / Q + 31) / 32 * 32;
  const size_t nbins = ((kKeyTop - kKeyBase) >> rt.key_shift) + 1;
  r.img_words = (uint32_t)(((size_t)ea.bucket * (ct.maxlen + 1) + 16u * (ea.bucket / ct.G + 1) + kNormBits + 31u) / 32u + 4u);
  r.off_img = (uint32_t)((nbins * sizeof(float4) + 127) & ~(size_t)127);
  r.off_sym = (uint32_t)((r.off_img + r.img_words * 4u + 15u) & ~15u);
  r.off_tab = (uint32_t)((r.off_sym + (uint32_t)ea.bucket + 15u) & ~15u);
  const size_t smem = r.off_tab + (sizeof(uint16_t) << (ct.maxlen + 1));
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)ea.K;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)((ea.nb - ea.b_first) * (size_t)ea.K));
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = c->stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t err = cudaSuccess;
#define QGX_SMALL(QQ, GG)                                                                    \
  do {                                                                                       \
    allow_max_dynamic_smem((const void*)k_exchange_small<QQ, GG>, c->device);                \
    if (!cluster_fits((const void*)k_exchange_small<QQ, GG>, c->device, ea.K, threads, smem)) return QGX_ERR_TOO_LARGE; \
    err = cudaLaunchKernelEx(&cfg, k_exchange_small<QQ, GG>, ea, r, lt, lt_kept, ct, key, rt); \
  } while (0)
#define QGX_SMALL_G(QQ)                          \
  do {                                           \
    if (ct.G == 32) QGX_SMALL(QQ, 32);           \
    else if (ct.G == 64) QGX_SMALL(QQ, 64);      \
    else QGX_SMALL(QQ, 128);                     \
  } while (0)
  if (Q == 1) QGX_SMALL_G(1);
  else if (Q == 2) QGX_SMALL_G(2);
  else QGX_SMALL_G(4);
#undef QGX_SMALL_G
#undef QGX_SMALL
  count_launch(c);
  return cuda_status(err != cudaSuccess ? err : cudaGetLastError());
}

}  // namespace qgx
