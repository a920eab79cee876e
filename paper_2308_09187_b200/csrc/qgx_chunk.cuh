// Chunks: 1024 coordinates of a bucket whose codewords a warp writes, 32 consecutive coordinates per lane, every lane's bits
// first as a stream of its own in shared memory (the chunk's image) and then, shifted, where they belong.
#pragma once

#include "qgx_common.cuh"

namespace qgx {

constexpr int kLaneCoords = 32;          // coordinates per lane
__host__ __device__ constexpr int pipe_lane_stride(int maxlen) { return (maxlen + 1) | 1; }   // words per lane, odd: no bank conflicts

// Stream bits of a lane as they are produced: a 64-bit window that new bits enter at the top (two funnel shifts, no masks);
// the oldest 32 go to the lane's words in shared memory once they are there.
struct LaneBits {
  uint32_t lo, hi;
  int pos;                                               // 64 - bits waiting in the window
  uint32_t wa;                                           // shared address of the next word
  __device__ __forceinline__ void open(uint32_t addr) { lo = hi = 0u; pos = 64; wa = addr; }
  // the low n bits of e (n <= 26, the entry's upper 6 bits; fewer than 32 bits are waiting)
  __device__ __forceinline__ void put(uint32_t e) {
    const uint32_t n = e >> 26;
    lo = __funnelshift_r(lo, hi, n);
    hi = __funnelshift_r(hi, e, n);
    pos -= (int)n;
    if (pos <= 32) {
      sts32(wa, __funnelshift_rc(lo, hi, (uint32_t)pos));
      wa += 4u;
      pos += 32;
    }
  }
  // stores what is waiting; the bits put since open(addr)
  __device__ __forceinline__ uint32_t close(uint32_t addr) {
    if (pos < 64) sts32(wa, hi >> ((uint32_t)pos - 32u));
    return 8u * (wa - addr) + (uint32_t)(64 - pos);
  }
};

// The chunk's part of its bucket.  dst: the bucket's first word; bit: where the chunk's bits start in the bucket; nbits: of the
// whole bucket; ib: the chunk's number in the bucket; nsub: the bucket's sub-blocks (0: none, G does not matter); cnt: bits per
// lane, of this chunk and the ones after it; last: the last 32 bits of this chunk, those of the chunk before it one earlier;
// img: shared address of this lane's words.
template <int G>
__device__ __forceinline__ void place_chunk(uint32_t* dst, uint32_t bit, uint32_t nbits, int ib, uint32_t nsub, float norm, const uint16_t* cnt,
                                            const uint32_t* last, uint32_t img, int lane) {
  const uint32_t cnt_sa = smem_addr(cnt);
  // The header's words of this chunk: two sub-blocks each, G / 32 lane counts per sub-block.
  constexpr uint32_t kWords = 1024 / G / 2;                            // 16, 8 or 4
  if ((uint32_t)lane < kWords && (uint32_t)ib * kWords + (uint32_t)lane < nsub / 2u) {
    uint32_t h;
    if (G == 32) {
      h = lds32(cnt_sa + 4u * (uint32_t)lane);
    } else {
      uint32_t f0 = 0, f1 = 0;
#pragma unroll
      for (int j = 0; j < G / 64; ++j) {
        const uint32_t c0 = lds32(cnt_sa + (uint32_t)lane * (G / 8) + 4u * j), c1 = lds32(cnt_sa + (uint32_t)lane * (G / 8) + (G / 16) + 4u * j);
        f0 += (c0 & 0xffffu) + (c0 >> 16);
        f1 += (c1 & 0xffffu) + (c1 >> 16);
      }
      h = f0 | (f1 << 16);
    }
    dst[1u + (uint32_t)ib * kWords + (uint32_t)lane] = h;
  }
  if (ib == 0 && lane == 0) dst[0] = __float_as_uint(norm);
  const uint32_t n_l = cnt[lane];
  const uint32_t p = bit + warp_incl_scan(n_l, lane) - n_l, sh = p & 31u, nw = ((p + n_l) >> 5) - (p >> 5);
  uint32_t* out = dst + (p >> 5);
  // Word j of the lane's part of the stream takes the end of its bits' word j - 1 and the beginning of word j; words
  // 0 .. nw - 1 end inside its bits, word nw is for the lane after it (past the lane's words the reads run into its
  // neighbour's: those bits are masked off).
  const uint32_t most = __reduce_max_sync(0xffffffffu, nw);
  uint32_t prev = lds32(img), tail = 0;
  const uint32_t first = prev << sh;
#pragma unroll
  for (uint32_t j = 1; j <= (uint32_t)QGX_MAX_CODE_LEN + 2u; ++j) {
    if (j > most) break;
    const uint32_t cur = lds32(img + 4u * j), x = __funnelshift_l(prev, cur, sh);
    if (j < nw) out[j] = x;
    if (j == nw) tail = x;
    prev = cur;
  }
  const uint32_t over = (p + n_l) & 31u, mask = (1u << over) - 1u;
  tail &= mask;
  uint32_t before = __shfl_up_sync(0xffffffffu, tail, 1);
  if (lane == 0) {
    before = 0;
    if (sh != 0u) {
      if (ib != 0) {
        before = last[-1] >> (32u - sh);                               // the last bits of the chunk before
      } else {                                                         // an odd number of sub-blocks: the last length shares a word
#pragma unroll
        for (int j = 0; j < G / kLaneCoords; ++j) before += cnt[(nsub - 1u) * (G / kLaneCoords) + j];
      }
    }
  }
  if (nw > 0u) out[0] = first | before;
  // the bucket's last word, when it is not whole
  if (n_l > 0u && p + n_l == nbits && over != 0u) out[nw] = nw > 0u ? tail : ((first & mask) | before);
}

}  // namespace qgx
