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

// the symbol that `bits` (the stream's next ones, first at bit 0) start with; where there is none, one bit is taken
struct NextSymbol { uint32_t level, bits; bool negative, known; };
__device__ __forceinline__ NextSymbol next_symbol(uint32_t bits, const CodeTable& ct) {
  NextSymbol s{0u, 1u, false, false};
  for (int j = 0; j < ct.nlev; ++j) {
    const uint32_t L = ct.len[j];
    if ((bits & ((1u << L) - 1u)) != ct.rev[j]) continue;
    s.known = true;
    s.level = (uint32_t)j;
    s.negative = j != 0 && ((bits >> L) & 1u);
    s.bits = L + (j != 0 ? 1u : 0u);
  }
  return s;
}
// entry i of the pair table; symbol(s) = the byte that stands for s
template <class F>
__device__ __forceinline__ uint32_t pair_entry_of(uint32_t i, const CodeTable& ct, F symbol) {
  const NextSymbol a = next_symbol(i, ct), b = next_symbol(i >> a.bits, ct);
  // the second symbol counts where the index holds all its bits (or all that could tell that there is none)
  const bool both = a.bits + (b.known ? b.bits : (uint32_t)ct.maxlen + 1u) <= (uint32_t)pair_bits(ct.maxlen);
  return (both ? (a.bits + b.bits) | (symbol(b) << 24) : a.bits | kPairEscape) | (a.bits << 8) | (symbol(a) << 16);
}

// ---- the walk ---------------------------------------------------------------------------------
// Words that a lane may read past the one that holds its sub-block's first bit: G symbols of at most 13 bits, the partial
// first word and the word fetched ahead.
template <int G>
struct WalkReach { static constexpr int kWords = (G * 13) / 32 + 4; };

// Position in a stream: the lowest five bits of `pos` are the place in w0, bit 5 says whether that has been left; what is above
// is junk (entries of the pair table are added as they are).  The two bits before the next symbol lie in the window, too, so
// that an index comes out as a byte offset.  SH: the words are in shared memory (32-bit addresses).
template <bool SH> struct WordAt { using Addr = uint32_t; };
template <> struct WordAt<false> { using Addr = const uint32_t*; };
template <bool SH>
struct Walk {
  typename WordAt<SH>::Addr next;        // of the word after w1
  uint32_t w0, w1, pos, old;             // old: pos when w0 was last checked
  static __device__ __forceinline__ uint32_t word(uint32_t a) { return lds32(a); }
  static __device__ __forceinline__ uint32_t word(const uint32_t* a) { return *a; }
  static __device__ __forceinline__ uint32_t step(uint32_t a, int words) { return a + 4u * (uint32_t)words; }
  static __device__ __forceinline__ const uint32_t* step(const uint32_t* a, int words) { return a + words; }
  static __device__ __forceinline__ uint32_t words_from(uint32_t a, uint32_t b) { return (a - b) >> 2; }
  static __device__ __forceinline__ uint32_t words_from(const uint32_t* a, const uint32_t* b) { return (uint32_t)(a - b); }
  // p = the word that holds the bit two before the first, sh = that bit's place in it
  __device__ __forceinline__ void open(typename WordAt<SH>::Addr p, uint32_t sh) {
    w0 = word(p);
    w1 = word(step(p, 1));
    next = step(p, 2);
    pos = old = sh;
  }
  __device__ __forceinline__ uint32_t window() const { return __funnelshift_r(w0, w1, pos); }
  // after at most 32 bits: moves on a word where the position has left w0
  __device__ __forceinline__ void settle() {
    if ((pos ^ old) & 32u) {
      w0 = w1;
      w1 = word(next);
      next = step(next, 1);
    }
    old = pos;
  }
  // bits taken since open(p, sh)
  __device__ __forceinline__ uint32_t taken(typename WordAt<SH>::Addr p, uint32_t sh) const { return 32u * (words_from(next, p) - 2u) + (pos & 31u) - sh; }
};

struct WalkTable {
  uint32_t pair;                         // shared address of the pair table, its mask for byte offsets
  uint32_t mask;
  __device__ __forceinline__ uint32_t entry(uint32_t window) const { return lds_table32(pair + (window & mask)); }
};
__device__ __forceinline__ uint32_t first_bits(uint32_t entry) { return (entry >> 8) & 31u; }

// The next four symbols, a byte each.  A window holds 30 bits to come, so two entries of at most 13; where an entry stands for one
// symbol only the second is looked up on its own, its bits taken at once and the entry's own cleared.
template <class W>
__device__ __forceinline__ uint32_t walk_four(W& w, const WalkTable& t) {
  uint32_t win = w.window();
  uint32_t e = t.entry(win);
  if (e & kPairEscape) {
    const uint32_t f = t.entry(__funnelshift_r(win, 0u, e));
    w.pos += (e & 31u) + first_bits(f);
    w.settle();
    win = w.window();
    e = prmt(prmt(e, f, 0x6200u), 0u, 0x3244u);                        // the two symbols, nothing taken
  }
  w.pos += e;
  win = __funnelshift_r(win, 0u, e);
  uint32_t f = t.entry(win);
  if (f & kPairEscape) {
    w.settle();
    w.pos += f & 31u;
    w.settle();
    const uint32_t g = t.entry(w.window());
    w.pos += first_bits(g);
    f = prmt(prmt(f, g, 0x6200u), 0u, 0x3244u);
  }
  w.pos += f;
  w.settle();
  return prmt(e, f, 0x7632u);
}
template <class W>
__device__ __forceinline__ uint32_t walk_one(W& w, const WalkTable& t) {
  const uint32_t e = t.entry(w.window());
  w.pos += first_bits(e);
  w.settle();
  return (e >> 16) & 0xffu;
}

// G symbols of one sub-block to row[0 .. G / 4) (shared address), four to a word
template <int G, bool SH>
__device__ __forceinline__ void walk_whole(Walk<SH>& w, uint32_t row, const WalkTable& t) {
#pragma unroll
  for (int i = 0; i < G; i += 4) sts32(row + (uint32_t)i, walk_four(w, t));
}
// the same, one symbol at a time, for `count` symbols (the vector's last sub-block)
template <bool SH>
__device__ __forceinline__ void walk_some(Walk<SH>& w, int count, uint32_t row, const WalkTable& t) {
#pragma unroll 1
  for (int i = 0; i < count; i += 4) {
    uint32_t word = 0;
#pragma unroll 1
    for (int q = 0; q < 4 && i + q < count; ++q) word |= walk_one(w, t) << (8 * q);
    sts32(row + (uint32_t)i, word);
  }
}

// ---- rows of sub-blocks -----------------------------------------------------------------------
// Row r of a worker: its sub-blocks 32 r .. 32 r + 31, of one bucket or of several in a row.
struct RowShape {
  uint32_t rows;                         // per worker
  uint32_t spb, spb_mul, spb_shift;      // sub-blocks per bucket; n / spb = (n * spb_mul >> 32) >> spb_shift
  uint32_t whole_subs, last_count;       // sub-blocks of G coordinates, and the coordinates of the one after them
  uint32_t hdr_bits, hdr_bits_last;      // of a bucket, of the last bucket
};
// for buckets of whole sub-blocks; false where there are too many
inline bool make_row_shape(size_t d, int bucket, int G, size_t nb, RowShape* r) {
  const size_t subs = (d + (size_t)G - 1) / (size_t)G;
  if (subs >= (1ull << 31)) return false;
  r->rows = (uint32_t)((subs + 31) / 32);
  // n / spb for n < 2^31: with 2^(L - 1) < spb <= 2^L the multiplier, 2^(31 + L) / spb rounded up, is below 2^32 and off by at
  // most spb / 2^(31 + L) of itself
  r->spb = (uint32_t)(bucket / G);
  int log2up = 1;
  while ((1u << log2up) < r->spb) ++log2up;
  r->spb_mul = (uint32_t)((1ull << (31 + log2up)) / r->spb + 1u);
  r->spb_shift = (uint32_t)log2up - 1u;
  r->whole_subs = (uint32_t)(d / (size_t)G);
  r->last_count = (uint32_t)(d % (size_t)G);
  r->hdr_bits = (uint32_t)kNormBits + 16u * r->spb;
  r->hdr_bits_last = (uint32_t)kNormBits + 16u * (uint32_t)(subs - (nb - 1) * (size_t)r->spb);
  return true;
}

struct RowPlace {
  uint32_t b, s;                         // the lane's bucket, the sub-block's number in it
  int count;                             // its coordinates, 0 beyond the end
};
template <int G>
__device__ __forceinline__ RowPlace row_place(const RowShape& h, uint32_t row, int lane) {
  const uint32_t gs = row * 32u + (uint32_t)lane;
  RowPlace p;
  p.count = gs < h.whole_subs ? G : (gs == h.whole_subs ? (int)h.last_count : 0);
  const uint32_t in = p.count > 0 ? gs : 0u;                           // beyond the end: the first bucket's first, to have some
  p.b = __umulhi(in, h.spb_mul) >> h.spb_shift;
  p.s = in - p.b * h.spb;
  return p;
}
template <int G>
__host__ __device__ constexpr uint32_t sym_row_bytes() { return 32u * (uint32_t)(G / 4 + 1) * 4u; }   // a word more than needed: no bank conflicts
// words that a row's sub-blocks and the headers between them can take
__host__ __device__ constexpr uint32_t row_words_worst(int G, int maxlen) { return (uint32_t)(G * (maxlen + 1) + 3 * 32 + (G * 13) / 32 + 12) & ~3u; }

}  // namespace qgx
