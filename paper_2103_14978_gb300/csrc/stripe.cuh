// Striped form of the per-pair filter's bit vectors: position p lives in word
// p mod S, row p / S.
//
// In the linear layout (filter.cuh, position p in word p / 32) a shift by one
// base moves bits inside every word, a funnel shift per word.  Striped, it
// renames the words: word w of the shifted vector is word w - 1, and only the
// word that wraps (S - 1 to 0) moves by a row.  A mask's dilation and erosion
// then take two one-row shifts each for the whole vector instead of two per
// word, the read's +k and -k copies one per plane and step instead of W, and
// with S a multiple of 4 a 4-base window of the run count (Sec. 2.1) is one
// row of four words.  What is left per mask and word are 3-input logic ops: 2
// for the difference, 1 for the dilation, 2 for the erosion, the vacated
// positions and the AND.
//
// Where a row sits in its word:
//   S even (4, 8)   row r at bit r; a row shift is a shift by one.  Linear
//                   words become stripes by byte permutes and bit exchanges,
//                   about eight operations per word.
//   S odd (3, 5, 11)  row r at bit (S r) mod 32: position p is at bit
//                   (p - p mod S) mod 32 of word p mod S, so that stripe w is
//                   the linear words' bits with (position mod S) = w, merged
//                   by S - 1 bit selects, rotated by w.  A row shift is a
//                   rotation by S; what leaves at one end enters at the other
//                   and lies outside the read (m <= 32 S - 4).
//
// S is the smallest of these that holds the read: 32 S positions, 2 (even) or
// 4 (odd) of them to spare.  Every step is bound by the integer ALU pipe (81-88% busy):
// logic ops and right shifts run there at 64 lanes per clock and SM, left
// shifts and additions partly on the multiply-add pipe, which is why the
// vectors below move up (to higher positions) wherever there is a choice.
#pragma once

#include "gk_internal.cuh"

namespace gk {

__host__ __device__ __forceinline__ uint32_t st_prmt(uint32_t x, uint32_t y, uint32_t s) {
#ifdef __CUDA_ARCH__
  return __byte_perm(x, y, s);
#else
  const uint64_t v = ((uint64_t)y << 32) | x;
  uint32_t r = 0;
  for (int i = 0; i < 4; ++i) r |= (uint32_t)((v >> (8 * ((s >> (4 * i)) & 7))) & 0xFFu) << (8 * i);
  return r;
#endif
}

__host__ __device__ __forceinline__ uint32_t st_popc(uint32_t x) {
#ifdef __CUDA_ARCH__
  return (uint32_t)__popc(x);
#else
  return (uint32_t)__builtin_popcount(x);
#endif
}

__host__ __device__ __forceinline__ uint32_t st_brev(uint32_t x) {
#ifdef __CUDA_ARCH__
  return __brev(x);
#else
  uint32_t r = 0;
  for (int i = 0; i < 32; ++i) r |= ((x >> i) & 1u) << (31 - i);
  return r;
#endif
}

// The low 32 bits of hi:lo >> s, s in 0..32.
__host__ __device__ __forceinline__ uint32_t st_shr64(uint32_t lo, uint32_t hi, uint32_t s) {
#ifdef __CUDA_ARCH__
  return __funnelshift_rc(lo, hi, s);
#else
  return (uint32_t)((((uint64_t)hi << 32) | lo) >> s);
#endif
}

// The 3-input logic function with truth table LUT (a = 0xF0, b = 0xCC, c =
// 0xAA).
template <uint32_t LUT>
__host__ __device__ __forceinline__ uint32_t lop3(uint32_t a, uint32_t b, uint32_t c) {
#ifdef __CUDA_ARCH__
  uint32_t r;
  asm("lop3.b32 %0, %1, %2, %3, %4;" : "=r"(r) : "r"(a), "r"(b), "r"(c), "n"(LUT));
  return r;
#else
  uint32_t r = 0;
  for (int i = 0; i < 8; ++i)
    if ((LUT >> i) & 1u) r |= ((i & 4) ? a : ~a) & ((i & 2) ? b : ~b) & ((i & 1) ? c : ~c);
  return r;
#endif
}

// Exchanges a word-index bit with bit `log2 s` of the bit index between words
// a (index bit 0) and b (index bit 1); m has 1s where that bit of the bit
// index is 0.
__host__ __device__ __forceinline__ void st_swap(uint32_t &a, uint32_t &b, uint32_t m, int s) {
  const uint32_t x = (a & m) | ((b << s) & ~m);
  b = ((a >> s) & m) | (b & ~m);
  a = x;
}

// Byte j of word i becomes byte i of word j.
__host__ __device__ __forceinline__ void st_bytes(uint32_t &a, uint32_t &b, uint32_t &c, uint32_t &d) {
  const uint32_t p = st_prmt(a, b, 0x5140), q = st_prmt(a, b, 0x7362);
  const uint32_t r = st_prmt(c, d, 0x5140), t = st_prmt(c, d, 0x7362);
  a = st_prmt(p, r, 0x5410);
  b = st_prmt(p, r, 0x7632);
  c = st_prmt(q, t, 0x5410);
  d = st_prmt(q, t, 0x7632);
}

// Linear words (position p in word p / 32, bit p mod 32) to stripes, about
// eight operations per word: index bits change places by byte permutes and by
// exchanges between words.  Linear word index j, bit index b4..b0:
//   S = 4: p = 32j + b, stripe (b1 b0), row (j1 j0 b4 b3 b2)
//   S = 8: stripe (b2 b1 b0), row (j2 j1 j0 b4 b3)
template <int S>
__host__ __device__ __forceinline__ void stripe_words(uint32_t (&x)[S]) {
  static_assert(S == 4 || S == 8, "stripes");
  if constexpr (S == 4) {
    st_bytes(x[0], x[1], x[2], x[3]);  // words (b4 b3), bits (j1 j0 b2 b1 b0)
    st_swap(x[0], x[2], 0x0F0F0F0Fu, 4);  // words (b2 b3), bits (j1 j0 b4 b1 b0)
    st_swap(x[1], x[3], 0x0F0F0F0Fu, 4);
    st_swap(x[0], x[1], 0x33333333u, 2);  // words (b2 b1), bits (j1 j0 b4 b3 b0)
    st_swap(x[2], x[3], 0x33333333u, 2);
    st_swap(x[0], x[2], 0x55555555u, 1);  // words (b0 b1), bits (j1 j0 b4 b3 b2)
    st_swap(x[1], x[3], 0x55555555u, 1);
    const uint32_t t = x[1];  // words in the order (b1 b0)
    x[1] = x[2];
    x[2] = t;
  } else {
    st_bytes(x[0], x[2], x[4], x[6]);  // words (b4 b3 j0), bits (j2 j1 b2 b1 b0)
    st_bytes(x[1], x[3], x[5], x[7]);
#pragma unroll
    for (int i = 0; i < 8; i += 2) st_swap(x[i], x[i + 1], 0x0F0F0F0Fu, 4);  // words (b4 b3 b2)
#pragma unroll
    for (int i = 0; i < 4; ++i) st_swap(x[i], x[i + 4], 0x33333333u, 2);  // words (b1 b3 b2)
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (!(i & 2)) st_swap(x[i], x[i + 2], 0x55555555u, 1);  // words (b1 b0 b2)
    uint32_t y[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) y[((i & 1) << 2) | (i >> 1)] = x[i];  // (b2 b1 b0)
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = y[i];
  }
}

// One row (S positions) up or down in a word: the step of the word that wraps
// when a vector moves by one base.
template <int S>
__host__ __device__ __forceinline__ uint32_t row_up(uint32_t x) {
  if constexpr (S & 1) return (x << S) | (x >> (32 - S));
  return x << 1;
}
template <int S>
__host__ __device__ __forceinline__ uint32_t row_down(uint32_t x) {
  if constexpr (S & 1) return (x >> S) | (x << (32 - S));
  return x >> 1;
}
template <int S>
__host__ __device__ __forceinline__ constexpr uint32_t row_bit(int r) {
  return 1u << ((S & 1) ? (S * r) & 31 : r & 31);
}

// Bits b of linear word j whose position 32 j + b is in stripe w.
template <int S>
__host__ __device__ constexpr uint32_t crt_mask(int j, int w) {
  uint32_t x = 0;
  for (int b = 0; b < 32; ++b)
    if ((32 * j + b) % S == w) x |= 1u << b;
  return x;
}

// The low W linear words (zero past the read) as S stripes.
template <int W, int S>
__host__ __device__ __forceinline__ void stripe_linear(const uint32_t (&x)[W], uint32_t (&y)[S]) {
  static_assert(W <= S, "stripes hold every linear word");
  if constexpr (S & 1) {
#pragma unroll
    for (int w = 0; w < S; ++w) {
      uint32_t v = W == S ? x[0] : x[0] & crt_mask<S>(0, w);
#pragma unroll
      for (int j = 1; j < W; ++j) v = (v & ~crt_mask<S>(j, w)) | (x[j] & crt_mask<S>(j, w));
      y[w] = w == 0 ? v : ((v >> w) | (v << ((32 - w) & 31)));
    }
  } else {
#pragma unroll
    for (int i = 0; i < S; ++i) y[i] = i < W ? x[i < W ? i : 0] : 0u;
    stripe_words<S>(y);
  }
}

// Longest read S stripes hold: two indices more than positions and, S odd, two
// rows' worth of zeros against the rotation.
template <int S>
__host__ __device__ constexpr uint32_t stripe_limit() {
  return (S & 1) ? 32u * S - 4u : 32u * S - 2u;
}

// Positions below m of every word, 32 (W - 1) < m <= 32 W + 2.
template <int W, int S>
__host__ __device__ __forceinline__ void stripe_masks(uint32_t m, uint32_t (&x)[S]) {
  if constexpr (S & 1) {
    // Linear mask words: all 1s below W - 1, then the last one or two.
    const uint32_t n = m - 32u * (W - 1);
    const uint32_t l0 = n >= 32 ? 0xffffffffu : (1u << n) - 1u, l1 = n > 32 ? (1u << (n - 32)) - 1u : 0u;
#pragma unroll
    for (int w = 0; w < S; ++w) {
      uint32_t c = 0;
#pragma unroll
      for (int j = 0; j < W - 1; ++j) c |= crt_mask<S>(j, w);
      const uint32_t v = c | (l0 & crt_mask<S>(W - 1, w)) | (W < S ? l1 & crt_mask<S>(W, w) : 0u);
      x[w] = w == 0 ? v : ((v >> w) | (v << ((32 - w) & 31)));
    }
  } else {
    const uint32_t a = m / S, b = m % S;
#pragma unroll
    for (int w = 0; w < S; ++w) {
      const uint32_t n = a + ((uint32_t)w < b ? 1u : 0u);
      x[w] = n >= 32 ? 0xffffffffu : (1u << n) - 1u;
    }
  }
}

// Position p <- d[p] | d[p-1] | d[p-2]: the dilation of a mask, moved up by one
// position, so that both row shifts go up.
template <int S>
__host__ __device__ __forceinline__ void stripe_or3(const uint32_t (&d)[S], uint32_t (&x)[S]) {
  const uint32_t a = row_up<S>(d[S - 1]), b = row_up<S>(d[S - 2]);
  x[0] = lop3<0xFE>(d[0], a, b);
  x[1] = lop3<0xFE>(d[1], d[0], a);
#pragma unroll
  for (int w = 2; w < S; ++w) x[w] = lop3<0xFE>(d[w], d[w - 1], d[w - 2]);
}

// Position p <- x[p] & x[p-1] & x[p-2]: the erosion, moved up by one more.
template <int S>
__host__ __device__ __forceinline__ void stripe_and3(const uint32_t (&x)[S], uint32_t (&y)[S]) {
  const uint32_t a = row_up<S>(x[S - 1]), b = row_up<S>(x[S - 2]);
  y[0] = lop3<0x80>(x[0], a, b);
  y[1] = lop3<0x80>(x[1], x[0], a);
#pragma unroll
  for (int w = 2; w < S; ++w) y[w] = lop3<0x80>(x[w], x[w - 1], x[w - 2]);
}

// Bits of word w at which a run may continue from the position below: those
// whose position, 2 below the index, does not start a window.
template <int S>
__host__ __device__ constexpr uint32_t start_mask(int w) {
  uint32_t x = 0;
  for (int r = 0; r < 32; ++r)
    if ((S * r + w + 2) % 4 != 0) x |= row_bit<S>(r);
  return x;
}

// The count of the final vector f, position p at index p + 2: runs of 1s per
// 4-base window, or its 1s.  With S a multiple of 4 a window is words 2, 3 of
// a row and the next two (of the next row past word S - 1).  Its runs start at
// f0, f1 & ~f0, f2 & ~f1 and f3 & ~f2; the first two exclude each other, as do
// the last two, so two population counts per four words hold them all.
template <int S>
__host__ __device__ __forceinline__ uint32_t stripe_count(const uint32_t (&f)[S], int count_mode) {
  uint32_t c = 0;
  if (count_mode == GK_COUNT_POPCOUNT) {
#pragma unroll
    for (int w = 0; w < S; ++w) c += st_popc(f[w]);
  } else if constexpr ((S & 3) == 0) {
#pragma unroll
    for (int w = 2; w < S; w += 4) {
      const uint32_t g = w + 2 < S ? f[w + 1] : row_up<S>(f[S - 1]);
      const uint32_t x = f[(w + 2) % S], y = f[(w + 3) % S];
      c += st_popc(f[w] | f[w + 1]) + st_popc(lop3<0x2E>(g, x, y));
    }
  } else {
#pragma unroll
    for (int w = 0; w < S; ++w)
      c += st_popc(f[w] & ~((w > 0 ? f[w > 0 ? w - 1 : 0] : row_up<S>(f[S - 1])) & start_mask<S>(w)));
  }
  return c;
}

// Exact masks at every shift count 0 .. K of NP pairs that share one read,
// each against its own window: after step k the running AND is the final
// vector of shift count k (Sec. 2.1, 3.4: dilate, erode, set the vacated
// positions, AND), counted from Klo on: emit(k, count).  r*, g*: striped
// planes, zero past m; K < m.  WHOLE: m is a multiple of S.
//
// Unlike the linear sweep this one erodes every mask: the deferred erosion's
// corrections next to the vacated runs would be spread over all S words and
// cost as much per threshold as the erosions they save.  Vectors move up by
// one position in the dilation and one more in the erosion, so the running
// AND holds position p at index p + 2; index p + 1 of a dilation one below
// position 0 and one past m - 1 is the mask's end bit, as the amendment rule
// wants it, without further work (m + 2 indices exist).
//
// Measured on GB300 against the linear sweep, launches alone: 20M pairs of 100
// bp at e = 0..10 1.206 -> 0.744 ms; 5M pairs of 150 bp at 0..15 0.548 -> 0.350
// ms, of 250 bp at 0..25 1.334 -> 0.844 ms; ALU operations per pair at 100 bp
// 1088 -> 651.  With the logic ops left to the compiler's own 3-input merging
// the step took 7 more of them (0.799 ms): it shares x[w] & x[w-1] between
// neighbours first, hence lop3.
template <int W, int S, int NP, bool WHOLE, typename Emit>
__host__ __device__ __forceinline__ void striped_exact(uint32_t m, uint32_t Klo, uint32_t K, int count_mode,
                                                       const uint32_t (&rh)[S], const uint32_t (&rl)[S],
                                                       const uint32_t (&gh)[NP][S], const uint32_t (&gl)[NP][S],
                                                       Emit emit) {
  uint32_t acc[NP][S], count[NP];
#pragma unroll
  for (int j = 0; j < NP; ++j) {  // shift 0: the Hamming mask, nothing vacated
    uint32_t d[S], x[S];
#pragma unroll
    for (int w = 0; w < S; ++w) d[w] = lop3<0xF6>(rh[w] ^ gh[j][w], rl[w], gl[j][w]);
    stripe_or3<S>(d, x);
    stripe_and3<S>(x, acc[j]);
  }
  if (Klo == 0) {
#pragma unroll
    for (int j = 0; j < NP; ++j) count[j] = stripe_count<S>(acc[j], count_mode);
    emit(0u, count);
  }
  // The read's +k and -k copies by their original word: at step k word w
  // compares with word (w - k) mod S of p and (w + k) mod S of n, and one word
  // of each wraps.  lm: positions below m; u: indices (position + 2) of the -k
  // copy that hold a read base, moving with it; v0..v2: rows below kb / S and
  // one and two more, the vacated indices of the +k mask.
  uint32_t ph[S], pl[S], nh[S], nl[S], lm[S], u[S];
#pragma unroll
  for (int w = 0; w < S; ++w) {
    ph[w] = nh[w] = rh[w];
    pl[w] = nl[w] = rl[w];
  }
  stripe_masks<W, S>(m, lm);
  stripe_masks<W, S>(m + 2, u);
  uint32_t v0 = 0u, v1 = row_bit<S>(0);
  // S odd: what a -k copy rotates out at the bottom would come back as bases
  // just below position 0.  (The +k copies' come back below position k - 2,
  // where the mask is vacated.)
  constexpr uint32_t kKeep = (S & 1) ? ~row_bit<S>(31) : 0xffffffffu;
  for (uint32_t kb = 0; kb < K; kb += S) {
    const uint32_t v2 = row_up<S>(v1) | 1u;
#pragma unroll
    for (int t = 0; t < S; ++t) {  // k = kb + t + 1: the words' names repeat every S steps
      const uint32_t k = kb + (uint32_t)t + 1u;
      if (k > K) break;
      constexpr int kS = S;
      const int up = (kS - 1 - t) % kS;
      ph[up] = row_up<S>(ph[up]);
      pl[up] = row_up<S>(pl[up]);
      if (WHOLE) {  // position m is in word 0: only the wrapping word carries a base past m
        ph[up] &= lm[0];
        pl[up] &= lm[0];
      }
      nh[t] = row_down<S>(nh[t]) & kKeep;
      nl[t] = row_down<S>(nl[t]) & kKeep;
      u[t] = row_down<S>(u[t]) & kKeep;
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        uint32_t d[S], x[S], y[S];
#pragma unroll
        for (int w = 0; w < S; ++w) {  // +k
          const int i = (w + kS - 1 - t) % kS;
          d[w] = lop3<0xF6>(ph[i] ^ gh[j][w], pl[i], gl[j][w]);
          if (!WHOLE) d[w] &= lm[w];  // the copy carries bases past m
        }
        stripe_or3<S>(d, x);
        stripe_and3<S>(x, y);
#pragma unroll
        for (int w = 0; w < S; ++w)
          acc[j][w] = lop3<0xE0>(acc[j][w], y[w], w < t + 3 - S ? v2 : (w < t + 3 ? v1 : v0));  // & (y | v)
#pragma unroll
        for (int w = 0; w < S; ++w) {  // -k
          const int i = (w + t + 1) % kS;
          d[w] = lop3<0xF6>(nh[i] ^ gh[j][w], nl[i], gl[j][w]);
        }
        stripe_or3<S>(d, x);
        stripe_and3<S>(x, y);
#pragma unroll
        for (int w = 0; w < S; ++w) acc[j][w] = lop3<0xD0>(acc[j][w], y[w], u[(w + t + 1) % kS]);  // & (y | ~u)
      }
      if (k >= Klo) {
#pragma unroll
        for (int j = 0; j < NP; ++j) count[j] = stripe_count<S>(acc[j], count_mode);
        emit(k, count);
      }
    }
    v0 = v1;
    v1 = v2;
  }
}

// Corrections next to the vacated runs of one shift count K <= 30 (the
// deferred erosion of filter.cuh, deferred_counts), from the linear planes:
// lo, bit p: position p <= K + 1; hi, bit b: position m - 32 + b.  1s are
// positions the final vector loses.
template <int W>
__host__ __device__ __forceinline__ void end_corrections(uint32_t m, uint32_t K, const uint32_t (&rh)[W],
                                                         const uint32_t (&rl)[W], const uint32_t (&gh)[W],
                                                         const uint32_t (&gl)[W], uint32_t &lo, uint32_t &hi) {
  static_assert(W >= 2, "more than one word");
  const uint32_t r1k = (2u << K) - 2u;  // bits 1..K
  auto terms = [&](uint32_t h, uint32_t l, uint32_t h0, uint32_t l0, uint32_t h1, uint32_t l1) -> uint32_t {
    // h, l: window bases from the end inwards; h0 .. l1: the read's end base and the next, broadcast
    const uint32_t a0 = (h ^ h0) | (l ^ l0), a1 = (h ^ h1) | (l ^ l1), vac = h | l;
    const uint32_t c2 = (vac << 1) | a0 | (a1 >> 1), c1 = (vac << 2) | (vac << 1) | a0;
    return (~(c1 & c2) & r1k) | ((~c2 & r1k) << 1);
  };
  const uint32_t tail = m - 32u * (W - 1);  // 1..32
  lo = terms(gh[0], gl[0], 0u - (rh[0] & 1u), 0u - (rl[0] & 1u), 0u - ((rh[0] >> 1) & 1u), 0u - ((rl[0] >> 1) & 1u));
  const uint32_t xh = st_shr64(rh[W - 2], rh[W - 1], tail), xl = st_shr64(rl[W - 2], rl[W - 1], tail);  // last 32
  hi = st_brev(terms(st_brev(st_shr64(gh[W - 2], gh[W - 1], tail)), st_brev(st_shr64(gl[W - 2], gl[W - 1], tail)),
                     0u - (xh >> 31), 0u - (xl >> 31), 0u - ((xh >> 30) & 1u), 0u - ((xl >> 30) & 1u)));
}

// The count at one shift count K (1 <= K <= 30, K < m) of NP pairs that share
// one read: deferred erosion (filter.cuh, deferred_counts) on stripes.  The
// loop ANDs dilations with the vacated positions set before them and the AND
// is eroded once; clo, chi are the pairs' end_corrections.  A step takes 8 S
// logic ops, 2 S fewer than an exact one; the corrections and their striping
// cost about 4 (S = 4) or 3 (S = 8) steps' worth of that.
template <int W, int S, int NP, bool WHOLE>
__host__ __device__ __forceinline__ void striped_deferred(uint32_t m, uint32_t K, int count_mode,
                                                          const uint32_t (&rh)[S], const uint32_t (&rl)[S],
                                                          const uint32_t (&gh)[NP][S], const uint32_t (&gl)[NP][S],
                                                          const uint32_t (&clo)[NP], const uint32_t (&chi)[NP],
                                                          uint32_t (&count)[NP]) {
  uint32_t acc[NP][S];  // position p at index p + 1
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    uint32_t d[S];
#pragma unroll
    for (int w = 0; w < S; ++w) d[w] = lop3<0xF6>(rh[w] ^ gh[j][w], rl[w], gl[j][w]);
    stripe_or3<S>(d, acc[j]);
  }
  // As in striped_exact, in positions: u: those of the -k copy that hold a
  // read base; v0, v1: the rows vacated in the +k mask.
  uint32_t ph[S], pl[S], nh[S], nl[S], lm[S], u[S];
  stripe_masks<W, S>(m, lm);
#pragma unroll
  for (int w = 0; w < S; ++w) {
    ph[w] = nh[w] = rh[w];
    pl[w] = nl[w] = rl[w];
    u[w] = lm[w];
  }
  // S odd: what rotates in at the top of u would be a read base past m.
  constexpr uint32_t kKeep = (S & 1) ? ~row_bit<S>(31) : 0xffffffffu;
  uint32_t v0 = 0u;
  for (uint32_t kb = 0; kb < K; kb += S) {
    const uint32_t v1 = row_up<S>(v0) | 1u;
#pragma unroll
    for (int t = 0; t < S; ++t) {  // k = kb + t + 1
      if (kb + (uint32_t)t + 1u > K) break;
      constexpr int kS = S;
      const int up = (kS - 1 - t) % kS;
      ph[up] = row_up<S>(ph[up]);
      pl[up] = row_up<S>(pl[up]);
      if (WHOLE) {
        ph[up] &= lm[0];
        pl[up] &= lm[0];
      }
      nh[t] = row_down<S>(nh[t]);
      nl[t] = row_down<S>(nl[t]);
      u[t] = row_down<S>(u[t]) & kKeep;
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        uint32_t d[S], x[S], y[S];
#pragma unroll
        for (int w = 0; w < S; ++w) {  // +k
          const int i = (w + kS - 1 - t) % kS;
          const uint32_t v = w <= t ? v1 : v0;
          if (WHOLE)
            d[w] = lop3<0xF6>(lop3<0xDE>(ph[i], v, gh[j][w]), pl[i], gl[j][w]);
          else
            d[w] = lop3<0xEA>(lop3<0xF6>(ph[i] ^ gh[j][w], pl[i], gl[j][w]), lm[w], v);
        }
        stripe_or3<S>(d, x);
#pragma unroll
        for (int w = 0; w < S; ++w) {  // -k
          const int i = (w + t + 1) % kS;
          d[w] = lop3<0xF6>(lop3<0x7B>(nh[i], u[i], gh[j][w]), nl[i], gl[j][w]);
        }
        if (S & 1) {  // positions past m, all vacated, must not come round to position 0
          d[S - 1] &= ~row_bit<S>(31);
          d[S - 2] &= ~row_bit<S>(31);
        }
        stripe_or3<S>(d, y);
#pragma unroll
        for (int w = 0; w < S; ++w) acc[j][w] = lop3<0x80>(acc[j][w], x[w], y[w]);
      }
    }
    v0 = v1;
  }
  // hi's bit b is index m - 30 + b of the final vector (position + 2).
  const uint32_t tail = m - 32u * (W - 1), sh = (tail + 2u) & 31u;
  const bool top = tail >= 30;
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    constexpr int kC = W < S ? W + 1 : W;
    uint32_t c[kC], cs[S], f[S];
#pragma unroll
    for (int w = 0; w < kC; ++w) c[w] = 0u;
    c[0] = clo[j] << 2;
    c[1] |= clo[j] >> 30;
    const uint32_t l = chi[j] << sh, h = st_shr64(chi[j], 0u, 32u - sh);
    c[W - 2] |= top ? 0u : l;
    c[W - 1] |= top ? l : h;
    if (W < S) c[W < S ? W : 0] |= top ? h : 0u;
    stripe_linear<kC, S>(c, cs);
    stripe_and3<S>(acc[j], f);
#pragma unroll
    for (int w = 0; w < S; ++w) f[w] &= ~cs[w];
    count[j] = stripe_count<S>(f, count_mode);
  }
}

}  // namespace gk
