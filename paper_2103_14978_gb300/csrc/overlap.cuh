// Small shift counts of one threshold: linear words that overlap by two bases.
//
// Word w holds positions 30w .. 30w + 31, so the dilation moved up by one
// (position p <- d[p] | d[p-1] | d[p-2]) needs no bit of another word: two plain
// left shifts, which run on the multiply-add pipe, where words side by side
// take two funnel shifts on the ALU pipe, the pipe that bounds the filter.
// (Its two lowest bits are wrong in every word but the first; the word below
// holds those positions.)  The read's copies at shift k are funnel shifts of
// the ordinary words by amounts fixed at compile time, so the steps unroll, up
// to kOverlapMax.  A step costs 7 logic ops per word and pair and 4 funnel
// shifts per word and read, against 11 and 4.  The stripes of stripe.cuh take fewer still but
// cost about three steps to set up; they serve larger shift counts.
#pragma once

#include "stripe.cuh"

namespace gk {

constexpr uint32_t kOverlapMax = 7;

// Reads W overlapping words hold: position m (and m + 1 of the dilation) too.
template <int W>
__host__ __device__ constexpr uint32_t overlap_limit() {
  return 30u * W;
}

// Bits [p, p + 32) of linear words, p a compile-time constant after unrolling
// (below 0 and past the words: zeros).
template <int W>
__host__ __device__ __forceinline__ uint32_t linear_bits(const uint32_t (&x)[W], int p) {
  const int q = p < 0 ? -1 : p / 32, s = p - 32 * q;
  const uint32_t lo = q >= 0 && q < W ? x[q >= 0 && q < W ? q : 0] : 0u;
  const uint32_t hi = q + 1 < W ? x[q + 1 < W ? q + 1 : 0] : 0u;
  return s == 0 ? lo : st_shr64(lo, hi, (uint32_t)s);
}

// Positions below n of the 32 from word w on, as a mask.
__host__ __device__ __forceinline__ uint32_t overlap_below(uint32_t n, int w) {
  const uint32_t k = n > 30u * (uint32_t)w ? n - 30u * (uint32_t)w : 0u;
  return k >= 32 ? 0xffffffffu : (1u << k) - 1u;
}

// The AND of the dilations of NP pairs that share one read, at shift count K
// (deferred erosion, filter.cuh): linear words of D'[p] = D[p - 1], p = 0 .. m +
// 1.  KC >= 0: K at compile time.  K <= kOverlapMax, K < m, 30 (W - 1) < m <= 30 W
// or less.
template <int W, int NP, int KC>
__host__ __device__ __forceinline__ void overlap_and(uint32_t m, uint32_t K, const uint32_t (&rh)[W],
                                                     const uint32_t (&rl)[W], const uint32_t (&gh)[NP][W],
                                                     const uint32_t (&gl)[NP][W], uint32_t (&out)[NP][W]) {
  constexpr int kMax = KC >= 0 ? KC : (int)kOverlapMax;
  // The last two words end past the read: bases there are masked (+k) or
  // vacated (-k); the others end before m - k.
  uint32_t acc[NP][W], oh[NP][W], ol[NP][W], in[W];
#pragma unroll
  for (int w = 0; w < W; ++w) in[w] = overlap_below(m, w);
#pragma unroll
  for (int j = 0; j < NP; ++j)
#pragma unroll
    for (int w = 0; w < W; ++w) {
      oh[j][w] = linear_bits<W>(gh[j], 30 * w);
      ol[j][w] = linear_bits<W>(gl[j], 30 * w);
      const uint32_t d = lop3<0xF6>(linear_bits<W>(rh, 30 * w) ^ oh[j][w], linear_bits<W>(rl, 30 * w), ol[j][w]);
      acc[j][w] = lop3<0xFE>(d, d << 1, d << 2);
    }
#pragma unroll
  for (int k = 1; k <= kMax; ++k) {
    if (KC < 0 && (uint32_t)k > K) break;
    const uint32_t lead = (1u << k) - 1u;  // vacated in mask +k: word 0
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const uint32_t ph = linear_bits<W>(rh, 30 * w - k), pl = linear_bits<W>(rl, 30 * w - k);
      const uint32_t nh = linear_bits<W>(rh, 30 * w + k), nl = linear_bits<W>(rl, 30 * w + k);
      // -k: vacated from m - k on
      const uint32_t held = w + 3 > W ? overlap_below(m - (uint32_t)k, w) : 0xffffffffu;
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        uint32_t d = lop3<0xF6>(w == 0 ? lop3<0xDE>(ph, lead, oh[j][w]) : ph ^ oh[j][w], pl, ol[j][w]);
        if (w + 2 >= W) d &= in[w];  // the +k copy carries bases past m
        uint32_t n = lop3<0xF6>(w + 3 > W ? lop3<0x7B>(nh, held, oh[j][w]) : nh ^ oh[j][w], nl, ol[j][w]);
        const uint32_t x = lop3<0xFE>(d, d << 1, d << 2), y = lop3<0xFE>(n, n << 1, n << 2);
        acc[j][w] = lop3<0x80>(acc[j][w], x, y);
      }
    }
  }
  // Back to words side by side: linear word v is bits 2v .. 31 of word v and,
  // above 31 - 2v, bits 2 .. of word v + 1.
#pragma unroll
  for (int j = 0; j < NP; ++j)
#pragma unroll
    for (int v = 0; v < W; ++v) {
      const uint32_t lo = acc[j][v] >> (2 * v);
      const uint32_t up = v == 0 || v + 1 >= W ? 0u : 0xffffffffu << ((32 - 2 * v) & 31);
      out[j][v] = up ? (lo & ~up) | ((acc[j][v + 1 < W ? v + 1 : v] << ((30 - 2 * v) & 31)) & up) : lo;
    }
}

// Counts of NP pairs at one shift count, as deferred_counts.
template <int W, int NP, int KC>
__host__ __device__ __forceinline__ void overlap_counts(uint32_t m, uint32_t K, int count_mode,
                                                        const uint32_t (&rh)[W], const uint32_t (&rl)[W],
                                                        const uint32_t (&gh)[NP][W], const uint32_t (&gl)[NP][W],
                                                        uint32_t (&count)[NP]) {
  static_assert(W >= 2, "more than one word");
  uint32_t x[NP][W];
  overlap_and<W, NP, KC>(m, K, rh, rl, gh, gl, x);
  const uint32_t tail = m - 32u * (W - 1);  // 1..28 bases in the last word
  const uint32_t lastmask = (1u << tail) - 1u;
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    uint32_t f[W], lo, hi;
#pragma unroll
    for (int w = 0; w < W; ++w) {  // f[p] = D[p-1] & D[p] & D[p+1]
      const uint32_t up = w + 1 < W ? x[j][w + 1 < W ? w + 1 : w] : 0u;
      f[w] = lop3<0x80>(x[j][w], st_shr64(x[j][w], up, 1u), st_shr64(x[j][w], up, 2u));
    }
    if (KC != 0) {
      end_corrections<W>(m, K, rh, rl, gh[j], gl[j], lo, hi);
      f[0] &= ~lo;
      f[W - 1] &= ~(hi >> (32u - tail));
      f[W - 2] &= ~(hi << tail);
    }
    f[W - 1] &= lastmask;
    uint32_t c = 0;
    if (count_mode == GK_COUNT_POPCOUNT) {
#pragma unroll
      for (int w = 0; w < W; ++w) c += st_popc(f[w]);
    } else {
#pragma unroll
      for (int w = 0; w < W; ++w) c += st_popc(f[w] & ~((f[w] << 1) & 0xEEEEEEEEu));
    }
    count[j] = c;
  }
}

}  // namespace gk
