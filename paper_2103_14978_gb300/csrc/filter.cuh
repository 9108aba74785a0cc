// The plain GateKeeper-GPU filter kernel: one thread per (read, candidate)
// pair, every mask held in registers as W = ceil(m/32) 32-bit words.
//
// Per pair (arxiv 2103.14978):
//   - undefined pairs (a non-ACGT base in the read or the window) pass with
//     accept = 1 and no filtration (Sec. 3.3);
//   - the window's two bit planes are funnel-shifted out of the resident
//     reference at the candidate offset;
//   - mask s compares the read shifted by s bases with the window: per base,
//     (high XOR) | (low XOR) is 1 when the 2-bit codes differ, and shifted-in
//     bases are code 00 (Sec. 2.1, Sec. 3.4).  The shifted read is kept
//     incrementally: each step moves the +k copy up and the -k copy down by
//     one base, a funnel shift per word and plane;
//   - amendment (Sec. 2.1) flips 0-streaks of length 1-2 bounded by 1s.  On a
//     bit vector with zeros outside [0, m) this equals a morphological closing
//     with a 3-base window: dilate (x | x<<1 | x>>1), then erode (AND of the
//     dilation and its two 1-base shifts); the erosion reads the dilation one
//     base beyond each end, which is the mask's own end bit;
//   - the edge OR of Sec. 3.4 sets, after amendment, the k vacated positions
//     of mask +k (the low end) and of mask -k (the high end).  The vacated
//     sets are kept as two incremental bit vectors and folded into the AND:
//     acc &= eroded | edge is one 3-input logic op.  With k < 32 the low set
//     lives in word 0 and the high set in the top two words only;
//   - the AND of the 2e+1 masks stays in registers; the count of the final
//     vector is per-window runs (a 1 starts a run unless the bit below it is
//     1 and in the same 4-base window) or a popcount (Sec. 2.1).
//
// A shift by k >= m vacates the whole mask, which the edge OR then fills with
// 1s, so only k <= m-1 are computed.  Without the edge OR (the original
// GateKeeper) such masks are the window compared with code 00, ANDed once.
#pragma once

#include <atomic>

#include "gk_internal.cuh"
#include "overlap.cuh"
#include "stripe.cuh"

namespace gk {

// Threads per block.  A block's warps load together and its registers are
// freed together, so smaller blocks interleave one block's loads with
// another's arithmetic: against 256 threads (same registers, GB300) 150 bp at
// e = 3 ran 0.248 -> 0.213 ms, 250 bp at e = 5 0.324 -> 0.259, 100 bp at e = 5
// 0.461 -> 0.434; 64 threads the same as 128.
constexpr int kFilterThreads = 128;
// The persistent warps of the queue of defined pairs already interleave
// (128 threads measured 1% slower).
constexpr int kQueueThreads = 256;

template <int W>
__device__ __forceinline__ void amend_and(const uint32_t (&d)[W], uint32_t (&acc)[W],
                                          const uint32_t (&edge)[W]) {
  uint32_t dil[W];
#pragma unroll
  for (int w = 0; w < W; ++w) {
    const uint32_t below = __funnelshift_l(w > 0 ? d[w - 1] : 0u, d[w], 1);      // bit i <- d[i-1]
    const uint32_t above = __funnelshift_r(d[w], w + 1 < W ? d[w + 1] : 0u, 1);  // bit i <- d[i+1]
    dil[w] = d[w] | below | above;
  }
#pragma unroll
  for (int w = 0; w < W; ++w) {
    // The dilation one base below position 0 is d[0]; one base above the
    // last word it is the last word's top bit of d.
    const uint32_t lo_in = w > 0 ? dil[w - 1] : (d[0] << 31);
    const uint32_t hi_in = w + 1 < W ? dil[w + 1] : (d[W - 1] >> 31);
    const uint32_t below = __funnelshift_l(lo_in, dil[w], 1);
    const uint32_t above = __funnelshift_r(dil[w], hi_in, 1);
    acc[w] &= (dil[w] & below & above) | edge[w];
  }
}

// Inputs of one pair.
template <int W>
struct PairData {
  uint32_t rid, off, e, m;  // m: this pair's read length
  int status;     // 0 filter, 1 undefined, 2 invalid
  uint32_t nflag; // read's N flag
  uint2 ni;       // N index word of the window start
  uint2 r[W];     // read words
  uint2 g[W + 1]; // reference words covering the window
};

// Read words 0..W-1 of a valid pair (W = ceil(m/32) <= the row stride) in
// 16-byte loads, half the requests of 8-byte loads.  With a 16-byte aligned
// read buffer and an even row stride every read row starts on 16 bytes (an
// odd W is below the stride, so the extra word is row padding); otherwise
// the read takes 8-byte loads.
template <int W>
__device__ __forceinline__ void load_read_wide(const uint2 *reads, uint32_t stride_words, PairData<W> &x) {
  const uint2 *rp = reads + (uint64_t)x.rid * stride_words;
  if ((stride_words & 1u) == 0 && (reinterpret_cast<uintptr_t>(reads) & 15u) == 0) {
    const uint4 *rq = reinterpret_cast<const uint4 *>(rp);
#pragma unroll
    for (int i = 0; i < (W + 1) / 2; ++i) {
      const uint4 v = rq[i];
      x.r[2 * i] = make_uint2(v.x, v.y);
      if (2 * i + 1 < W) x.r[2 * i + 1] = make_uint2(v.z, v.w);
    }
  } else {
#pragma unroll
    for (int w = 0; w < W; ++w) x.r[w] = rp[w];
  }
}

// Genome window words off/32 .. off/32 + W of a valid pair (off + m within
// the genome) in aligned 16-byte loads from the even word at or below
// off/32: ceil((W+1)/2) loads, one more when W and off/32 are both odd; the
// last word read is at most n_words + 1, inside the genome's two zero tail
// words.
template <int W>
__device__ __forceinline__ void load_window_wide(const uint2 *ref_hl, PairData<W> &x) {
  constexpr int NE = (W + 2) / 2;  // ceil((W + 1) / 2)
  const uint32_t s = x.off >> 5;
  const bool odd = (s & 1u) != 0;
  const uint4 *gq = reinterpret_cast<const uint4 *>(ref_hl + (s & ~1u));
  uint2 v[2 * NE + 2];
#pragma unroll
  for (int i = 0; i < NE; ++i) {
    const uint4 q = gq[i];
    v[2 * i] = make_uint2(q.x, q.y);
    v[2 * i + 1] = make_uint2(q.z, q.w);
  }
  v[2 * NE] = v[2 * NE + 1] = make_uint2(0u, 0u);
  if ((W & 1) && odd) {
    const uint4 q = gq[NE];
    v[2 * NE] = make_uint2(q.x, q.y);
  }
#pragma unroll
  for (int w = 0; w <= W; ++w) x.g[w] = odd ? v[w + 1] : v[w];
}

template <int W>
__device__ __forceinline__ void load_words_wide(const uint2 *reads, uint32_t stride_words, const uint2 *ref_hl,
                                                PairData<W> &x) {
  load_read_wide<W>(reads, stride_words, x);
  load_window_wide<W>(ref_hl, x);
}

// Window words off/32 .. off/32 + W of a valid pair in 8-byte loads: 40
// contiguous bytes, two 32-byte sectors.  SKIP_LAST: word off/32 + W only
// when the window reaches into it ((off mod 32) + m > 32W); otherwise its
// bits land past m, where the planes are masked (at 100 bp 29 pairs in 32
// skip it).  (A copy of the genome holding overlapping word pairs, read in
// 16-byte loads, measured 13% slower at e = 0: its three loads touch three
// sectors.)
template <int W, bool WIDE, bool SKIP_LAST = false>
__device__ __forceinline__ void load_window(const FilterArgs &a, PairData<W> &x) {
  if (WIDE) {
    load_window_wide<W>(a.ref_hl, x);
  } else {
    const uint2 *gp = a.ref_hl + (x.off >> 5);
#pragma unroll
    for (int w = 0; w < W; ++w) x.g[w] = gp[w];
    if (SKIP_LAST)
      x.g[W] = (x.off & 31u) + x.m > 32u * W ? gp[W] : make_uint2(0u, 0u);
    else
      x.g[W] = gp[W];
  }
}

// Loads pair p.  WIDE: read and window words in 16-byte loads.  The plain
// kernel keeps 8-byte loads: at e <= 2 (the launches waiting on loads) the
// wide form measured 2-6% slower at 100 and 150 bp.  share (nullable): a
// pair loaded before; when it is valid and has the same read, its read words
// and N flag are copied instead of loaded again.
template <int W, bool WIDE = false, bool SKIP_LAST = false>
__device__ __forceinline__ void load_pair(const FilterArgs &a, uint64_t p, PairData<W> &x,
                                          const PairData<W> *share = nullptr) {
  x.rid = a.pair_read[p];
  x.off = a.pair_off[p];
  x.e = a.pair_e ? (uint32_t)a.pair_e[p] : a.fixed_e;
  x.m = a.m;
  x.status = (x.rid > a.rid_last || x.off >= a.off_end) ? 2 : 0;
  x.nflag = 0;
  x.ni = make_uint2(0, 0xffffffffu);
  if (x.status == 0 && a.m > 0) {
    if (a.ref_nidx) x.ni = a.ref_nidx[x.off >> 5];
    if (share && share->status == 0 && share->rid == x.rid) {
      x.nflag = share->nflag;
#pragma unroll
      for (int w = 0; w < W; ++w) x.r[w] = share->r[w];
    } else {
      if (a.read_nflag) x.nflag = a.read_nflag[x.rid];
      if (WIDE) {
        load_read_wide<W>(a.reads, a.stride_words, x);
      } else {
        const uint2 *rp = a.reads + (uint64_t)x.rid * a.stride_words;
#pragma unroll
        for (int w = 0; w < W; ++w) x.r[w] = rp[w];
      }
    }
    load_window<W, WIDE, SKIP_LAST>(a, x);
  }
}

// Filters one loaded pair; returns the count.
template <int W, bool SMALL_K>
__device__ __forceinline__ uint32_t filter_loaded(const FilterArgs &a, const PairData<W> &x) {
  const uint32_t m = x.m;
  const uint32_t tail = m - 32u * (W - 1);  // 1..32 bases in the last word
  const uint32_t lastmask = tail >= 32 ? 0xffffffffu : ((1u << tail) - 1u);

  uint32_t rh[W], rl[W], gh[W], gl[W];
  const uint32_t sh = x.off & 31;
#pragma unroll
  for (int w = 0; w < W; ++w) {
    rh[w] = x.r[w].x;
    rl[w] = x.r[w].y;
    gh[w] = __funnelshift_r(x.g[w].x, x.g[w + 1].x, sh);
    gl[w] = __funnelshift_r(x.g[w].y, x.g[w + 1].y, sh);
  }
  // Both sequences zero past m: the Hamming and -k masks need no masking.
  rh[W - 1] &= lastmask;
  rl[W - 1] &= lastmask;
  gh[W - 1] &= lastmask;
  gl[W - 1] &= lastmask;

  uint32_t acc[W], d[W], zero[W];
#pragma unroll
  for (int w = 0; w < W; ++w) {
    acc[w] = 0xffffffffu;
    zero[w] = 0;
    d[w] = (rh[w] ^ gh[w]) | (rl[w] ^ gl[w]);
  }
  amend_and<W>(d, acc, zero);  // shift 0: the Hamming mask, no edge

  const uint32_t kmax = min(x.e, m - 1);
  const bool edge_on = a.edge_on != 0;
  if (kmax > 0) {
    uint32_t ph[W], pl[W], nh[W], nl[W], lead[W], trail[W];
#pragma unroll
    for (int w = 0; w < W; ++w) {
      ph[w] = nh[w] = rh[w];
      pl[w] = nl[w] = rl[w];
      lead[w] = 0;
      trail[w] = 0;  // positions >= m - k (and above m, which acc already cleared)
    }
    if (edge_on) trail[W - 1] = ~lastmask;
    const uint32_t lead_fill = edge_on ? 0x80000000u : 0u;
    const uint32_t trail_fill = edge_on ? 0xffffffffu : 0u;
    for (uint32_t k = 1; k <= kmax; ++k) {
#pragma unroll
      for (int w = W - 1; w >= 0; --w) {  // +k copy: one base up
        ph[w] = __funnelshift_l(w > 0 ? ph[w - 1] : 0u, ph[w], 1);
        pl[w] = __funnelshift_l(w > 0 ? pl[w - 1] : 0u, pl[w], 1);
        // vacated low positions [0, k): with k < 32 only word 0 holds them
        if (!SMALL_K || w == 0) lead[w] = __funnelshift_l(w > 0 ? lead[w - 1] : lead_fill, lead[w], 1);
      }
#pragma unroll
      for (int w = 0; w < W; ++w) {  // -k copy: one base down
        nh[w] = __funnelshift_r(nh[w], w + 1 < W ? nh[w + 1] : 0u, 1);
        nl[w] = __funnelshift_r(nl[w], w + 1 < W ? nl[w + 1] : 0u, 1);
        // vacated high positions [m-k, m): with k < 32 only the top two words
        if (!SMALL_K || w + 2 >= W) trail[w] = __funnelshift_r(trail[w], w + 1 < W ? trail[w + 1] : trail_fill, 1);
      }
#pragma unroll
      for (int w = 0; w < W; ++w) d[w] = (ph[w] ^ gh[w]) | (pl[w] ^ gl[w]);
      d[W - 1] &= lastmask;  // the +k copy carries read bases past m
      amend_and<W>(d, acc, lead);
#pragma unroll
      for (int w = 0; w < W; ++w) d[w] = (nh[w] ^ gh[w]) | (nl[w] ^ gl[w]);
      amend_and<W>(d, acc, trail);
    }
  }
  if (!edge_on && x.e >= m) {
    // Fully vacated masks of the original GateKeeper: window vs code 00.
#pragma unroll
    for (int w = 0; w < W; ++w) d[w] = gh[w] | gl[w];
    amend_and<W>(d, acc, zero);
  }

  uint32_t count = 0;
  if (a.count_mode == GK_COUNT_POPCOUNT) {
#pragma unroll
    for (int w = 0; w < W; ++w) count += __popc(acc[w]);
  } else {
#pragma unroll
    for (int w = 0; w < W; ++w) count += __popc(acc[w] & ~((acc[w] << 1) & 0xEEEEEEEEu));
  }
  return count;
}

// Deferred-erosion form of filter_loaded for the edge OR on and every shift
// count k <= 30.  Erosion commutes with AND (the AND of erosions is the
// erosion of the AND), so the loop ANDs dilated masks only and erodes once at
// the end.  Mask +k is ORed with its dilated vacated set [-1, k] and mask -k
// with [m-k-1, m]; that agrees with "erode, then OR the vacated set" at every
// position except the two next to each vacated run (k and k+1, m-k-2 and
// m-k-1), where the erosion of the true mask needs two dilation bits the OR
// hid.  Those bits depend only on the read's first or last two bases against
// the window and on which window bases are 'A', so their corrections for all
// k are computed once per pair; so are the two values of the AND one base
// outside each end that the final erosion reads.
// Deferred-erosion counts of NP pairs that share one read and one shift
// count K, each against its own window: the read's +k and -k copies (4W
// funnel shifts per step) are built once for all NP windows.  rh/rl and
// gh/gl are the read's and the windows' planes, zero past m.
template <int W, int NP, bool DIRECT = false>
__device__ __forceinline__ void deferred_counts(const FilterArgs &a, uint32_t m, uint32_t K,
                                                const uint32_t (&rh)[W], const uint32_t (&rl)[W],
                                                const uint32_t (&gh)[NP][W], const uint32_t (&gl)[NP][W],
                                                uint32_t (&count)[NP]) {
  const uint32_t tail = m - 32u * (W - 1);  // 1..32 bases in the last word
  const uint32_t lastmask = tail >= 32 ? 0xffffffffu : ((1u << tail) - 1u);

  uint32_t acc[NP][W], d[W], dn[W];
  // dilation of a mask: bit i <- d[i-1] | d[i] | d[i+1], zeros outside the words
  auto dil = [&](const uint32_t (&dd)[W], int w) -> uint32_t {
    const uint32_t below = __funnelshift_l(w > 0 ? dd[w - 1] : 0u, dd[w], 1);
    const uint32_t above = __funnelshift_r(dd[w], w + 1 < W ? dd[w + 1] : 0u, 1);
    return dd[w] | below | above;
  };
#pragma unroll
  for (int j = 0; j < NP; ++j) {
#pragma unroll
    for (int w = 0; w < W; ++w) d[w] = (rh[w] ^ gh[j][w]) | (rl[w] ^ gl[j][w]);
#pragma unroll
    for (int w = 0; w < W; ++w) acc[j][w] = dil(d, w);  // shift 0
  }
  {
    // DIRECT (a shift count fixed at compile time): the read's +k and -k
    // copies come straight from rh/rl by k-base funnel shifts, no copy carried
    // from step to step (fewer live registers: measured faster at K = 0..2);
    // otherwise each step moves the carried copies by one base (faster for a
    // runtime K and in the sweep).
    uint32_t ph[W], pl[W], nh[W], nl[W];
    if (!DIRECT) {
#pragma unroll
      for (int w = 0; w < W; ++w) {
        ph[w] = nh[w] = rh[w];
        pl[w] = nl[w] = rl[w];
      }
    }
    // The vacated positions of each shifted mask are ORed into its difference
    // vector before the dilation: dil(d | V) = dil(d) | dil(V), the mask ORed
    // with its dilated vacated set.
    uint32_t lead = 0u;               // mask +k: positions 0..k-1 (word 0)
    uint32_t tv_hi = ~lastmask;       // mask -k: positions >= m-k (and >= m), top word
    uint32_t tv_lo = 0u;              // and the word below it
    for (uint32_t k = 1; k <= K; ++k) {
      if (DIRECT) {
#pragma unroll
        for (int w = 0; w < W; ++w) {
          ph[w] = __funnelshift_l(w > 0 ? rh[w - 1] : 0u, rh[w], k);
          pl[w] = __funnelshift_l(w > 0 ? rl[w - 1] : 0u, rl[w], k);
          nh[w] = __funnelshift_r(rh[w], w + 1 < W ? rh[w + 1] : 0u, k);
          nl[w] = __funnelshift_r(rl[w], w + 1 < W ? rl[w + 1] : 0u, k);
        }
      } else {
#pragma unroll
        for (int w = W - 1; w >= 0; --w) {
          ph[w] = __funnelshift_l(w > 0 ? ph[w - 1] : 0u, ph[w], 1);
          pl[w] = __funnelshift_l(w > 0 ? pl[w - 1] : 0u, pl[w], 1);
        }
#pragma unroll
        for (int w = 0; w < W; ++w) {
          nh[w] = __funnelshift_r(nh[w], w + 1 < W ? nh[w + 1] : 0u, 1);
          nl[w] = __funnelshift_r(nl[w], w + 1 < W ? nl[w + 1] : 0u, 1);
        }
      }
      lead = 2u * lead + 1u;
      tv_lo = __funnelshift_r(tv_lo, tv_hi, 1);
      tv_hi = __funnelshift_r(tv_hi, 0xffffffffu, 1);
#pragma unroll
      for (int j = 0; j < NP; ++j) {
#pragma unroll
        for (int w = 0; w < W; ++w) {
          const uint32_t vp = w == 0 ? lead : 0u;
          const uint32_t vn = w == W - 1 ? tv_hi : (w == W - 2 ? tv_lo : 0u);
          d[w] = (ph[w] ^ gh[j][w]) | vp | (pl[w] ^ gl[j][w]);
          dn[w] = (nh[w] ^ gh[j][w]) | vn | (nl[w] ^ gl[j][w]);
        }
        d[W - 1] &= lastmask;  // the +k copy carries read bases past m
#pragma unroll
        for (int w = 0; w < W; ++w) acc[j][w] &= dil(d, w) & dil(dn, w);
      }
    }
  }

  // ---- once per pair: end values of the AND, corrections, final erosion ----
  const uint32_t rangeK = (2u << K) - 1u;  // bits 0..K
  const uint32_t r1k = rangeK & ~1u;       // bits 1..K
  // The read's last 32 bases mirrored: bit j is position m-1-j (positions
  // below 0 read as code 00).  The high end's terms are the low end's
  // formulas on mirrored vectors, in 32-bit words.
  const uint32_t xrh = __funnelshift_rc(W >= 2 ? rh[W >= 2 ? W - 2 : 0] : 0u, rh[W - 1], tail);
  const uint32_t xrl = __funnelshift_rc(W >= 2 ? rl[W >= 2 ? W - 2 : 0] : 0u, rl[W - 1], tail);
  const uint32_t b0h = 0u - (xrh >> 31), b0l = 0u - (xrl >> 31);                // R[m-1]
  const uint32_t b1h = 0u - ((xrh >> 30) & 1u), b1l = 0u - ((xrl >> 30) & 1u);  // R[m-2]
  const uint32_t r0h = 0u - (rh[0] & 1u), r0l = 0u - (rl[0] & 1u);              // R[0]
  const uint32_t r1h = 0u - ((rh[0] >> 1) & 1u), r1l = 0u - ((rl[0] >> 1) & 1u);  // R[1]
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    // AND one base below position 0: every non-positive shift compares G[0]
    // with R[i], i = 0..K.
    const uint32_t g0h = 0u - (gh[j][0] & 1u), g0l = 0u - (gl[j][0] & 1u);
    const uint32_t q0 = (rh[0] ^ g0h) | (rl[0] ^ g0l);
    const uint32_t vlo = ((~q0 & rangeK) == 0) ? 1u : 0u;
    // The window's last 32 bases mirrored.
    const uint32_t mgh = __brev(__funnelshift_rc(W >= 2 ? gh[j][W >= 2 ? W - 2 : 0] : 0u, gh[j][W - 1], tail));
    const uint32_t mgl = __brev(__funnelshift_rc(W >= 2 ? gl[j][W >= 2 ? W - 2 : 0] : 0u, gl[j][W - 1], tail));
    // AND one base above position m-1, needed only when m fills the words:
    // every non-negative shift compares G[m-1] with R[m-1-i], i = 0..K.
    uint32_t vtop = 0u;
    if (tail == 32) {
      const uint32_t gmh = 0u - (mgh & 1u), gml = 0u - (mgl & 1u);
      const uint32_t qm = (__brev(xrh) ^ gmh) | (__brev(xrl) ^ gml);
      vtop = ((~qm & rangeK) == 0) ? 1u : 0u;
    }
    uint32_t f[W];
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const uint32_t lo_in = w > 0 ? acc[j][w - 1] : (vlo << 31);
      const uint32_t hi_in = w + 1 < W ? acc[j][w + 1] : vtop;
      f[w] = acc[j][w] & __funnelshift_l(lo_in, acc[j][w], 1) & __funnelshift_r(acc[j][w], hi_in, 1);
    }
    // Low-end corrections (positions 1..K+1, word 0).
    {
      const uint32_t v0 = W == 1 ? lastmask : 0xffffffffu;
      const uint32_t a0 = (gh[j][0] ^ r0h) | (gl[j][0] ^ r0l);
      const uint32_t a1 = ((gh[j][0] ^ r1h) | (gl[j][0] ^ r1l)) & v0;
      const uint32_t vac = gh[j][0] | gl[j][0];
      const uint32_t c1 = (vac << 2) | (vac << 1) | a0;
      const uint32_t c2 = (vac << 1) | a0 | (a1 >> 1);
      f[0] &= ~((~(c1 & c2) & r1k) | ((~c2 & r1k) << 1));
    }
    // High-end corrections (positions m-K-2..m-2), computed mirrored and
    // mapped back: mirrored bit j is position m-1-j.
    {
      const uint32_t a0 = (mgh ^ b0h) | (mgl ^ b0l);
      const uint32_t a1 = (mgh ^ b1h) | (mgl ^ b1l);
      const uint32_t vac = mgh | mgl;
      const uint32_t c1 = (vac << 2) | (vac << 1) | a0;
      const uint32_t c2 = (vac << 1) | a0 | (a1 >> 1);
      const uint32_t nc = __brev((~(c1 & c2) & r1k) | ((~c2 & r1k) << 1));  // bit b: position m-32+b
      f[W - 1] &= ~(nc >> (32u - tail));
      if (W >= 2 && tail < 32) f[W >= 2 ? W - 2 : 0] &= ~(nc << tail);
    }
    f[W - 1] &= lastmask;

    uint32_t c = 0;
    if (a.count_mode == GK_COUNT_POPCOUNT) {
#pragma unroll
      for (int w = 0; w < W; ++w) c += __popc(f[w]);
    } else {
#pragma unroll
      for (int w = 0; w < W; ++w) c += __popc(f[w] & ~((f[w] << 1) & 0xEEEEEEEEu));
    }
    count[j] = c;
  }
}

template <int NP>
struct FinishPrep;
template <int W, int NP>
__device__ __forceinline__ void deferred_prep(int j, uint32_t tail, uint32_t lastmask, const uint32_t (&rh)[W],
                                              const uint32_t (&rl)[W], const uint32_t (&gh)[NP][W],
                                              const uint32_t (&gl)[NP][W], FinishPrep<NP> &pr);
template <int W, int NP>
__device__ __forceinline__ void deferred_finish(const FilterArgs &a, uint32_t K, uint32_t tail,
                                                uint32_t lastmask, const uint32_t (&acc)[NP][W],
                                                const FinishPrep<NP> &pr, uint32_t (&count)[NP]);

// deferred_counts at every shift count K = Klo .. K of a threshold sweep in
// one pass: the 2k+1 masks of shift count k are those of k-1 and the two
// shifted by k, so the running AND after step k is the AND of shift count k,
// and the once-per-pair finish (end values, erosion, corrections, count)
// runs on it at each k from Klo on; emit(k, count) receives the counts.  The
// finish's shift-independent terms are prepared once per pair.
template <int W, int NP, typename Emit>
__device__ __forceinline__ void deferred_sweep_counts(const FilterArgs &a, uint32_t m, uint32_t K,
                                                      const uint32_t (&rh)[W], const uint32_t (&rl)[W],
                                                      const uint32_t (&gh)[NP][W], const uint32_t (&gl)[NP][W],
                                                      uint32_t (&count)[NP], uint32_t Klo, Emit emit) {
  const uint32_t tail = m - 32u * (W - 1);  // 1..32 bases in the last word
  const uint32_t lastmask = tail >= 32 ? 0xffffffffu : ((1u << tail) - 1u);

  uint32_t acc[NP][W], d[W], dn[W];
  FinishPrep<NP> pr;
#pragma unroll
  for (int j = 0; j < NP; ++j) deferred_prep<W, NP>(j, tail, lastmask, rh, rl, gh, gl, pr);
  auto finish = [&](uint32_t Kf) { deferred_finish<W, NP>(a, Kf, tail, lastmask, acc, pr, count); };
  // dilation of a mask: bit i <- d[i-1] | d[i] | d[i+1], zeros outside the words
  auto dil = [&](const uint32_t (&dd)[W], int w) -> uint32_t {
    const uint32_t below = __funnelshift_l(w > 0 ? dd[w - 1] : 0u, dd[w], 1);
    const uint32_t above = __funnelshift_r(dd[w], w + 1 < W ? dd[w + 1] : 0u, 1);
    return dd[w] | below | above;
  };
#pragma unroll
  for (int j = 0; j < NP; ++j) {
#pragma unroll
    for (int w = 0; w < W; ++w) d[w] = (rh[w] ^ gh[j][w]) | (rl[w] ^ gl[j][w]);
#pragma unroll
    for (int w = 0; w < W; ++w) acc[j][w] = dil(d, w);  // shift 0
  }
  if (Klo == 0) {
    finish(0);
    emit(0u, count);
  }
  {
    uint32_t ph[W], pl[W], nh[W], nl[W];
#pragma unroll
    for (int w = 0; w < W; ++w) {
      ph[w] = nh[w] = rh[w];
      pl[w] = nl[w] = rl[w];
    }
    // The vacated positions of each shifted mask are ORed into its difference
    // vector before the dilation: dil(d | V) = dil(d) | dil(V), the mask ORed
    // with its dilated vacated set.
    uint32_t lead = 0u;               // mask +k: positions 0..k-1 (word 0)
    uint32_t tv_hi = ~lastmask;       // mask -k: positions >= m-k (and >= m), top word
    uint32_t tv_lo = 0u;              // and the word below it
    for (uint32_t k = 1; k <= K; ++k) {
#pragma unroll
      for (int w = W - 1; w >= 0; --w) {
        ph[w] = __funnelshift_l(w > 0 ? ph[w - 1] : 0u, ph[w], 1);
        pl[w] = __funnelshift_l(w > 0 ? pl[w - 1] : 0u, pl[w], 1);
      }
#pragma unroll
      for (int w = 0; w < W; ++w) {
        nh[w] = __funnelshift_r(nh[w], w + 1 < W ? nh[w + 1] : 0u, 1);
        nl[w] = __funnelshift_r(nl[w], w + 1 < W ? nl[w + 1] : 0u, 1);
      }
      lead = 2u * lead + 1u;
      tv_lo = __funnelshift_r(tv_lo, tv_hi, 1);
      tv_hi = __funnelshift_r(tv_hi, 0xffffffffu, 1);
#pragma unroll
      for (int j = 0; j < NP; ++j) {
#pragma unroll
        for (int w = 0; w < W; ++w) {
          const uint32_t vp = w == 0 ? lead : 0u;
          const uint32_t vn = w == W - 1 ? tv_hi : (w == W - 2 ? tv_lo : 0u);
          d[w] = (ph[w] ^ gh[j][w]) | vp | (pl[w] ^ gl[j][w]);
          dn[w] = (nh[w] ^ gh[j][w]) | vn | (nl[w] ^ gl[j][w]);
        }
        d[W - 1] &= lastmask;  // the +k copy carries read bases past m
#pragma unroll
        for (int w = 0; w < W; ++w) acc[j][w] &= dil(d, w) & dil(dn, w);
      }
      if (k >= Klo) {
        finish(k);
        emit(k, count);
      }
    }
  }
}

// The shift-count-independent terms of the once-per-pair end: per pair, the
// compare of window base 0 with the read's first bases (the AND one base
// below position 0), of window base m-1 with the read's last bases (the AND
// one base above m-1, when m fills the words), and the correction words at
// both ends before they are limited to the positions of a shift count.
template <int NP>
struct FinishPrep {
  // The AND one base below position 0 is 1 at shift count K iff K < t0 (t0:
  // the number of trailing 1s of the compare of window base 0 with the
  // read's first bases); likewise above m-1 with tm.
  uint32_t t0[NP], tm[NP];
  uint32_t lx[NP], ly[NP];  // low end: bit p set where a correction clears position p (from mask p) / p+1 (mask p-1)
  uint32_t hx[NP], hy[NP];  // high end, mirrored (bit j: position m-1-j), bit-reversed; hy pre-shifted by 1
};

// The high-end words are kept bit-reversed, so that each finish reverses one
// mask instead of one word per pair.
template <int W, int NP>
__device__ __forceinline__ void deferred_prep(int j, uint32_t tail, uint32_t lastmask, const uint32_t (&rh)[W],
                                              const uint32_t (&rl)[W], const uint32_t (&gh)[NP][W],
                                              const uint32_t (&gl)[NP][W], FinishPrep<NP> &pr) {
  // The read's last 32 bases mirrored: bit j is position m-1-j (positions
  // below 0 read as code 00).  The high end's terms are the low end's
  // formulas on mirrored vectors, in 32-bit words.
  const uint32_t xrh = __funnelshift_rc(W >= 2 ? rh[W >= 2 ? W - 2 : 0] : 0u, rh[W - 1], tail);
  const uint32_t xrl = __funnelshift_rc(W >= 2 ? rl[W >= 2 ? W - 2 : 0] : 0u, rl[W - 1], tail);
  const uint32_t b0h = 0u - (xrh >> 31), b0l = 0u - (xrl >> 31);                // R[m-1]
  const uint32_t b1h = 0u - ((xrh >> 30) & 1u), b1l = 0u - ((xrl >> 30) & 1u);  // R[m-2]
  const uint32_t r0h = 0u - (rh[0] & 1u), r0l = 0u - (rl[0] & 1u);              // R[0]
  const uint32_t r1h = 0u - ((rh[0] >> 1) & 1u), r1l = 0u - ((rl[0] >> 1) & 1u);  // R[1]
  {
    // Window base 0 against R[i] (bit i), every non-positive shift.
    const uint32_t g0h = 0u - (gh[j][0] & 1u), g0l = 0u - (gl[j][0] & 1u);
    pr.t0[j] = __ffs(~((rh[0] ^ g0h) | (rl[0] ^ g0l))) - 1u;  // 0xFFFFFFFF (all 1s): every K
    // The window's last 32 bases mirrored.
    const uint32_t mgh = __brev(__funnelshift_rc(W >= 2 ? gh[j][W >= 2 ? W - 2 : 0] : 0u, gh[j][W - 1], tail));
    const uint32_t mgl = __brev(__funnelshift_rc(W >= 2 ? gl[j][W >= 2 ? W - 2 : 0] : 0u, gl[j][W - 1], tail));
    // Window base m-1 against R[m-1-i] (bit i), every non-negative shift;
    // used only when m fills the words.
    pr.tm[j] = 0u;
    if (tail == 32) {
      const uint32_t gmh = 0u - (mgh & 1u), gml = 0u - (mgl & 1u);
      pr.tm[j] = __ffs(~((__brev(xrh) ^ gmh) | (__brev(xrl) ^ gml))) - 1u;
    }
    {  // low end (positions 1..K+1, word 0)
      const uint32_t v0 = W == 1 ? lastmask : 0xffffffffu;
      const uint32_t a0 = (gh[j][0] ^ r0h) | (gl[j][0] ^ r0l);
      const uint32_t a1 = ((gh[j][0] ^ r1h) | (gl[j][0] ^ r1l)) & v0;
      const uint32_t vac = gh[j][0] | gl[j][0];
      const uint32_t c1 = (vac << 2) | (vac << 1) | a0;
      const uint32_t c2 = (vac << 1) | a0 | (a1 >> 1);
      pr.lx[j] = ~(c1 & c2);
      pr.ly[j] = ~c2 << 1;  // applied one position up
    }
    {  // high end (positions m-K-2..m-2), mirrored; kept bit-reversed
      const uint32_t a0 = (mgh ^ b0h) | (mgl ^ b0l);
      const uint32_t a1 = (mgh ^ b1h) | (mgl ^ b1l);
      const uint32_t vac = mgh | mgl;
      const uint32_t c1 = (vac << 2) | (vac << 1) | a0;
      const uint32_t c2 = (vac << 1) | a0 | (a1 >> 1);
      pr.hx[j] = __brev(~(c1 & c2));
      pr.hy[j] = __brev(~c2) >> 1;  // applied one position down (mirrored)
    }
  }
}

// The once-per-pair end of deferred_sweep_counts for shift count K: the
// AND's values one base outside each end, the erosion, the corrections next
// to the vacated runs and the count (acc is read, not changed), as at the end
// of deferred_counts.
template <int W, int NP>
__device__ __forceinline__ void deferred_finish(const FilterArgs &a, uint32_t K, uint32_t tail,
                                                uint32_t lastmask, const uint32_t (&acc)[NP][W],
                                                const FinishPrep<NP> &pr, uint32_t (&count)[NP]) {
  // ---- once per pair: end values of the AND, corrections, final erosion ----
  const uint32_t r1k = (2u << K) - 2u;  // bits 1..K
  const uint32_t r2k = r1k << 1;         // bits 2..K+1
  const uint32_t r1kr = __brev(r1k);     // bits 1..K, mirrored
  const uint32_t r2kr = r1kr >> 1;       // bits 2..K+1, mirrored
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    // AND one base below position 0 (every non-positive shift compares G[0]
    // with R[i], i = 0..K) and, when m fills the words, above m-1.
    const uint32_t lo0 = K < pr.t0[j] ? 0x80000000u : 0u;
    const uint32_t vtop = (tail == 32 && K < pr.tm[j]) ? 1u : 0u;
    uint32_t f[W];
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const uint32_t lo_in = w > 0 ? acc[j][w - 1] : lo0;
      const uint32_t hi_in = w + 1 < W ? acc[j][w + 1] : vtop;
      f[w] = acc[j][w] & __funnelshift_l(lo_in, acc[j][w], 1) & __funnelshift_r(acc[j][w], hi_in, 1);
    }
    // Low-end corrections (positions 1..K+1, word 0).
    f[0] &= ~((pr.lx[j] & r1k) | (pr.ly[j] & r2k));
    // High-end corrections (positions m-K-2..m-2), mapped back from the
    // mirrored words: bit b of nc is position m-32+b; the last word also
    // drops the positions past m.
    {
      const uint32_t nc = (pr.hx[j] & r1kr) | (pr.hy[j] & r2kr);
      f[W - 1] &= ~(nc >> (32u - tail)) & lastmask;
      if (W >= 2 && tail < 32) f[W >= 2 ? W - 2 : 0] &= ~(nc << tail);
    }

    uint32_t c = 0;
    if (a.count_mode == GK_COUNT_POPCOUNT) {
#pragma unroll
      for (int w = 0; w < W; ++w) c += __popc(f[w]);
    } else {
#pragma unroll
      for (int w = 0; w < W; ++w) c += __popc(f[w] & ~((f[w] << 1) & 0xEEEEEEEEu));
    }
    count[j] = c;
  }
}

// Window planes of a loaded pair, zero past m.
template <int W>
__device__ __forceinline__ void window_planes(const PairData<W> &x, uint32_t (&gh)[W], uint32_t (&gl)[W]) {
  const uint32_t tail = x.m - 32u * (W - 1);
  const uint32_t lastmask = tail >= 32 ? 0xffffffffu : ((1u << tail) - 1u);
  const uint32_t sh = x.off & 31;
#pragma unroll
  for (int w = 0; w < W; ++w) {
    gh[w] = __funnelshift_r(x.g[w].x, x.g[w + 1].x, sh);
    gl[w] = __funnelshift_r(x.g[w].y, x.g[w + 1].y, sh);
  }
  gh[W - 1] &= lastmask;
  gl[W - 1] &= lastmask;
}

// Read planes of a loaded pair, zero past m.
template <int W>
__device__ __forceinline__ void read_planes(const PairData<W> &x, uint32_t (&rh)[W], uint32_t (&rl)[W]) {
  const uint32_t tail = x.m - 32u * (W - 1);
  const uint32_t lastmask = tail >= 32 ? 0xffffffffu : ((1u << tail) - 1u);
#pragma unroll
  for (int w = 0; w < W; ++w) {
    rh[w] = x.r[w].x;
    rl[w] = x.r[w].y;
  }
  rh[W - 1] &= lastmask;
  rl[W - 1] &= lastmask;
}

template <int W>
__device__ __forceinline__ void pair_planes(const PairData<W> &x, uint32_t (&rh)[W], uint32_t (&rl)[W],
                                            uint32_t (&gh)[W], uint32_t (&gl)[W]) {
  read_planes<W>(x, rh, rl);
  window_planes<W>(x, gh, gl);
}

// The same as S stripes.
template <int W, int S>
__device__ __forceinline__ void striped_window(const PairData<W> &x, uint32_t (&gh)[S], uint32_t (&gl)[S]) {
  uint32_t h[W], l[W];
  window_planes<W>(x, h, l);
  stripe_linear<W, S>(h, gh);
  stripe_linear<W, S>(l, gl);
}
template <int W, int S>
__device__ __forceinline__ void striped_read(const PairData<W> &x, uint32_t (&rh)[S], uint32_t (&rl)[S]) {
  uint32_t h[W], l[W];
  read_planes<W>(x, h, l);
  stripe_linear<W, S>(h, rh);
  stripe_linear<W, S>(l, rl);
}

// Counts at one shift count K (0 .. 30, below m) of NP pairs that share one
// read (x0's), striped with deferred erosion.
template <int W, int S, int NP, bool WHOLE>
__device__ __forceinline__ void striped_counts(const PairData<W> &x0, const PairData<W> &x1, uint32_t m, uint32_t K,
                                               int count_mode, uint32_t (&count)[NP]) {
  uint32_t rh[S], rl[S], gh[NP][S], gl[NP][S], h[W], l[W], wh[W], wl[W], lo[NP], hi[NP];
  read_planes<W>(x0, h, l);
  stripe_linear<W, S>(h, rh);
  stripe_linear<W, S>(l, rl);
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    window_planes<W>(j ? x1 : x0, wh, wl);
    end_corrections<W>(m, K, h, l, wh, wl, lo[j], hi[j]);
    stripe_linear<W, S>(wh, gh[j]);
    stripe_linear<W, S>(wl, gl[j]);
  }
  striped_deferred<W, S, NP, WHOLE>(m, K, count_mode, rh, rl, gh, gl, lo, hi, count);
}

// One pair's count at the launch's one length (uniform: its masks stay in
// scalar registers) and shift count K <= 30, striped.
template <int W, int S>
__device__ __forceinline__ uint32_t filter_loaded_striped(const FilterArgs &a, const PairData<W> &x, uint32_t K) {
  uint32_t c[1];
  if (a.m % S == 0)
    striped_counts<W, S, 1, true>(x, x, a.m, K, a.count_mode, c);
  else
    striped_counts<W, S, 1, false>(x, x, a.m, K, a.count_mode, c);
  return c[0];
}

template <int W, bool DIRECT = false>
__device__ __forceinline__ uint32_t filter_loaded_deferred(const FilterArgs &a, const PairData<W> &x) {
  uint32_t rh[W], rl[W], gh[1][W], gl[1][W], count[1];
  pair_planes<W>(x, rh, rl, gh[0], gl[0]);
  deferred_counts<W, 1, DIRECT>(a, x.m, min(x.e, x.m - 1), rh, rl, gh, gl, count);
  return count[0];
}

// Resident blocks per SM the compiler must allow: of 256 threads in the
// compacting loop, of 128 elsewhere.  One thread per pair: small reads keep
// enough registers free for 40 warps per SM, which hides the dependent loads
// of a pair (ids, then read and window words); W = 5 and 6 fit 32 and 24 warps
// without spilling (at 150 bp, e = 0..2, 32 warps run 9-18% faster than 16).
// The compacting loop stages its words with cp.async and carries a chunk
// pipeline, so it keeps fewer resident warps.
// The striped loops use 64 registers (S <= 4), 80 (S = 5), 91 (S = 8; 128 in
// the compacting loop) and 128 (S = 11).
template <int W, bool COMPACT, int S = 0>
struct MinBlocks {
  static constexpr int value =
      S > 0 ? (COMPACT ? 1 : 2) * (S <= 4 ? 4 : (S == 5 ? 3 : 2))
      : COMPACT ? (W <= 2 ? 5 : (W <= 4 ? 4 : (W <= 6 ? 3 : (W <= 8 ? 2 : 1))))
              : (W <= 2 ? 12 : (W <= 4 ? 10 : (W == 5 ? 8 : (W == 6 ? 6 : (W <= 8 ? 4 : 2)))));
};

// Status of a loaded pair: 0 filter, 1 undefined (N in read or window),
// 2 invalid.
template <int W>
__device__ __forceinline__ int pair_status(const FilterArgs &a, const PairData<W> &x) {
  int status = x.status;
  if (status == 0 && a.m > 0) {
    if (x.nflag) status = 1;
    if (a.ref_nidx) {  // a valid pair's window ends below 2^32
      const uint32_t q = x.ni.x >> (x.off & 31);
      const uint32_t first = q ? x.off + (uint32_t)(__ffs(q) - 1) : x.ni.y;
      if (first < x.off + a.m) status = 1;
    }
  }
  return status;
}

// SWEEP (VARIANT 3): the outcome goes to the row of every threshold.
template <bool SWEEP = false>
__device__ __forceinline__ void write_trivial(const FilterArgs &a, uint64_t p, int status) {
  const uint32_t rows = SWEEP ? a.sweep_hi - a.fixed_e + 1 : 1;
  uint8_t *acc = a.accept + p;
  if (a.result_byte) {
    const uint8_t b = status == 0 ? 0 : (status == 1 ? GK_RESULT_UNDEFINED : GK_RESULT_INVALID);
    for (uint32_t i = 0; i < rows; ++i, acc += a.out_stride) *acc = b;
    return;
  }
  uint16_t *ed = a.edits + p;
  const uint8_t acc_v = status != 2;
  const uint16_t ed_v = status == 0 ? 0 : (status == 1 ? GK_EDITS_UNDEFINED : GK_EDITS_INVALID);
  for (uint32_t i = 0; i < rows; ++i, acc += a.out_stride, ed += a.out_stride) {
    *acc = acc_v;
    *ed = ed_v;
  }
}

// The result of a filtered pair: accept bit and count, or the result byte.
__device__ __forceinline__ void write_count(const FilterArgs &a, uint64_t p, uint32_t count, uint32_t e) {
  if (a.result_byte) {
    a.accept[p] = (uint8_t)min(count, GK_RESULT_MAX_COUNT);
    return;
  }
  a.accept[p] = count <= e;
  a.edits[p] = (uint16_t)count;
}

// Threshold sweep of one loaded pair (VARIANT 3): thresholds e = a.fixed_e ..
// a.sweep_hi have shift counts K = min(e, m-1); the shift loop runs once to
// the largest and the results of each K go to its rows (every e >= m-1
// shares K = m-1).  S > 0: striped in S words, else linear with deferred
// erosion.
template <int W, int S>
__device__ __forceinline__ void sweep_and_write(const FilterArgs &a, uint64_t p, const PairData<W> &x) {
  const uint32_t e_lo = a.fixed_e, e_hi = a.sweep_hi, kmax = x.m - 1;
  const uint32_t Klo = min(e_lo, kmax), Khi = min(e_hi, kmax);
  // The rows come in order, one per K and, at K = m-1, all that are left:
  // their pointers advance by a row each.
  uint8_t *acc_row = a.accept + p;
  uint16_t *ed_row = a.edits + p;
  auto emit = [&](uint32_t K, const uint32_t (&c)[1]) {
    const uint32_t last = K == kmax ? e_hi : K;
    uint32_t e = max(K, e_lo);
#pragma unroll 1
    do {
      if (a.result_byte) {
        *acc_row = (uint8_t)min(c[0], GK_RESULT_MAX_COUNT);
      } else {
        *acc_row = c[0] <= e;
        *ed_row = (uint16_t)c[0];
      }
      acc_row += a.out_stride;
      ed_row += a.out_stride;
    } while (++e <= last);
  };
  if constexpr (S > 0) {
    uint32_t rh[S], rl[S], gh[1][S], gl[1][S];
    striped_read<W, S>(x, rh, rl);
    striped_window<W, S>(x, gh[0], gl[0]);
    if (x.m % S == 0)
      striped_exact<W, S, 1, true>(x.m, Klo, Khi, a.count_mode, rh, rl, gh, gl, emit);
    else
      striped_exact<W, S, 1, false>(x.m, Klo, Khi, a.count_mode, rh, rl, gh, gl, emit);
  } else {
    uint32_t rh[W], rl[W], gh[1][W], gl[1][W], count[1];
    pair_planes<W>(x, rh, rl, gh[0], gl[0]);
    deferred_sweep_counts<W, 1>(a, x.m, Khi, rh, rl, gh, gl, count, Klo, emit);
  }
}

template <int W, int VARIANT, int S = 0>
__device__ __forceinline__ void filter_and_write(const FilterArgs &a, uint64_t p, const PairData<W> &x) {
  if constexpr (VARIANT == 3) {
    sweep_and_write<W, S>(a, p, x);
  } else {
    uint32_t count;
    if constexpr (S > 0) {
      count = filter_loaded_striped<W, S>(a, x, min(a.fixed_e, a.m - 1));
    } else if constexpr (S < 0) {
      uint32_t rh[W], rl[W], gh[1][W], gl[1][W], c[1];
      pair_planes<W>(x, rh, rl, gh[0], gl[0]);
      overlap_counts<W, 1, -1>(a.m, min(a.fixed_e, a.m - 1), a.count_mode, rh, rl, gh, gl, c);
      count = c[0];
    } else if constexpr (VARIANT == 6) {  // one form per warp
      count = __any_sync(__activemask(), min(x.e, a.m - 1) > 30) ? filter_loaded<W, false>(a, x)
                                                                 : filter_loaded_deferred<W>(a, x);
    } else
      count = VARIANT == 4   ? filter_loaded_deferred<W, true>(a, x)
              : VARIANT == 2 ? filter_loaded_deferred<W>(a, x)
                             : filter_loaded<W, VARIANT == 1>(a, x);
    write_count(a, p, count, x.e);
  }
}

// The classify phase of the compacting loop, in two steps so that the loads
// of one chunk are in flight while the warp works on another.
// ChunkLoads holds one lane's pair of a chunk: its ids and, for a valid pair,
// the read's N flag and the N index word of its window (loaded together).
struct ChunkLoads {
  uint32_t rid, off;
  uint32_t nflag;
  uint2 ni;
  int state;  // -1 no pair, 2 invalid, 3 empty read, 0 defined unless N
};

__device__ __forceinline__ void chunk_issue(const FilterArgs &a, ChunkLoads &x) {
  x.nflag = 0;
  x.ni = make_uint2(0u, 0xffffffffu);
  if (x.state < 0) return;
  if (x.rid > a.rid_last || x.off >= a.off_end) {
    x.state = 2;
  } else if (a.m == 0) {
    x.state = 3;
  } else {
    x.state = 0;
    if (a.read_nflag) x.nflag = a.read_nflag[x.rid];
    if (a.ref_nidx) x.ni = a.ref_nidx[x.off >> 5];
  }
}

// 0 filter, 1 undefined, 2 invalid, 3 empty read, -1 no pair.
__device__ __forceinline__ int chunk_status(const FilterArgs &a, const ChunkLoads &x) {
  if (x.state != 0) return x.state;
  if (x.nflag) return 1;
  const uint32_t q = x.ni.x >> (x.off & 31);
  const uint32_t first = q ? x.off + (uint32_t)(__ffs(q) - 1) : x.ni.y;
  return first < x.off + a.m ? 1 : 0;
}

__device__ __forceinline__ void chunk_ids(const FilterArgs &a, uint64_t c, uint64_t n_chunks, int lane,
                                          uint32_t &rid, uint32_t &off, int &state) {
  const uint64_t p = c * 32 + lane;
  state = -1;
  if (c < n_chunks && p < a.n_pairs) {
    rid = a.pair_read[p];
    off = a.pair_off[p];
    state = 0;
  }
}

// 8-byte asynchronous global -> shared copy (bypasses registers) and its
// group fences.
__device__ __forceinline__ void cp_async8(void *smem_dst, const void *gsrc) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

constexpr int kFilterWarps = kFilterThreads / 32, kQueueWarps = kQueueThreads / 32;

// Words of one staged batch (32 pairs): W read words and W + 1 window words
// per pair, stored word-major ([word][lane]) so that lanes touch consecutive
// 8-byte slots.  Two batches per warp are staged at a time.
template <int W>
constexpr int kStageWords = (2 * W + 1) * 32;
template <int W>
constexpr size_t compact_smem_bytes() {
  return (size_t)kQueueWarps * 2 * kStageWords<W> * sizeof(uint2);
}

// VARIANT 0: any thresholds; 1: every shift count of the launch is < 32;
// 2: edge OR on and one threshold in 2..30, deferred erosion; 3: edge OR on,
// a sweep of thresholds up to 30 (sweep_and_write).  2 and 3 are striped in S
// words (S > 0), 2 and 4 in overlapping words (S = -1, shift counts up to
// kOverlapMax) or linear (S = 0).  6: edge OR on, per-pair thresholds in pair
// order, deferred erosion where a warp's shift counts allow it.
//
// COMPACT false: one thread per pair.  COMPACT true (inputs with many
// undefined pairs): persistent warps take 32 pairs at a time (their ids
// loaded one chunk ahead), write the trivial outcomes at once and queue the
// pairs that need filtering in a 64-slot per-warp shared queue.  Each full
// batch of 32 queued pairs has its read and window words copied into shared
// memory by cp.async while the warp filters the previous batch, so that no
// lane idles next to an undefined pair and the word loads of one batch hide
// behind the arithmetic of the other.  Dynamic shared memory:
// compact_smem_bytes<W>().
template <int W, int VARIANT, bool COMPACT, int S = 0>
__global__ void __launch_bounds__(COMPACT ? kQueueThreads : kFilterThreads, MinBlocks<W, COMPACT, S>::value)
    filter_kernel(const FilterArgs a) {
  if (!COMPACT) {
    const uint64_t p = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    const bool active = p < a.n_pairs;
    PairData<W> cur;
    cur.status = 0;
    if (active) load_pair<W>(a, p, cur);
    if (a.err_count) {
      const unsigned bad = __ballot_sync(0xffffffffu, active && cur.status == 2);
      if (bad && (threadIdx.x & 31) == 0) atomicAdd(a.err_count, (unsigned)__popc(bad));
    }
    if (!active) return;
    const int status = pair_status<W>(a, cur);
    if (status != 0 || a.m == 0) {
      write_trivial<VARIANT == 3>(a, p, status);
      return;
    }
    filter_and_write<W, VARIANT, S>(a, p, cur);
    return;
  }
  extern __shared__ uint2 stage_all[];
  __shared__ uint32_t q_p[kQueueWarps][64], q_rid[kQueueWarps][64], q_off[kQueueWarps][64];
  // A sweep writes a settled pair to every row: those queue too, so that whole
  // warps write them (10M pairs of 150 bp, 26% undefined, e = 0..15: 786 -> 766
  // us).
  constexpr bool kSweep = VARIANT == 3;
  __shared__ uint32_t t_p[kSweep ? kQueueWarps : 1][64];
  __shared__ uint8_t t_status[kSweep ? kQueueWarps : 1][64];
  uint32_t tn = 0;  // warp-uniform length of the settled pairs' queue
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  uint2 *stage = stage_all + wib * 2 * kStageWords<W>;
  const uint64_t n_chunks = (a.n_pairs + 31) / 32;
  const uint64_t n_warps = (uint64_t)gridDim.x * kQueueWarps;
  uint64_t c = blockIdx.x * (uint64_t)kQueueWarps + wib;
  // Load pipeline over this warp's chunks.  Wide reads (W >= 7, registers to
  // spare) run it two deep: while the warp classifies chunk c and filters,
  // the N information of its next chunk and the ids of the chunk after are
  // in flight.  Narrower reads keep one deep (the ids of the next chunk), as
  // two deep spills registers there and measured slower at 150 bp.
  constexpr bool kDeep = W >= 7;
  ChunkLoads cur;
  cur.rid = cur.off = 0;
  chunk_ids(a, c, n_chunks, lane, cur.rid, cur.off, cur.state);
  uint32_t next_rid = 0, next_off = 0;
  int next_state = -1;
  if (kDeep) {
    chunk_issue(a, cur);
    chunk_ids(a, c + n_warps, n_chunks, lane, next_rid, next_off, next_state);
  }
  uint32_t qn = 0;         // warp-uniform queue length
  int pend = -1;           // stage buffer of the batch in flight, or none
  bool pend_has = false;   // this lane holds a pair of that batch
  uint32_t pend_p = 0, pend_off = 0, pend_e = 0;
  auto filter_staged = [&]() {
    if (!pend_has) return;
    const uint2 *sb = stage + pend * kStageWords<W>;
    PairData<W> x;
    x.m = a.m;
    x.off = pend_off;
    x.e = pend_e;
    x.status = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) x.r[w] = sb[w * 32 + lane];
#pragma unroll
    for (int w = 0; w <= W; ++w) x.g[w] = sb[(W + w) * 32 + lane];
    filter_and_write<W, VARIANT, S>(a, pend_p, x);
  };
  for (;; c += n_warps) {
    const bool more = c < n_chunks;
    if (more) {
      const uint64_t p = c * 32 + lane;
      const bool active = p < a.n_pairs;
      int status;
      const uint32_t rid = cur.rid, off = cur.off;
      if (kDeep) {
        status = chunk_status(a, cur);
        cur.rid = next_rid;
        cur.off = next_off;
        cur.state = next_state;
        chunk_issue(a, cur);
        chunk_ids(a, c + 2 * n_warps, n_chunks, lane, next_rid, next_off, next_state);
      } else {
        ChunkLoads x = cur;
        chunk_ids(a, c + n_warps, n_chunks, lane, cur.rid, cur.off, cur.state);
        chunk_issue(a, x);
        status = chunk_status(a, x);
      }
      if (a.err_count) {
        const unsigned bad = __ballot_sync(0xffffffffu, status == 2);
        if (bad && lane == 0) atomicAdd(a.err_count, (unsigned)__popc(bad));
      }
      const bool settled = status > 0 && active;
      if constexpr (kSweep) {
        const unsigned set = __ballot_sync(0xffffffffu, settled);
        if (settled) {
          const uint32_t slot = tn + __popc(set & ((1u << lane) - 1u));
          t_p[wib][slot] = (uint32_t)p;
          t_status[wib][slot] = status == 3 ? 0 : (uint8_t)status;
        }
        tn += __popc(set);
        __syncwarp();
        if (tn >= 32) {
          tn -= 32;
          write_trivial<true>(a, t_p[wib][tn + lane], t_status[wib][tn + lane]);
          __syncwarp();
        }
      } else if (settled) {
        write_trivial(a, p, status == 3 ? 0 : status);
      }
      const unsigned need = __ballot_sync(0xffffffffu, status == 0);
      if ((need >> lane) & 1u) {
        const uint32_t slot = qn + __popc(need & ((1u << lane) - 1u));
        q_p[wib][slot] = (uint32_t)p;
        q_rid[wib][slot] = rid;
        q_off[wib][slot] = off;
      }
      qn += __popc(need);
      __syncwarp();
    }
    // One place filters, the drain included: the code of a second one would
    // not fit the instruction cache beside it.
    while (qn >= 32 || (!more && (qn > 0 || pend >= 0))) {
      const uint32_t take = qn < 32 ? qn : 32;
      const bool has = (uint32_t)lane < take;
      const int nb = pend == 0 ? 1 : 0;
      uint32_t np = 0, noff = 0, ne = a.fixed_e;
      if (has) {
        const uint32_t i = qn - take + lane;
        np = q_p[wib][i];
        const uint32_t rid = q_rid[wib][i];
        noff = q_off[wib][i];
        // a queued pair is valid: its read row holds W words and its window
        // words off/32 .. off/32 + W lie inside the genome's n_words + 2
        const uint2 *rp = a.reads + (uint64_t)rid * a.stride_words;
        const uint2 *gp = a.ref_hl + (noff >> 5);
        uint2 *sb = stage + nb * kStageWords<W>;
#pragma unroll
        for (int w = 0; w < W; ++w) cp_async8(sb + w * 32 + lane, rp + w);
#pragma unroll
        for (int w = 0; w <= W; ++w) cp_async8(sb + (W + w) * 32 + lane, gp + w);
        if (a.pair_e) ne = a.pair_e[np];
      }
      cp_async_commit();
      __syncwarp();
      qn -= take;
      if (pend >= 0) {
        cp_async_wait<1>();  // the previous batch's copies have landed
        filter_staged();
      }
      pend = take > 0 ? nb : -1;
      pend_has = has;
      pend_p = np;
      pend_off = noff;
      pend_e = ne;
    }
    if (!more) break;
  }
  if (kSweep && (uint32_t)lane < tn) write_trivial<true>(a, t_p[wib][lane], t_status[wib][lane]);
}

// The two-pairs-per-thread kernel gathers in 8-byte loads except at a
// compile-time shift count 0: 16-byte loads (load_words_wide) measured 2-4%
// slower at every other shift count at 100 bp.
constexpr bool kPair2Wide = false;

// Resident blocks of 128 threads per SM of the two-pairs-per-thread kernel: 8
// (64 registers, a few spilled) measured faster than 6 (80 registers, no spill) at every
// threshold 1..10 and in the 0..10 sweep at 100 bp on GB300 (e = 2: 53.3 ->
// 57.5 Gpairs/s; the sweep 1.307 -> 1.280 ms), the same at e = 0.
template <int W>
struct MinBlocks2 {
  static constexpr int value = 8;
};

// Deferred erosion (VARIANT 2), two pairs per thread: pairs 2t and 2t+1.  When both are filtered and share their read
// (the candidates of one read usually sit next to each other), the read is
// loaded once and its shifted copies serve both windows: a shift step costs
// about 13W integer operations per pair instead of 15W.  Otherwise each pair
// is filtered on its own.  VARIANT 4: one threshold whose shift count KC
// (0..2, below m) is a compile-time constant, so the shift steps unroll and
// the end corrections of K = 0 vanish.
//
// S > 0: striped; of pairs that do not share a read the second is then loaded
// anew, as in the sweep.  S = -1: in overlapping words (overlap.cuh).
template <int W, int VARIANT, int KC = -1, int S = 0>
__global__ void __launch_bounds__(kFilterThreads, S == 5 ? 6 : MinBlocks2<W>::value)
    filter_pair2_kernel(const FilterArgs a) {
  const uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  const uint64_t p0 = 2 * t, p1 = p0 + 1;
  const bool act0 = p0 < a.n_pairs, act1 = p1 < a.n_pairs;
  PairData<W> x0, x1;
  x0.status = x1.status = 0;
  // Shift count 0: read and window in 16-byte loads (e0 82.3 -> 85.4 Gpairs/s
  // at 100 bp); 1 and 2: the window's last word loaded only when the window
  // reaches into it (e1 68.2 -> 70.1, e2 58.7 -> 59.4); each measured slower
  // with the other's choice.
  constexpr bool kWide = kPair2Wide || KC == 0, kSkipLast = KC >= 1;
  if (act0) load_pair<W, kWide, kSkipLast>(a, p0, x0);
  if (act1) load_pair<W, kWide, kSkipLast>(a, p1, x1, act0 ? &x0 : nullptr);
  if (a.err_count) {
    const unsigned b0 = __ballot_sync(0xffffffffu, act0 && x0.status == 2);
    const unsigned b1 = __ballot_sync(0xffffffffu, act1 && x1.status == 2);
    if ((b0 | b1) && (threadIdx.x & 31) == 0) atomicAdd(a.err_count, (unsigned)(__popc(b0) + __popc(b1)));
  }
  const int s0 = act0 ? pair_status<W>(a, x0) : -1;
  const int s1 = act1 ? pair_status<W>(a, x1) : -1;
  if (s0 > 0) write_trivial(a, p0, s0);
  if (s1 > 0) write_trivial(a, p1, s1);
  // One form per warp, as in sweep_pair2_kernel.
  const bool shared = s0 == 0 && s1 == 0 && x0.rid == x1.rid;
  if (!__any_sync(0xffffffffu, !shared && (s0 == 0 || s1 == 0))) {
    if (!shared) return;
    const uint32_t K = KC >= 0 ? (uint32_t)KC : min(a.fixed_e, a.m - 1);
    uint32_t count[2];
    if constexpr (S > 0) {
      if (a.m % S == 0)
        striped_counts<W, S, 2, true>(x0, x1, a.m, K, a.count_mode, count);
      else
        striped_counts<W, S, 2, false>(x0, x1, a.m, K, a.count_mode, count);
    } else {
      uint32_t rh[W], rl[W], gh[2][W], gl[2][W];
      pair_planes<W>(x0, rh, rl, gh[0], gl[0]);
      window_planes<W>(x1, gh[1], gl[1]);
      if constexpr (S < 0)
        overlap_counts<W, 2, KC>(a.m, K, a.count_mode, rh, rl, gh, gl, count);
      else
        deferred_counts<W, 2, (KC >= 0)>(a, a.m, K, rh, rl, gh, gl, count);
    }
    // The two pairs are adjacent: one 2-byte accept store and one 4-byte
    // count store when the buffers allow it.
    if (!a.result_byte && ((uintptr_t)a.accept & 1u) == 0 && ((uintptr_t)a.edits & 3u) == 0) {
      const uint32_t e = a.fixed_e;
      *reinterpret_cast<uint32_t *>(a.edits + p0) = count[0] | (count[1] << 16);
      *reinterpret_cast<uint16_t *>(a.accept + p0) =
          (uint16_t)((count[0] <= e ? 1u : 0u) | (count[1] <= e ? 0x100u : 0u));
    } else {
      write_count(a, p0, count[0], a.fixed_e);
      write_count(a, p1, count[1], a.fixed_e);
    }
  } else if constexpr (S > 0) {
#pragma unroll 1
    for (int j = 0; j < 2; ++j) {
      if ((j ? s1 : s0) != 0) continue;
      if (j) load_pair<W>(a, p1, x0);
      filter_and_write<W, VARIANT, S>(a, p0 + j, x0);
    }
  } else {
    if (s0 == 0) filter_and_write<W, VARIANT, S>(a, p0, x0);
    if (s1 == 0) filter_and_write<W, VARIANT, S>(a, p1, x1);
  }
}

// The threshold sweep, two pairs per thread (2t and 2t+1): when both are
// filtered and share their read, its shifted copies and their masks serve both
// windows, and each threshold's two results go out as one 2-byte and one
// 4-byte store.  Rows are addressed as a block's base plus a 32-bit offset, so
// that their advance is scalar work.  Of pairs that do not share a read the
// second is loaded anew (keeping both beside the shared form's registers
// spills).
// S: stripes, or 0 for the linear form.  Blocks per SM: 64 registers hold S <=
// 4 (3 blocks measured 1% slower at 100 bp), 80 S = 5 (2 blocks 7% slower at
// 150 bp; one pair per thread 12% slower).
template <int W, int S>
__global__ void __launch_bounds__(kFilterThreads, S == 5 ? 6 : 8) sweep_pair2_kernel(const FilterArgs a) {
  const uint64_t base = blockIdx.x * (uint64_t)(2 * kFilterThreads);
  const uint32_t lo = 2 * threadIdx.x;
  const uint64_t p0 = base + lo, p1 = p0 + 1;
  const bool act0 = p0 < a.n_pairs, act1 = p1 < a.n_pairs;
  PairData<W> x0, x1;
  x0.status = x1.status = 0;
  if (act0) load_pair<W>(a, p0, x0);
  if (act1) load_pair<W>(a, p1, x1, act0 ? &x0 : nullptr);
  if (a.err_count) {
    const unsigned b0 = __ballot_sync(0xffffffffu, act0 && x0.status == 2);
    const unsigned b1 = __ballot_sync(0xffffffffu, act1 && x1.status == 2);
    if ((b0 | b1) && (threadIdx.x & 31) == 0) atomicAdd(a.err_count, (unsigned)(__popc(b0) + __popc(b1)));
  }
  const int s0 = act0 ? pair_status<W>(a, x0) : -1;
  const int s1 = act1 ? pair_status<W>(a, x1) : -1;
  if (s0 > 0) write_trivial<true>(a, p0, s0);
  if (s1 > 0) write_trivial<true>(a, p1, s1);
  // One form per warp: pairs of different reads in a few lanes (a read's
  // candidates ending on an odd pair) would make it run both (10M pairs of 100
  // bp, 13 candidates per read, e = 0..10: 0.85 -> 0.48 ms).
  const bool shared = s0 == 0 && s1 == 0 && x0.rid == x1.rid;
  if (!__any_sync(0xffffffffu, !shared && (s0 == 0 || s1 == 0))) {
    if (!shared) return;
    const uint32_t e_lo = a.fixed_e, e_hi = a.sweep_hi, kmax = a.m - 1;
    const uint32_t Klo = min(e_lo, kmax), Khi = min(e_hi, kmax);
    // Pairs 2t and 2t+1 are adjacent in every row: packed stores when the
    // rows keep that alignment.
    const bool pack = (((uintptr_t)a.accept | (a.result_byte ? 0u : (uintptr_t)a.edits)) & 3u) == 0 &&
                      (a.out_stride & 1u) == 0;
    uint8_t *acc_row = a.accept + base;
    uint16_t *ed_row = a.edits + base;
    auto emit = [&](uint32_t K, const uint32_t (&c)[2]) {  // rows in order, as in sweep_and_write
      const uint32_t last = K == kmax ? e_hi : K;
      uint32_t e = max(K, e_lo);
#pragma unroll 1
      do {
        uint32_t b0 = c[0] <= e ? 1u : 0u, b1 = c[1] <= e ? 1u : 0u;
        if (a.result_byte) {
          b0 = min(c[0], GK_RESULT_MAX_COUNT);
          b1 = min(c[1], GK_RESULT_MAX_COUNT);
        } else if (pack) {
          *reinterpret_cast<uint32_t *>(ed_row + lo) = c[0] | (c[1] << 16);
        } else {
          ed_row[lo] = (uint16_t)c[0];
          ed_row[lo + 1] = (uint16_t)c[1];
        }
        if (pack) {
          *reinterpret_cast<uint16_t *>(acc_row + lo) = (uint16_t)(b0 | (b1 << 8));
        } else {
          acc_row[lo] = (uint8_t)b0;
          acc_row[lo + 1] = (uint8_t)b1;
        }
        acc_row += a.out_stride;
        ed_row += a.out_stride;
      } while (++e <= last);
    };
    if constexpr (S > 0) {
      uint32_t rh[S], rl[S], gh[2][S], gl[2][S];
      striped_read<W, S>(x0, rh, rl);
      striped_window<W, S>(x0, gh[0], gl[0]);
      striped_window<W, S>(x1, gh[1], gl[1]);
      if (a.m % S == 0)
        striped_exact<W, S, 2, true>(a.m, Klo, Khi, a.count_mode, rh, rl, gh, gl, emit);
      else
        striped_exact<W, S, 2, false>(a.m, Klo, Khi, a.count_mode, rh, rl, gh, gl, emit);
    } else {
      uint32_t rh[W], rl[W], gh[2][W], gl[2][W], count[2];
      pair_planes<W>(x0, rh, rl, gh[0], gl[0]);
      window_planes<W>(x1, gh[1], gl[1]);
      deferred_sweep_counts<W, 2>(a, a.m, Khi, rh, rl, gh, gl, count, Klo, emit);
    }
  } else {
#pragma unroll 1
    for (int j = 0; j < 2; ++j) {
      if ((j ? s1 : s0) != 0) continue;
      if (j) load_pair<W>(a, p1, x0);
      sweep_and_write<W, S>(a, p0 + j, x0);
    }
  }
}

// Classes of shift counts that a tile of pairs is sorted by: each K up to 30
// (deferred erosion) its own, above that steps that widen with K (31..62 by 2,
// 63..126 by 8, then by 16: at most an eighth of K, so that a warp's pairs still
// take about the same number of exact steps).
constexpr uint32_t kShiftClasses = 64, kExactClass = 31;  // kExactClass: K = 31, 32
__host__ __device__ __forceinline__ uint32_t shift_class(uint32_t K) {  // K <= 255
  return K <= 30 ? K : (K <= 62 ? 31u + (K - 31u) / 2u : (K <= 126 ? 47u + (K - 63u) / 8u : 55u + (K - 127u) / 16u));
}

// A counting sort's rank of each lane's class among the equal ones before it
// (class none: no rank), one counter update per class and warp.
__device__ __forceinline__ uint32_t class_rank(uint32_t cls, uint32_t none, uint32_t *s_n) {
  const uint32_t lane = threadIdx.x & 31u;
  const unsigned peers = __match_any_sync(0xffffffffu, cls);
  const int leader = __ffs(peers) - 1;
  uint32_t at = 0;
  if (cls != none && (int)lane == leader) at = atomicAdd(&s_n[cls], (unsigned)__popc(peers));
  return __shfl_sync(0xffffffffu, at, leader) + __popc(peers & ((1u << lane) - 1u));
}

// Counts per class into each class's first slot, the largest first (one warp,
// two classes per lane); returns the slots used in lane 31.
__device__ __forceinline__ uint32_t class_starts(uint32_t *s_n) {
  const uint32_t lane = threadIdx.x & 31u, c = kShiftClasses - 1u - 2u * lane;
  const uint32_t n0 = s_n[c], n1 = s_n[c - 1];
  uint32_t v = n0 + n1;
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t o = __shfl_up_sync(0xffffffffu, v, d);
    if (lane >= (uint32_t)d) v += o;
  }
  s_n[c] = v - n0 - n1;
  s_n[c - 1] = v - n1;
  return v;
}

// Per-pair thresholds with the edge OR on, one read length.  In pair order a
// warp takes as many shift steps as its largest threshold asks for.  Here a
// block takes a tile of pairs, writes the trivial outcomes, and sorts the
// others by shift count in shared memory (a counting sort over shift_class),
// so that a warp's pairs need about the same number of steps, of the deferred
// form (striped in S words where shift counts reach FROM; S = 0: linear) up to
// 30 and exact above.  Results are staged in shared memory and written in pair
// order.  A genome's undefined pairs drop out with the sort, so N-dense inputs
// need no queue.
//
// A tile keeps its order where the sort would cost more than it saves
// (worth_sorting).  It saves half the spread of the shift counts (a warp takes
// its largest) and, for lanes idle on settled pairs, their share of a pair's
// steps; it costs about two shift steps per pair in tiles of 512, half that in
// tiles of 1024, twice that in smaller ones, and twice again above 10 words,
// whose rows it gathers out of order.  The largest tiles are nearly always worth
// it and rank their pairs while the next batch loads.
//
// Measured on GB300, one pair per thread with exact erosion / always sorted and
// striped / here: 10M pairs of 150 bp, thresholds 3, 8 and 15 mixed 1112 / 441 /
// 446 us; 2M pairs with thresholds 0..2 of 100 bp 47 / 62 / 46, with threshold 2
// of 170 bp 62 / 109 / 57, of 300 bp 107 / 150 / 88; with thresholds 0..255 of 300
// bp 6180 / 6098 / 3542 (one class above 30 before).
constexpr int kTilePairs = 1024;  // pairs of a tile, at most

template <int W, int S, int FROM, int TILE>
__global__ void __launch_bounds__(kFilterThreads, S > 0 ? MinBlocks<W, false, S>::value : (W <= 2 ? 10 : (W <= 4 ? 8 : MinBlocks<W, true>::value * 2)))
    filter_by_e_kernel(const FilterArgs a, uint32_t tile) {
  // Batches of two pairs where a thread may have no more.
  constexpr bool kEarly = TILE == kTilePairs;
  constexpr int kBatch = kEarly ? 4 : 2, kPer = TILE / kFilterThreads;
  constexpr uint8_t kSettled = 0xff;
  __shared__ uint32_t s_rid[TILE], s_off[TILE];
  __shared__ uint16_t s_at[TILE], s_edits[TILE];
  __shared__ uint8_t s_e[TILE], s_class[TILE], s_accept[TILE], s_class_of[256];
  __shared__ uint32_t s_n[kShiftClasses], s_range[kFilterWarps], s_used, s_plan;
  const int lane = threadIdx.x & 31;
  const uint64_t base = blockIdx.x * (uint64_t)tile;
  const uint32_t n_here = (uint32_t)min_u64(tile, a.n_pairs - base);
  if (threadIdx.x < kShiftClasses) s_n[threadIdx.x] = 0;
#pragma unroll
  for (int k = 0; k < 256; k += kFilterThreads) s_class_of[k + threadIdx.x] = (uint8_t)shift_class(k + threadIdx.x);
  __syncthreads();

  // Classify and, kEarly, rank, a batch of pairs per thread at a time: ids, then
  // what they point to.
  uint32_t rid[kPer], off[kPer], rank[kPer];
  uint8_t e[kPer], cls[kPer];
  uint32_t low = kSettled, high = 0, settled = 0;  // this thread's classes; pairs without one
#pragma unroll
  for (int r0 = 0; r0 < kPer; r0 += kBatch) {
    if (r0 * kFilterThreads >= (int)tile) break;
    uint32_t nflag[kBatch];
    uint2 ni[kBatch];
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      const uint32_t i = (uint32_t)(r0 + b) * kFilterThreads + threadIdx.x;
      rid[r0 + b] = 0xffffffffu;
      off[r0 + b] = 0xffffffffu;
      e[r0 + b] = 0;
      if (i < n_here) {
        rid[r0 + b] = a.pair_read[base + i];
        off[r0 + b] = a.pair_off[base + i];
        e[r0 + b] = a.pair_e[base + i];
      }
    }
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      const uint32_t i = (uint32_t)(r0 + b) * kFilterThreads + threadIdx.x;
      const bool ok = i < n_here && rid[r0 + b] <= a.rid_last && off[r0 + b] < a.off_end;
      nflag[b] = ok && a.read_nflag ? a.read_nflag[rid[r0 + b]] : 0u;
      ni[b] = ok && a.ref_nidx ? a.ref_nidx[off[r0 + b] >> 5] : make_uint2(0u, 0xffffffffu);
    }
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      const int r = r0 + b;
      const uint32_t i = (uint32_t)r * kFilterThreads + threadIdx.x;
      const bool active = i < n_here;
      int status = 0;  // 0 filter, 1 undefined, 2 invalid
      if (rid[r] > a.rid_last || off[r] >= a.off_end) {
        status = 2;
      } else {
        const uint32_t q = ni[b].x >> (off[r] & 31);
        const uint32_t first = q ? off[r] + (uint32_t)(__ffs(q) - 1) : ni[b].y;
        if (nflag[b] || first < off[r] + a.m) status = 1;
      }
      if (a.err_count) {
        const unsigned bad = __ballot_sync(0xffffffffu, active && status == 2);
        if (bad && lane == 0) atomicAdd(a.err_count, (unsigned)__popc(bad));
      }
      cls[r] = kSettled;
      if (active && status != 0) {
        s_accept[i] = status != 2;
        s_edits[i] = status == 1 ? GK_EDITS_UNDEFINED : GK_EDITS_INVALID;
        ++settled;
      }
      if (active && status == 0) {
        cls[r] = s_class_of[min((uint32_t)e[r], a.m - 1)];
        low = min(low, (uint32_t)cls[r]);
        high = max(high, (uint32_t)cls[r]);
      }
      if (kEarly) rank[r] = class_rank(cls[r], kSettled, s_n);
    }
  }
  auto worth_sorting = [&]() {
    const uint32_t saves = (7 * n_here * (high - low) + 10 * settled * (high + 1)) * (max(tile, 256u) / 256u);
    return low < kSettled && saves > (W <= 10 ? 48u : 96u) * n_here;
  };
  bool sorted = true;
  if (!kEarly) {
    low = __reduce_min_sync(0xffffffffu, low);
    high = __reduce_max_sync(0xffffffffu, high);
    settled = __reduce_add_sync(0xffffffffu, settled);
    if (lane == 0) s_range[threadIdx.x / 32] = low | (high << 8) | (settled << 16);
    __syncthreads();
    low = kSettled;
    high = settled = 0;
#pragma unroll
    for (int w = 0; w < kFilterWarps; ++w) {
      const uint32_t v = s_range[w];
      low = min(low, v & 0xFFu);
      high = max(high, (v >> 8) & 0xFFu);
      settled += v >> 16;
    }
    sorted = worth_sorting();
    if (sorted) {
#pragma unroll
      for (int r = 0; r < kPer; ++r) {
        if (r * kFilterThreads >= (int)tile) break;
        rank[r] = class_rank(cls[r], kSettled, s_n);
      }
    }
  }
  if (kEarly || sorted) {
    __syncthreads();
    if (threadIdx.x < 32) {
      // kEarly: the counts say how far the classes reach.
      const uint32_t c = kShiftClasses - 1u - 2u * (uint32_t)lane, n0 = s_n[c], n1 = s_n[c - 1];
      const unsigned any = __ballot_sync(0xffffffffu, (n0 | n1) != 0);
      high = __shfl_sync(0xffffffffu, n0 ? c : c - 1, any ? __ffs(any) - 1 : 0);
      low = any ? __shfl_sync(0xffffffffu, n1 ? c - 1 : c, 31 - __clz(any)) : kSettled;
      const uint32_t used = __shfl_sync(0xffffffffu, class_starts(s_n), 31);
      settled = n_here - used;
      if (lane == 0) {
        s_used = used;
        s_plan = high | (worth_sorting() ? 0x100u : 0u);
      }
    }
    __syncthreads();
    high = s_plan & 0xFFu;
    sorted = s_plan >= 0x100u;
  }
#pragma unroll
  for (int r = 0; r < kPer; ++r) {
    if (r * kFilterThreads >= (int)tile) break;
    const uint32_t i = (uint32_t)r * kFilterThreads + threadIdx.x;
    if (sorted && cls[r] == kSettled) continue;
    const uint32_t s = sorted ? s_n[cls[r]] + rank[r] : i;
    s_rid[s] = rid[r];
    s_off[s] = off[r];
    s_e[s] = e[r];
    s_class[s] = cls[r];
    s_at[s] = (uint16_t)i;
  }
  if (sorted) __syncthreads();  // in order a thread reads the entries that it wrote
  const uint32_t n_list = sorted ? s_used : n_here;
#pragma unroll 1
  for (uint32_t s = threadIdx.x; s < n_list; s += kFilterThreads) {
    const uint32_t cl = s_class[s];
    if (cl == kSettled) continue;
    PairData<W> x;
    x.rid = s_rid[s];
    x.off = s_off[s];
    x.e = s_e[s];
    x.m = a.m;
    const uint2 *rp = a.reads + (uint64_t)x.rid * a.stride_words;
#pragma unroll
    for (int w = 0; w < W; ++w) x.r[w] = rp[w];
    load_window<W, false>(a, x);
    uint32_t count;
    if (cl < kExactClass) {
      if constexpr (S > 0)
        // One form per tile: both forms' code does not fit the instruction cache
        // beside the exact one's; at W = 5 one per warp (one on both sides of
        // FROM runs striped).
        count = (W != 5 ? high >= (uint32_t)FROM : __any_sync(__activemask(), cl >= (uint32_t)FROM))
                    ? filter_loaded_striped<W, S>(a, x, cl)
                    : filter_loaded_deferred<W>(a, x);
      else
        count = filter_loaded_deferred<W>(a, x);
    } else {
      count = filter_loaded<W, false>(a, x);
    }
    const uint32_t i = s_at[s];
    s_accept[i] = count <= x.e;
    s_edits[i] = (uint16_t)count;
  }
  if (sorted) __syncthreads();
  for (uint32_t i = threadIdx.x; i < n_here; i += kFilterThreads) {
    a.accept[base + i] = s_accept[i];
    a.edits[base + i] = s_edits[i];
  }
}

// Launches one instantiation of the plain filter over a.n_pairs pairs.
template <int W, int VARIANT, int S = 0>
cudaError_t launch_filter_variant(const FilterArgs &a, cudaStream_t stream) {
  unsigned blocks = (unsigned)((a.n_pairs + kFilterThreads - 1) / kFilterThreads);
  if (a.compact == 0) {
    const uint64_t threads = (a.n_pairs + 1) / 2;
    const unsigned grid = (unsigned)((threads + kFilterThreads - 1) / kFilterThreads);
    // Two pairs per thread for W <= 4 and striped at W = 5: the linear form
    // there (2 blocks per SM with its registers unspilled) measured 40% slower
    // at e = 2, 150 bp.  W > 1 implies m > 0.
    constexpr bool kPairs = VARIANT >= 2 && VARIANT <= 4 && (W <= 4 || S == 5);
    if constexpr (kPairs) {
      if (W > 1 || a.m > 0) {
        if constexpr (VARIANT == 3) {
          sweep_pair2_kernel<W, S><<<grid, kFilterThreads, 0, stream>>>(a);
        } else if constexpr (VARIANT == 4) {
          // shift count = the threshold, 0..2, below m (checked by the caller)
          switch (a.fixed_e) {
            case 0: filter_pair2_kernel<W, 4, 0, S><<<grid, kFilterThreads, 0, stream>>>(a); break;
            case 1: filter_pair2_kernel<W, 4, 1, S><<<grid, kFilterThreads, 0, stream>>>(a); break;
            case 2: filter_pair2_kernel<W, 4, 2, S><<<grid, kFilterThreads, 0, stream>>>(a); break;
            default: return cudaErrorInvalidValue;
          }
        } else {
          filter_pair2_kernel<W, VARIANT, -1, S><<<grid, kFilterThreads, 0, stream>>>(a);
        }
        return cudaGetLastError();
      }
    }
    if constexpr (VARIANT == 4 || (kPairs && W > 1)) {
      return cudaErrorInvalidValue;  // the two-pair kernels only
    } else {
      filter_kernel<W, VARIANT, false, S><<<blocks, kFilterThreads, 0, stream>>>(a);
      return cudaGetLastError();
    }
  }
  if constexpr (VARIANT == 4) {
    return cudaErrorInvalidValue;
  } else {
  // Persistent warps: a few waves of resident blocks.  The dynamic shared
  // memory limit and the occupancy are set up once per device (threads that
  // race here repeat the same idempotent setup; the block count is
  // published after the SM count).
  constexpr int kMaxDev = 64;
  int dev = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err != cudaSuccess) return err;
  if (dev < 0 || dev >= kMaxDev) return cudaErrorInvalidDevice;
  static std::atomic<int> per_sm[kMaxDev], sms[kMaxDev];
  const size_t smem = compact_smem_bytes<W>();
  int blocks_per_sm = per_sm[dev].load(std::memory_order_acquire);
  if (blocks_per_sm == 0) {
    err = cudaFuncSetAttribute(filter_kernel<W, VARIANT, true, S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)smem);
    if (err != cudaSuccess) return err;
    int count = 0;
    err = cudaDeviceGetAttribute(&count, cudaDevAttrMultiProcessorCount, dev);
    if (err != cudaSuccess) return err;
    int n = 0;
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, filter_kernel<W, VARIANT, true, S>, kQueueThreads, smem);
    if (err != cudaSuccess) return err;
    blocks_per_sm = n < 1 ? 1 : n;
    sms[dev].store(count, std::memory_order_relaxed);
    per_sm[dev].store(blocks_per_sm, std::memory_order_release);
  }
  blocks = (unsigned)((a.n_pairs + kQueueThreads - 1) / kQueueThreads);
  const uint64_t wave = 4ull * (uint64_t)sms[dev].load(std::memory_order_relaxed) * (uint64_t)blocks_per_sm;
  if (blocks > wave) blocks = (unsigned)wave;
  filter_kernel<W, VARIANT, true, S><<<blocks, kQueueThreads, smem, stream>>>(a);
  return cudaGetLastError();
  }
}

// Launches the threshold sweep over reads of W = ceil(m/32) words: striped
// where the stripes hold the read (stripe_limit) and beat the linear form at
// the sweep's largest shift count, also where neighbouring pairs name
// different reads.  Measured on GB300, launches alone from e = 0, linear /
// striped in us, pairs in fours of one read (in brackets: each its own read):
//   50 bp  8M  e 1  90 / 88 (122 / 119), 5 190 / 168 (224 / 205)
//   76 bp  8M  e 1 105 / 96 (142 / 135), 8 344 / 246 (424 / 301)
//   96 bp  8M  e 2 138 / 136 (172 / 178), 3 172 / 158, 10 416 / 305
//   100 bp 10M e 1 160 / 158 (240 / 224), 5 345 / 248 (439 / 316), 10 603 / 383
//   128 bp 8M  e 2 161 / 166 (222 / 221), 6 322 / 298 (409 / 346)
//   150 bp 6M  e 1 121 / 109 (125 / 154), 3 191 / 148 (193 / 195), 15 686 / 438
//   160 bp 6M  e 3 191 / 252, 8 396 / 397, 16 730 / 645
//   170 bp 5M  e 3 177 / 221, 9 407 / 379, 17 719 / 605
//   200 bp 4M  e 2 135 / 158, 4 201 / 193, 20 773 / 519
//   250 bp 4M  e 2 158 / 162, 5 263 / 222, 25 1062 / 660
//   280 bp 3M  e 6 248 / 267, 14 514 / 496
//   300 bp 3M  e 6 269 / 279, 15 594 / 533, 30 1136 / 891
// Striped, every step erodes its masks; linear, each written threshold is
// eroded and corrected by itself.  So few thresholds at the end of many steps
// favour the linear form (2M pairs of 64 bp at e = 12..15 79 us, striped 88; of
// 160 bp at 5..10 138 / 146, at 12..15 168 / 184), and rows counts them.  (One
// threshold alone is gk_filter's.)  The queue of defined pairs keeps W = 9, 10
// linear: 11 stripes leave it one block of 256 an SM (2M pairs of 300 bp, 0.1%
// N, e = 0..10 306 us, striped 383).  At 150 bp and largest shift count 3, pairs
// of different reads run 5% slower striped, pairs that share theirs 20% faster.
// W = 1 needs one linear word and three stripes; from W = 11 the stripes spill.
template <int W, int S>
__host__ bool sweep_striped(uint32_t K, uint32_t rows, int queue) {
  if (S == 11) return !queue && K >= (W == 9 ? 14u : 12u) && rows >= 6;
  if (W == 2) return 3 * rows > K;
  if (W == 4 && S == 5) return K >= 3 && 3 * rows > K;
  if (W == 5 && S == 8) return K >= 10 && rows >= 9;
  if (W == 6) return K >= 9 && rows >= 6;
  if (W == 7) return K >= 4;
  if (W == 5) return K >= 3;
  return (W == 3 && S == 3) || W == 4 || (K >= 3 && K + rows >= 7);
}
template <int W>
cudaError_t launch_sweep(const FilterArgs &a, cudaStream_t stream) {
  if constexpr (W >= 2 && W <= 10) {
    constexpr int S0 = W <= 3 ? 3 : (W <= 5 ? W : (W <= 8 ? 8 : 11));
    constexpr int S1 = W == 3 ? 4 : (W == 4 ? 5 : (W == 5 ? 8 : 0));  // reads S0 does not hold
    const uint32_t K = min(a.sweep_hi, a.m - 1), rows = K - min(a.fixed_e, a.m - 1) + 1;
    if (a.m <= stripe_limit<S0>()) {
      if (sweep_striped<W, S0>(K, rows, a.compact)) return launch_filter_variant<W, 3, S0>(a, stream);
    } else if constexpr (S1 > 0) {
      if (sweep_striped<W, S1>(K, rows, a.compact)) return launch_filter_variant<W, 3, S1>(a, stream);
    }
  }
  return launch_filter_variant<W, 3>(a, stream);
}

// Launches VARIANT 2 (one threshold, shift count 2 .. 30, edge OR on) over
// reads of W words: striped from the shift count at which it wins, also where
// neighbouring pairs name different reads (they cost it a second load).
// Striping a read and a window takes as long as about three shift steps, and
// rows are partly empty at m well below 32 S.  Measured on GB300, launches
// alone, linear / striped in us, pairs in fours of one read: 8M pairs of 76 bp
// K = 4 144 / 135 (every pair its own read: 168 / 187), K = 8 211 / 186 (248 /
// 236); 10M of 100 bp K = 5 232 / 232, 7 289 / 257, 10 375 / 302 (455 / 407); 6M
// of 150 bp K = 5 197 / 158, 8 266 / 193 (267 / 263), 15 441 / 285; 5M of 170 bp
// K = 9 279 / 315, 17 477 / 451; of 200 bp K = 7 258 / 267, 10 340 / 311; 4M of
// 250 bp K = 5 188 / 209, 8 257 / 242, 25 687 / 473; 3M of 280 bp K = 14 345 /
// 326; of 300 bp K = 9 258 / 258, 15 400 / 347; 128 and 160 bp (S = 5 and 8 with
// 20 rows) no faster up to K = 16.  In the queue of defined pairs 11 stripes win
// from K = 25 (2M pairs of 300 bp, 0.1% N: K = 12 237 / 282 us, 20 341 / 348, 25
// 401 / 392, 30 467 / 432).
//
// Up to shift count 7 in overlapping words where they hold the read (m <= 30 W)
// and W <= 8, ordinary / overlapping words in us on the same launches: 50 bp K =
// 2 97 / 91, 7 150 / 134; 76 bp K = 2 112 / 107, 7 193 / 168; 100 bp K = 3 187 /
// 174, 5 234 / 209, 7 290 / 253; 150 bp K = 2 135 / 135, 5 197 / 184; 200 bp K =
// 2 123 / 111, 7 209 / 187; 240 bp K = 3 156 / 138, 7 232 / 205.
template <int W>
__host__ constexpr uint32_t single_striped_from() {
  return W == 6 ? 16 : (W == 7 ? 9 : (W == 9 ? 14 : (W == 10 ? 12 : 8)));
}
template <int W>
__host__ bool single_overlaps(const FilterArgs &a) {
  return W >= 2 && W <= 8 && a.m <= overlap_limit<W>() && a.fixed_e <= kOverlapMax && (W != 5 || a.fixed_e >= 3);
}
template <int W>
cudaError_t launch_single(const FilterArgs &a, cudaStream_t stream) {
  if constexpr (W >= 2 && W <= 8)
    if (single_overlaps<W>(a)) return launch_filter_variant<W, 2, -1>(a, stream);
  if constexpr (W >= 3 && W <= 10) {
    constexpr int S = W <= 5 ? W : (W <= 8 ? 8 : 11);
    if (a.m <= stripe_limit<S>() && a.fixed_e >= (S == 11 && a.compact ? 25u : single_striped_from<W>()))
      return launch_filter_variant<W, 2, S>(a, stream);
  }
  return launch_filter_variant<W, 2>(a, stream);
}

// VARIANT 4 (thresholds 0 .. 2, W <= 4): 100 bp K = 0 113 / 112, 1 135 / 130, 2 158
// / 148 us for 10M pairs.
template <int W>
cudaError_t launch_small(const FilterArgs &a, cudaStream_t stream) {
  if constexpr (W >= 2 && W <= 4)
    if (a.m <= overlap_limit<W>()) return launch_filter_variant<W, 4, -1>(a, stream);
  return launch_filter_variant<W, 4>(a, stream);
}

// Launches per-pair thresholds (edge OR on, m > 0).  Tiles shrink with the
// launch, so that a small one still spreads over the chip.
template <int W, int S, int FROM>
cudaError_t launch_by_e_striped(const FilterArgs &a, cudaStream_t stream) {
  uint32_t tile = kTilePairs;
  while (tile > (uint32_t)kFilterThreads && a.n_pairs / tile < 2048) tile /= 2;
  const uint64_t blocks = (a.n_pairs + tile - 1) / tile;
  if (tile == (uint32_t)kTilePairs)
    filter_by_e_kernel<W, S, FROM, kTilePairs><<<(unsigned)blocks, kFilterThreads, 0, stream>>>(a, tile);
  else
    filter_by_e_kernel<W, S, FROM, kTilePairs / 2><<<(unsigned)blocks, kFilterThreads, 0, stream>>>(a, tile);
  return cudaGetLastError();
}
template <int W>
cudaError_t launch_by_e(const FilterArgs &a, cudaStream_t stream) {
  // W = 6 linear: with both forms registers hold 4 blocks an SM, without 6.
  if constexpr (W >= 4 && W <= 10 && W != 6) {
    constexpr int S = W <= 5 ? W : (W <= 8 ? 8 : 11);
    if (a.m <= stripe_limit<S>()) return launch_by_e_striped<W, S, single_striped_from<W>()>(a, stream);
  }
  return launch_by_e_striped<W, 0, 0>(a, stream);
}

}  // namespace gk
