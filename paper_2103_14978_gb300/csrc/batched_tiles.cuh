// Batched filter, one pair per lane (words_per_thread 1).
//
// A block takes a tile of consecutive pairs into shared memory, settles the
// invalid, undefined and empty ones, and sorts the rest by the code that
// filters them (their group: words per read, striped or linear) and, within a
// group, by shift count, largest first.  Then
//   small launches   filter the tile in the same block (tiles_kernel): warps
//                    take 32 pairs of one group at a time from the sorted
//                    list, results stay in shared memory and go out in pair
//                    order.  One launch, no scratch.
//   large launches   write the tile's pairs as 16-byte records in sorted order
//                    (plan_kernel); filter launches, one per range of read
//                    lengths or one for all, then take one group of 8 tiles
//                    at a time
//                    (groups_kernel).  All blocks of a launch run one group's
//                    code at about the same time: with 50-300 bp mixed, a
//                    tile's groups in turn waited for instructions a fifth of
//                    the time (18 groups, 200 KB of code) and ran at 62% of
//                    the ALU pipe, here at 90%.
//
// A launch-wide counting sort in place of the tiles (histogram, scan, scatter
// of the records to their final slots) read every pair's ids twice and took
// 1.15 of 5.3 ms for 50M pairs.
//
// Measured on GB300, 50M pairs of 50-300 bp, per-pair thresholds of 2, 5 and
// 10%, random order: 5.43 -> 4.65 ms per graph launch (planning
// 0.7, bound by the gathers of read length and N flag; the filters by the ALU
// pipe, those of up to 128 bp by the gathers of shuffled read rows); a server round of 3M pairs
// of 100, 150 and 250 bp (three calls) 0.392 -> 0.268 ms.
#pragma once

#include "batched.cuh"

namespace gk {

constexpr int kTilesThreads = 256;  // of tiles_kernel
constexpr int kPlanThreads = 512;   // of plan_kernel
constexpr int kPlanPer = 8;         // pairs of a plan_kernel thread
constexpr uint32_t kPlanPairs = kPlanThreads * kPlanPer;  // its tile
constexpr uint32_t kTilesPairs = 1024;  // pairs of tiles_kernel's tile, at most

// Launches of up to this many pairs filter in their tiles.  How many lengths a
// launch mixes is not known on the host; rows of up to 4 words hold few (8
// groups).  Measured, in tiles / through records: 50-300 bp, 0.25M pairs 0.123
// ms / 0.217 (a launch-wide sort), 0.5M 0.222 / not measured, 1M 0.293 / 0.132;
// 250 bp 1M 0.129 / 0.110.
template <int WHI>
constexpr uint64_t tiles_fused() {
  return WHI <= 4 ? 2000000 : 300000;
}
// Up to this many pairs the records of all lengths (of up to 10 words) are
// filtered by one launch; above, one per range of lengths has more warps in
// flight for the short ones (4 words: 32 a SM, else 16).  Mixed, 3M pairs: 0.338
// ms in one, 0.342 in four.
constexpr uint64_t kTilesOneRange = 8000000;
constexpr uint32_t kGroupTiles = 8;     // tiles of a work item of groups_kernel
constexpr uint32_t kSliceRecords = 1024;  // of its slices, at most
constexpr int kGroupThreads = 128;

// Shared bytes of a tile: read id, offset (later the result), length, key,
// list of sorted pairs (with each group's last warp padded), threshold.
template <int WHI>
constexpr size_t tiles_smem(uint32_t tile) {
  return (size_t)tile * (4 + 4 + 2 + 2 + 2 + 1) + 2 * WHI * 32 * 2;
}

// A tile's arrays in dynamic shared memory.
struct TileArrays {
  uint32_t *rid, *off;
  uint16_t *m, *key, *list;
  uint8_t *e;
  __device__ __forceinline__ TileArrays(uint32_t *mem, uint32_t tile, int groups) {
    rid = mem;
    off = rid + tile;
    m = reinterpret_cast<uint16_t *>(off + tile);
    key = m + tile;
    list = key + tile;
    e = reinterpret_cast<uint8_t *>(list + tile + groups * 32);
  }
};
constexpr uint32_t kNoSlot = 0xFFFFu;

// Stripes for reads of W words in the batched filter (0: linear only), and the
// shift count from which they win over the linear form, one pair per lane.
template <int W>
__host__ __device__ constexpr int tiles_stripes() {
  return W == 4 || W == 5 ? W : (W == 7 || W == 8 ? 8 : 0);
}
template <int W>
__host__ __device__ constexpr uint32_t tiles_stripe_from() {
  return W == 4 ? 8 : (W == 5 ? 11 : (W == 7 ? 14 : 10));
}

// Whether a read of m bases is filtered striped at shift count K.
template <int WHI, int W = WHI>
__device__ __forceinline__ bool tiles_striped(uint32_t Wp, uint32_t m, uint32_t K) {
  if constexpr (W < 4) {
    return false;
  } else {
    if (Wp != (uint32_t)W) return tiles_striped<WHI, W - 1>(Wp, m, K);
    constexpr int S = tiles_stripes<W>();
    if constexpr (S == 0)
      return false;
    else
      return K >= tiles_stripe_from<W>() && K <= 30 && m <= stripe_limit<S>();
  }
}

// The count of one pair, by its group: 2 (WHI - W) striped, one more linear.
template <int WHI, int WLO = 1, int W = WHI>
__device__ __forceinline__ uint32_t tiles_count(const FilterArgs &a, uint32_t group, uint32_t rid, uint32_t off,
                                                uint32_t m, uint32_t e) {
  if (group / 2 == (uint32_t)(WHI - W)) {
    PairData<W> x;
    x.rid = rid;
    x.off = off;
    x.m = m;
    x.e = e;
    x.status = 0;
    load_words_wide<W>(a.reads, a.stride_words, a.ref_hl, x);
    const uint32_t K = min(e, m - 1);
    if constexpr (tiles_stripes<W>() > 0) {
      if ((group & 1u) == 0) {
        uint32_t c[1];
        striped_counts<W, tiles_stripes<W>(), 1, false>(x, x, m, K, a.count_mode, c);
        return c[0];
      }
    }
    if (K <= 30) return a.edge_on ? filter_loaded_deferred<W>(a, x) : filter_loaded<W, true>(a, x);
    return filter_loaded<W, false>(a, x);
  }
  if constexpr (W > WLO)
    return tiles_count<WHI, WLO, W - 1>(a, group, rid, off, m, e);
  else
    return 0;
}

// What R pairs per thread need to be classified: pair r of a thread is first +
// r * THREADS + threadIdx.x of the launch, up to end.  Ids first, then what
// they point to: two rounds of independent loads.
template <int R, int THREADS>
struct PairBatch {
  uint32_t rid[R], off[R], e[R], m[R], nf[R];
  uint2 ni[R];
  __device__ __forceinline__ void load(const BatchArgs &b, uint64_t first, uint64_t end) {
    const FilterArgs &a = b.f;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const uint64_t p = first + (uint64_t)r * THREADS + threadIdx.x;
      rid[r] = 0xffffffffu;
      off[r] = 0xffffffffu;
      e[r] = a.fixed_e;
      if (p < end) {
        rid[r] = a.pair_read[p];
        off[r] = a.pair_off[p];
        if (a.pair_e) e[r] = a.pair_e[p];
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const uint64_t p = first + (uint64_t)r * THREADS + threadIdx.x;
      m[r] = 0;
      nf[r] = 0;
      ni[r] = make_uint2(0u, 0xffffffffu);
      if ((uint64_t)rid[r] < a.n_reads && p < end) {
        m[r] = b.read_len[rid[r]];
        if (a.read_nflag) nf[r] = a.read_nflag[rid[r]];
      }
      if (a.ref_nidx && (uint64_t)off[r] < a.ref_len) ni[r] = a.ref_nidx[off[r] >> 5];
    }
  }
  // 0 filter, 1 undefined, 2 invalid, 3 empty read.
  __device__ __forceinline__ int status(const FilterArgs &a, int r) const {
    if ((uint64_t)rid[r] >= a.n_reads || m[r] > GK_MAX_LEN || m[r] > 32u * a.stride_words ||
        (uint64_t)off[r] + m[r] > a.ref_len)
      return 2;
    if (m[r] == 0) return 3;
    if (nf[r]) return 1;
    if (a.ref_nidx) {  // a valid pair's window ends below 2^32
      const uint32_t q = ni[r].x >> (off[r] & 31);
      const uint32_t first = q ? off[r] + (uint32_t)(__ffs(q) - 1) : ni[r].y;
      if (first < off[r] + m[r]) return 1;
    }
    return 0;
  }
};

// Sort key of a pair to filter: its group, then its shift count, largest first
// (31 and more in one class).
template <int WHI>
__device__ __forceinline__ uint32_t tiles_key(const FilterArgs &a, uint32_t m, uint32_t e) {
  const uint32_t W = (m + 31) / 32, K = min(e, m - 1);
  const bool striped = a.edge_on && tiles_striped<WHI>(W, m, K);
  return ((uint32_t)(WHI - (int)W) * 2u + (striped ? 0u : 1u)) * 32u + (31u - min(K, 31u));
}

// Turns the counts of n_keys keys into each key's first list slot; PAD: groups
// of 32 keys start on multiples of 32.  Returns the slots used (in lane 31).
template <bool PAD>
__device__ __forceinline__ uint32_t tiles_scan(uint32_t *s_n, int groups) {
  const int lane = threadIdx.x & 31;
  uint32_t total = 0;
  if (lane < groups)
    for (int k = 0; k < 32; ++k) total += s_n[lane * 32 + k];
  const uint32_t width = PAD ? (total + 31u) & ~31u : total;
  uint32_t end = width;
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t o = __shfl_up_sync(0xffffffffu, end, d);
    if (lane >= d) end += o;
  }
  uint32_t at = end - width;
  if (lane < groups)
    for (int k = 0; k < 32; ++k) {
      const uint32_t n = s_n[lane * 32 + k];
      s_n[lane * 32 + k] = at;
      at += n;
    }
  return end;
}

// Classifies and sorts a tile.  On return (after a barrier) t.list holds the
// pairs' indices by key, each group's from a multiple of 32 slots, empty slots
// kNoSlot; slots[0] the slots used.  Pairs that are settled have no slot, their
// result (accept or result byte << 16 | count) is in t.off.
template <int WHI>
__device__ __forceinline__ void tile_sort(const BatchArgs &b, uint32_t tile, const TileArrays &t, uint32_t *s_n,
                                          uint32_t *slots) {
  constexpr int kGroups = 2 * WHI, kBatch = kTilesPairs / kTilesThreads;
  const FilterArgs &a = b.f;
  const int lane = threadIdx.x & 31;
  const uint64_t base = blockIdx.x * (uint64_t)tile;
  const uint32_t n_here = (uint32_t)min_u64(tile, a.n_pairs - base);
  for (int i = threadIdx.x; i < kGroups * 32; i += kTilesThreads) s_n[i] = 0;
  for (uint32_t i = threadIdx.x; i < tile + kGroups * 32; i += kTilesThreads) t.list[i] = kNoSlot;
  __syncthreads();
  PairBatch<kBatch, kTilesThreads> x;
  x.load(b, base, base + n_here);
#pragma unroll
  for (int r = 0; r < kBatch; ++r) {
    const uint32_t i = (uint32_t)r * kTilesThreads + threadIdx.x;
    const bool active = i < n_here;
    const int status = x.status(a, r);
    if (a.err_count) {
      const unsigned bad = __ballot_sync(0xffffffffu, active && status == 2);
      if (bad && lane == 0) atomicAdd(a.err_count, (unsigned)__popc(bad));
    }
    if (!active) continue;
    uint32_t key = kNoSlot;
    if (status == 0) {
      key = tiles_key<WHI>(a, x.m[r], x.e[r]);
      atomicAdd(&s_n[key], 1u);
      t.rid[i] = x.rid[r];
      t.off[i] = x.off[r];
      t.m[i] = (uint16_t)x.m[r];
      t.e[i] = (uint8_t)x.e[r];
    } else if (a.result_byte) {
      t.off[i] = (status == 1 ? GK_RESULT_UNDEFINED : status == 2 ? GK_RESULT_INVALID : 0u) << 16;
    } else {
      t.off[i] = status == 1 ? (0x10000u | GK_EDITS_UNDEFINED) : status == 2 ? GK_EDITS_INVALID : 0x10000u;
    }
    t.key[i] = (uint16_t)key;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    const uint32_t end = tiles_scan<true>(s_n, kGroups);
    if (lane == 31) slots[0] = end;
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < n_here; i += kTilesThreads) {
    const uint32_t key = t.key[i];
    if (key != kNoSlot) t.list[atomicAdd(&s_n[key], 1u)] = (uint16_t)i;
  }
  __syncthreads();
}

// Resident blocks of tiles_kernel per SM.
template <int WHI>
constexpr int kTilesBlocks = WHI <= 4 ? 4 : (WHI <= 10 ? 2 : 1);

// Reads of at most WHI words (the row stride bounds them): sorted and filtered.
template <int WHI>
__global__ void __launch_bounds__(kTilesThreads, kTilesBlocks<WHI>)
    tiles_kernel(const BatchArgs b, uint32_t tile) {
  extern __shared__ uint32_t s_mem[];
  __shared__ uint32_t s_n[2 * WHI * 32], s_slots, s_next;
  const TileArrays t(s_mem, tile, 2 * WHI);
  const FilterArgs &a = b.f;
  const int lane = threadIdx.x & 31;
  const uint64_t base = blockIdx.x * (uint64_t)tile;
  const uint32_t n_here = (uint32_t)min_u64(tile, a.n_pairs - base);
  if (threadIdx.x == 0) s_next = 0;
  tile_sort<WHI>(b, tile, t, s_n, &s_slots);

  // ---- filter: 32 list slots at a time, the heaviest first ----
  const uint32_t slots = s_slots;
  for (;;) {
    uint32_t s = 0;
    if (lane == 0) s = atomicAdd(&s_next, 32u);
    s = __shfl_sync(0xffffffffu, s, 0);
    if (s >= slots) break;
    const uint32_t i = t.list[s + (uint32_t)lane];
    const uint32_t group = t.key[t.list[s]] / 32u;  // the warp's; its first slot is never padding
    if (i != kNoSlot) {
      const uint32_t e = t.e[i];
      const uint32_t count = tiles_count<WHI>(a, group, t.rid[i], t.off[i], t.m[i], e);
      t.off[i] = a.result_byte ? min(count, GK_RESULT_MAX_COUNT) << 16 : ((count <= e ? 0x10000u : 0u) | count);
    }
    __syncwarp();
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < n_here; i += kTilesThreads) {
    const uint32_t v = t.off[i];
    a.accept[base + i] = (uint8_t)(v >> 16);
    if (!a.result_byte) a.edits[base + i] = (uint16_t)v;
  }
}

// Classifies a tile (settled pairs get their results) and writes its other
// pairs as records in sorted order at the tile's own place, and per group their
// range: desc[group * tiles + tile] = first | count << 16.  Clears the filter
// launches' item counters.  The pairs stay in registers: counting atomics
// without a return value, a scan, then one returning atomic and one 16-byte
// store per pair; L2 joins the stores, which fall into 64 KB.
template <int WHI>
__global__ void __launch_bounds__(kPlanThreads, 2) plan_kernel(const BatchArgs b, uint32_t *desc) {
  __shared__ uint32_t s_n[2 * WHI * 32];
  const FilterArgs &a = b.f;
  const int lane = threadIdx.x & 31;
  const uint64_t base = blockIdx.x * (uint64_t)kPlanPairs;
  const uint64_t end = min_u64(base + kPlanPairs, a.n_pairs);
  if (blockIdx.x == 0 && threadIdx.x < 8) b.s.counters[threadIdx.x] = 0;
  for (int i = threadIdx.x; i < 2 * WHI * 32; i += kPlanThreads) s_n[i] = 0;
  PairBatch<kPlanPer, kPlanThreads> x;
  x.load(b, base, end);
  __syncthreads();
  uint32_t key[kPlanPer];
#pragma unroll
  for (int r = 0; r < kPlanPer; ++r) {
    const uint64_t p = base + (uint64_t)r * kPlanThreads + threadIdx.x;
    const bool active = p < end;
    const int status = x.status(a, r);
    if (a.err_count) {
      const unsigned bad = __ballot_sync(0xffffffffu, active && status == 2);
      if (bad && lane == 0) atomicAdd(a.err_count, (unsigned)__popc(bad));
    }
    key[r] = kNoSlot;
    if (active && status == 0) {
      key[r] = tiles_key<WHI>(a, x.m[r], x.e[r]);
      atomicAdd(&s_n[key[r]], 1u);
    } else if (active) {
      write_trivial(a, p, status == 3 ? 0 : status);  // an empty read: count 0, accepted
    }
  }
  __syncthreads();
  if (threadIdx.x < 32) tiles_scan<false>(s_n, 2 * WHI);
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kPlanPer; ++r)
    if (key[r] != kNoSlot)
      b.s.rec[base + atomicAdd(&s_n[key[r]], 1u)] =
          make_uint4((uint32_t)(base + (uint64_t)r * kPlanThreads + threadIdx.x), x.rid[r], x.off[r],
                     x.e[r] | (x.m[r] << 16));
  __syncthreads();
  if (threadIdx.x < 2 * WHI) {
    // s_n: the slot past each key's last pair; a group's first is the group before's last
    const uint32_t first = threadIdx.x ? s_n[threadIdx.x * 32 - 1] : 0u, last = s_n[threadIdx.x * 32 + 31];
    desc[(uint64_t)threadIdx.x * gridDim.x + blockIdx.x] = first | ((last - first) << 16);
  }
}

// The groups of reads of WLO .. WTOP words out of records planned for reads of
// at most WHI: persistent blocks take one group of kGroupTiles tiles at a time,
// all tiles of the longest reads first.  Where a launch is small, or most pairs
// are of one group (up to 32768 records), these items are too few to go round
// the SMs, so a group's are cut into slices: of a quarter of a block's share, at
// most kSliceRecords, as the counts of 32 tiles, evenly spread, suggest (the
// same tiles for every block).
template <int WHI, int WLO, int WTOP>
__global__ void __launch_bounds__(kGroupThreads, WTOP <= 4 ? 8 : (WTOP <= 5 ? 6 : (WTOP <= 10 ? 4 : 2)))
    groups_kernel(const BatchArgs b, uint32_t tiles, const uint32_t *desc, uint32_t *counter) {
  constexpr uint32_t kFirst = 2 * (WHI - WTOP), kCount = 2 * (WTOP - WLO + 1);
  __shared__ uint32_t s_first[kGroupTiles], s_end[kGroupTiles + 1], s_item, s_slices[kCount];
  const FilterArgs &a = b.f;
  const uint32_t parts = (tiles + kGroupTiles - 1) / kGroupTiles;
  for (uint32_t g = threadIdx.x / 32; g < kCount; g += kGroupThreads / 32) {
    const uint32_t at = (uint32_t)((uint64_t)tiles * (threadIdx.x & 31u) / 32u);
    const uint32_t count = __reduce_add_sync(0xffffffffu, desc[(uint64_t)(kFirst + g) * tiles + at] >> 16);
    if ((threadIdx.x & 31u) == 0) s_slices[g] = count;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    const uint32_t count = threadIdx.x < kCount ? s_slices[threadIdx.x] : 0u;
    const uint64_t range = (uint64_t)__reduce_add_sync(0xffffffffu, count) * tiles / 32u;
    const uint32_t slice = max((uint32_t)kGroupThreads, (uint32_t)min_u64(kSliceRecords, range / (4u * gridDim.x)));
    if (threadIdx.x < kCount) s_slices[threadIdx.x] = max(1u, count / (32u / kGroupTiles * slice));
  }
  for (;;) {
    if (threadIdx.x == 0) s_item = atomicAdd(counter, 1u);
    __syncthreads();
    uint32_t item = s_item, g = 0, slices = s_slices[0];
    while (g < kCount && item >= parts * slices) {
      item -= parts * slices;
      if (++g < kCount) slices = s_slices[g];
    }
    if (g == kCount) break;
    const uint32_t group = kFirst + g, t0 = item / slices * kGroupTiles, slice = item % slices;
    if (threadIdx.x < 32) {
      const uint32_t lane = threadIdx.x;
      const uint32_t d = lane < kGroupTiles && t0 + lane < tiles ? desc[(uint64_t)group * tiles + t0 + lane] : 0u;
      uint32_t end = d >> 16;
      for (int k = 1; k < 32; k <<= 1) {
        const uint32_t o = __shfl_up_sync(0xffffffffu, end, k);
        if (lane >= (uint32_t)k) end += o;
      }
      if (lane < kGroupTiles) {
        s_first[lane] = d & 0xFFFFu;
        s_end[lane + 1] = end;
      }
      if (lane == 0) s_end[0] = 0;
    }
    __syncthreads();
    const uint32_t all = s_end[kGroupTiles];
    const uint32_t per = ((all + slices - 1) / slices + kGroupThreads - 1) / kGroupThreads * kGroupThreads;
    const uint32_t n = min(all, (slice + 1) * per), j0 = slice * per + threadIdx.x;
    auto record = [&](uint32_t j) -> uint4 {
      uint32_t q = 0;  // the tile that holds record j
#pragma unroll
      for (uint32_t step = kGroupTiles / 2; step > 0; step /= 2)
        if (s_end[q + step] <= j) q += step;
      return b.s.rec[(uint64_t)(t0 + q) * kPlanPairs + s_first[q] + (j - s_end[q])];
    };
    // The next pair's record is loaded while this one's words are.
    uint4 next = j0 < n ? record(j0) : make_uint4(0u, 0u, 0u, 0u);
    for (uint32_t j = j0; j < n; j += kGroupThreads) {
      const uint4 rec = next;
      if (j + kGroupThreads < n) next = record(j + kGroupThreads);
      const uint32_t e = rec.w & 0xFFFFu;
      write_count(a, rec.x, tiles_count<WHI, WLO, WTOP>(a, group, rec.y, rec.z, rec.w >> 16, e), e);
    }
    __syncthreads();
  }
}

template <int WHI, int WLO, int WTOP>
cudaError_t launch_groups(const BatchArgs &b, uint32_t tiles, const uint32_t *desc, uint32_t *counter, uint32_t sms,
                          cudaStream_t stream) {
  if (b.f.stride_words < (uint32_t)WLO) return cudaSuccess;  // no read is that long
  constexpr uint32_t kPerSm = WTOP <= 4 ? 8 : (WTOP <= 5 ? 6 : (WTOP <= 10 ? 4 : 2));
  groups_kernel<WHI, WLO, WTOP><<<sms * kPerSm, kGroupThreads, 0, stream>>>(b, tiles, desc, counter);
  return cudaGetLastError();
}

template <int WHI>
cudaError_t launch_tiles(const BatchArgs &b, cudaStream_t stream) {
  int dev = 0, sms = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err == cudaSuccess) err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (err != cudaSuccess) return err;
  if (b.f.n_pairs <= tiles_fused<WHI>()) {
    // The smallest tile whose blocks all run at once: larger ones fill their
    // groups' warps, but leave SMs without a block.  50-300 bp mixed, 300k pairs:
    // tiles of 256 128 us, of 1024 60; 250 bp 300k 53 / 36; 36-512 bp 300k 871 / 310;
    // 150 bp 50k 11 us, of 1024 16.
    uint32_t tile = kTilesThreads;
    while (tile < kTilesPairs && b.f.n_pairs > (uint64_t)tile * (uint32_t)sms * kTilesBlocks<WHI>) tile *= 2;
    tiles_kernel<WHI><<<(unsigned)((b.f.n_pairs + tile - 1) / tile), kTilesThreads, tiles_smem<WHI>(tile), stream>>>(
        b, tile);
    return cudaGetLastError();
  }
  const uint32_t tiles = (uint32_t)((b.f.n_pairs + kPlanPairs - 1) / kPlanPairs), n = (uint32_t)sms;
  uint32_t *desc = b.s.km;  // 2 WHI <= 32 words per 4096 pairs, out of a word per pair
  plan_kernel<WHI><<<tiles, kPlanThreads, 0, stream>>>(b, desc);
  err = cudaGetLastError();
  if constexpr (WHI > 10)
    if (err == cudaSuccess) err = launch_groups<WHI, 11, WHI>(b, tiles, desc, b.s.counters + 4, n, stream);
  if constexpr (WHI > 4)
    if (b.f.n_pairs <= kTilesOneRange) {
      constexpr int kTop = WHI < 10 ? WHI : 10;
      if (err == cudaSuccess) err = launch_groups<WHI, 1, kTop>(b, tiles, desc, b.s.counters, n, stream);
      return err;
    }
  if constexpr (WHI > 8)
    if (err == cudaSuccess) err = launch_groups<WHI, 9, 10>(b, tiles, desc, b.s.counters + 3, n, stream);
  if constexpr (WHI > 4) {
    if (err == cudaSuccess) err = launch_groups<WHI, 6, 8>(b, tiles, desc, b.s.counters + 2, n, stream);
    if (err == cudaSuccess) err = launch_groups<WHI, 5, 5>(b, tiles, desc, b.s.counters + 1, n, stream);
  }
  if (err == cudaSuccess) err = launch_groups<WHI, 1, 4>(b, tiles, desc, b.s.counters, n, stream);
  return err;
}

}  // namespace gk
