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
//                    (plan_kernel, a cluster of blocks per tile); filter
//                    launches, one per range of read lengths or one for all,
//                    then take a slice of one group of one tile at a time
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
// Measured on GB300 against that sort, 50M pairs of 50-300 bp, per-pair
// thresholds of 2, 5 and 10%, random order: 5.30 -> 4.53 ms per graph launch
// (planning 0.81, bound by the gathers of read length and N flag; the filters by
// the ALU pipe, those of up to 128 bp by the gathers of shuffled read rows); a
// server round of 3M pairs of 100, 150 and 250 bp (three calls) 0.400 -> 0.241
// ms.  9M pairs of 36-512 bp 1.97 -> 2.11, of 200-512 bp 2.70 -> 2.78: a launch
// above 8M pairs whose rows have more than 10 words is the slower one.
#pragma once

#include <cooperative_groups.h>

#include "batched.cuh"

namespace gk {

constexpr int kTilesThreads = 256;  // of tiles_kernel
constexpr int kPlanThreads = 512;   // of plan_kernel
constexpr int kPlanPer = 7;         // pairs of a plan_kernel thread
constexpr uint32_t kBlockPairs = kPlanThreads * kPlanPer;
constexpr uint32_t kPlanCluster = 4;  // blocks that sort together
constexpr uint32_t kPlanPairs = kPlanCluster * kBlockPairs;  // their tile
constexpr uint32_t kTilesPairs = 1024;  // pairs of tiles_kernel's tile, at most

// Launches of up to this many pairs filter in their tiles.  How many lengths a
// launch mixes is not known on the host; rows of up to 4 words hold few (8
// groups).  Measured, thresholds of 2, 5 and 10%, in tiles / through records in
// us: 100 bp 300k pairs 18 / 26, 2M 76 / 85, 3M 113 / 120; 150 bp 300k 24 / 34, 1M
// 69 / 67; 512 bp 300k 186 / 184; mixed, 50-300 bp 150k 44 / 40, 300k 60 / 47, 450k
// 91 / 57, 36-512 bp 300k 305 / 120; with threshold 2 for all 33 / 46 (36-512 bp).
template <int WHI>
constexpr uint64_t tiles_fused() {
  return WHI <= 4 ? 2000000 : 300000;
}
// Up to this many pairs the records of all lengths (of up to 10 words) are
// filtered by one launch; above, one per range of lengths has more warps in
// flight for the short ones (4 words: 32 a SM, else 16).  One launch / one per
// range, 9M pairs: 150 bp 506 / 478 us, 50-300 bp 746 / 778; 50M: 150 bp 2674 /
// 2466, 50-300 bp 4060 / 3914.
constexpr uint64_t kTilesOneRange = 8000000;
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
    // one form per warp: shift counts on both sides of the class run exact
    if (!__any_sync(__activemask(), K >= kExactClass))
      return a.edge_on ? filter_loaded_deferred<W>(a, x) : filter_loaded<W, true>(a, x);
    return filter_loaded<W, false>(a, x);
  }
  if constexpr (W > WLO)
    return tiles_count<WHI, WLO, W - 1>(a, group, rid, off, m, e);
  else
    return 0;
}

// What R pairs per thread need to be classified: pair r of a thread is first +
// r * THREADS + threadIdx.x of the launch, up to first + n.  Ids first, then what
// they point to: two rounds of independent loads.
template <int R, int THREADS>
struct PairBatch {
  uint32_t rid[R], off[R], e[R], m[R], nf[R];
  uint2 ni[R];
  __device__ __forceinline__ void load(const BatchArgs &b, uint64_t first, uint32_t n) {
    const FilterArgs &a = b.f;
    const uint32_t *pr = a.pair_read + first, *po = a.pair_off + first;
    const uint8_t *pe = a.pair_e ? a.pair_e + first : nullptr;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const uint32_t i = (uint32_t)r * THREADS + threadIdx.x;
      rid[r] = 0xffffffffu;
      off[r] = 0xffffffffu;
      e[r] = a.fixed_e;
      if (i < n) {
        rid[r] = pr[i];
        off[r] = po[i];
        if (pe) e[r] = pe[i];
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const uint32_t i = (uint32_t)r * THREADS + threadIdx.x;
      m[r] = 0;
      nf[r] = 0;
      ni[r] = make_uint2(0u, 0xffffffffu);
      if ((uint64_t)rid[r] < a.n_reads && i < n) {
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

// Sort key of a pair to filter: its group, then its shift class, largest first.
template <int WHI>
__device__ __forceinline__ uint32_t tiles_key(const FilterArgs &a, uint32_t m, uint32_t e) {
  const uint32_t W = (m + 31) / 32, K = min(e, m - 1);
  const bool striped = a.edge_on && tiles_striped<WHI>(W, m, K);
  return ((uint32_t)(WHI - (int)W) * 2u + (striped ? 0u : 1u)) * kShiftClasses + (kShiftClasses - 1u - shift_class(K));
}

// The keys of a block's THREADS threads, in order: a group's are those of
// THREADS / 32 threads of one warp.  mine: how many pairs this thread's keys
// have.  Returns the first list slot of its first key; PAD: groups start on
// multiples of 32.  slots: the slots used.  s_group: 2 WHI words.
template <int THREADS>
constexpr int kScanLanes = THREADS / 32;
template <int THREADS>
constexpr int kScanKeys = (int)kShiftClasses / kScanLanes<THREADS>;
template <int WHI, int THREADS, bool PAD>
__device__ __forceinline__ uint32_t tiles_scan(uint32_t mine, uint32_t *s_group, uint32_t &slots) {
  constexpr int kLanes = kScanLanes<THREADS>, kGroups = 2 * WHI;
  static_assert(kGroups <= 32, "a lane per group");
  const int lane = threadIdx.x & 31, group = threadIdx.x / kLanes, part = threadIdx.x % kLanes;
  uint32_t upto = mine;
  for (int d = 1; d < kLanes; d <<= 1) {
    const uint32_t o = __shfl_up_sync(0xffffffffu, upto, d, kLanes);
    if (part >= d) upto += o;
  }
  if (group < kGroups && part == kLanes - 1) s_group[group] = upto;
  __syncthreads();
  const uint32_t n = lane < kGroups ? s_group[lane] : 0u, width = PAD ? (n + 31u) & ~31u : n;
  uint32_t end = width;
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t o = __shfl_up_sync(0xffffffffu, end, d);
    if (lane >= d) end += o;
  }
  slots = __shfl_sync(0xffffffffu, end, 31);
  return __shfl_sync(0xffffffffu, end - width, group & 31) + upto - mine;
}

// Classifies and sorts a tile.  On return (after a barrier) t.list holds the
// pairs' indices by key, each group's from a multiple of 32 slots, empty slots
// kNoSlot.  Returns the slots used.  Pairs that are settled have no slot, their
// result (accept or result byte << 16 | count) is in t.off.
template <int WHI>
__device__ __forceinline__ uint32_t tile_sort(const BatchArgs &b, uint32_t tile, const TileArrays &t, uint32_t *s_n,
                                              uint32_t *s_group) {
  constexpr int kGroups = 2 * WHI, kBatch = kTilesPairs / kTilesThreads;
  const FilterArgs &a = b.f;
  const int lane = threadIdx.x & 31;
  const uint64_t base = blockIdx.x * (uint64_t)tile;
  const uint32_t n_here = (uint32_t)min_u64(tile, a.n_pairs - base);
  for (int i = threadIdx.x; i < kGroups * (int)kShiftClasses; i += kTilesThreads) s_n[i] = 0;
  for (uint32_t i = threadIdx.x; i < tile + kGroups * 32; i += kTilesThreads) t.list[i] = kNoSlot;
  __syncthreads();
  PairBatch<kBatch, kTilesThreads> x;
  x.load(b, base, n_here);
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
  constexpr int kKeys4 = kScanKeys<kTilesThreads> / 4;
  const bool has = threadIdx.x < kGroups * kScanLanes<kTilesThreads>;
  uint4 *keys = reinterpret_cast<uint4 *>(s_n) + threadIdx.x * kKeys4, n[kKeys4];
  uint32_t mine = 0, slots;
#pragma unroll
  for (int k = 0; k < kKeys4; ++k) {
    n[k] = has ? keys[k] : make_uint4(0u, 0u, 0u, 0u);
    mine += n[k].x + n[k].y + n[k].z + n[k].w;
  }
  uint32_t at = tiles_scan<WHI, kTilesThreads, true>(mine, s_group, slots);
#pragma unroll
  for (int k = 0; k < kKeys4; ++k) {
    if (has) keys[k] = make_uint4(at, at + n[k].x, at + n[k].x + n[k].y, at + n[k].x + n[k].y + n[k].z);
    at += n[k].x + n[k].y + n[k].z + n[k].w;
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < n_here; i += kTilesThreads) {
    const uint32_t key = t.key[i];
    if (key != kNoSlot) t.list[atomicAdd(&s_n[key], 1u)] = (uint16_t)i;
  }
  __syncthreads();
  return slots;
}

// Resident blocks of tiles_kernel per SM.
template <int WHI>
constexpr int kTilesBlocks = WHI <= 4 ? 4 : (WHI <= 10 ? 2 : 1);

// Reads of at most WHI words (the row stride bounds them): sorted and filtered.
template <int WHI>
__global__ void __launch_bounds__(kTilesThreads, kTilesBlocks<WHI>)
    tiles_kernel(const BatchArgs b, uint32_t tile) {
  extern __shared__ uint32_t s_mem[];
  __shared__ __align__(16) uint32_t s_n[2 * WHI * kShiftClasses];
  __shared__ uint32_t s_group[2 * WHI], s_next;
  const TileArrays t(s_mem, tile, 2 * WHI);
  const FilterArgs &a = b.f;
  const int lane = threadIdx.x & 31;
  const uint64_t base = blockIdx.x * (uint64_t)tile;
  const uint32_t n_here = (uint32_t)min_u64(tile, a.n_pairs - base);
  if (threadIdx.x == 0) s_next = 0;
  const uint32_t slots = tile_sort<WHI>(b, tile, t, s_n, s_group);

  // ---- filter: 32 list slots at a time, the heaviest first ----
  for (;;) {
    uint32_t s = 0;
    if (lane == 0) s = atomicAdd(&s_next, 32u);
    s = __shfl_sync(0xffffffffu, s, 0);
    if (s >= slots) break;
    const uint32_t i = t.list[s + (uint32_t)lane];
    const uint32_t group = t.key[t.list[s]] / kShiftClasses;  // the warp's; its first slot is never padding
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
// launches' item counters.  A tile is a cluster of kPlanCluster blocks, which
// add up their counts per key through each other's shared memory: out of 3584
// pairs, those of one block, a group has so few per threshold that a quarter of
// the filter's warps straddle two and pay for the larger (9M pairs of 36-512
// bp, thresholds of 2, 5 and 10%: sorted by single blocks 2604 us, by four 2109;
// eight wait for each other longer than that gains).  The pairs stay in registers: counting
// atomics without a return value, a scan, then one returning atomic and one
// 16-byte store per pair; L2 joins the stores, which fall into 229 KB.
template <int WHI>
__global__ void __launch_bounds__(kPlanThreads, 1024 / kPlanThreads) plan_kernel(const BatchArgs b, uint32_t *desc) {
  namespace cg = cooperative_groups;
  constexpr int kGroups = 2 * WHI;
  constexpr int kKeys4 = kScanKeys<kPlanThreads> / 4;
  __shared__ __align__(16) uint32_t s_n[kGroups * kShiftClasses], s_at[kGroups * kShiftClasses];
  __shared__ uint32_t s_group[kGroups];
  const cg::cluster_group cluster = cg::this_cluster();
  const FilterArgs &a = b.f;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster.block_rank(), tile = blockIdx.x / kPlanCluster;
  const uint64_t base = min_u64(blockIdx.x * (uint64_t)kBlockPairs, a.n_pairs);  // the last cluster's blocks may be past the end
  const uint32_t n_here = (uint32_t)min_u64(kBlockPairs, a.n_pairs - base);
  if (blockIdx.x == 0 && threadIdx.x < 8) b.s.counters[threadIdx.x] = 0;
  for (int i = threadIdx.x; i < kGroups * (int)kShiftClasses; i += kPlanThreads) s_n[i] = 0;
  PairBatch<kPlanPer, kPlanThreads> x;
  x.load(b, base, n_here);
  __syncthreads();
  // A pair to filter: threshold, length << 8, key << 18 (registers: three words a pair).
  constexpr uint32_t kNone = 0xffffffffu;
  static_assert(GK_MAX_LEN < 1024 && 2 * 16 * kShiftClasses < (1u << 14), "fields of a word");
  uint32_t pair[kPlanPer];
#pragma unroll
  for (int r = 0; r < kPlanPer; ++r) {
    const uint32_t i = (uint32_t)r * kPlanThreads + threadIdx.x;
    const bool active = i < n_here;
    const int status = x.status(a, r);
    if (a.err_count) {
      const unsigned bad = __ballot_sync(0xffffffffu, active && status == 2);
      if (bad && lane == 0) atomicAdd(a.err_count, (unsigned)__popc(bad));
    }
    pair[r] = kNone;
    if (active && status == 0) {
      const uint32_t key = tiles_key<WHI>(a, x.m[r], x.e[r]);
      atomicAdd(&s_n[key], 1u);
      pair[r] = x.e[r] | (x.m[r] << 8) | (key << 18);
    } else if (active) {
      write_trivial(a, base + i, status == 3 ? 0 : status);  // an empty read: count 0, accepted
    }
  }
  cluster.sync();  // every block's counts are in its s_n, which stays as it is
  const bool has = threadIdx.x < kGroups * kScanLanes<kPlanThreads>;
  uint4 all[kKeys4], before[kKeys4];  // of this thread's keys: in the cluster, in the blocks before
  uint32_t mine = 0;
#pragma unroll
  for (int i = 0; i < kKeys4; ++i) {
    all[i] = before[i] = make_uint4(0u, 0u, 0u, 0u);
    if (!has) continue;
#pragma unroll
    for (uint32_t k = 0; k < kPlanCluster; ++k) {
      const uint4 n = reinterpret_cast<const uint4 *>(cluster.map_shared_rank(s_n, k))[threadIdx.x * kKeys4 + i];
      if (k == rank) before[i] = all[i];
      all[i].x += n.x;
      all[i].y += n.y;
      all[i].z += n.z;
      all[i].w += n.w;
    }
    mine += all[i].x + all[i].y + all[i].z + all[i].w;
  }
  cluster.barrier_arrive();  // done with the other blocks' memory; waited for before the block ends
  uint32_t slots;
  const uint32_t first = tiles_scan<WHI, kPlanThreads, false>(mine, s_group, slots);
  uint32_t at = first;
#pragma unroll
  for (int i = 0; i < kKeys4; ++i) {
    const uint4 n = all[i], o = before[i];
    if (has)
      reinterpret_cast<uint4 *>(s_at)[threadIdx.x * kKeys4 + i] =
          make_uint4(at + o.x, at + n.x + o.y, at + n.x + n.y + o.z, at + n.x + n.y + n.z + o.w);
    at += n.x + n.y + n.z + n.w;
  }
  if (rank == 0 && has && threadIdx.x % kScanLanes<kPlanThreads> == 0) {
    const uint32_t group = threadIdx.x / kScanLanes<kPlanThreads>;
    desc[(uint64_t)group * (gridDim.x / kPlanCluster) + tile] = first | (s_group[group] << 16);
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kPlanPer; ++r)
    if (pair[r] != kNone)
      b.s.rec[(uint64_t)tile * kPlanPairs + atomicAdd(&s_at[pair[r] >> 18], 1u)] =
          make_uint4((uint32_t)base + (uint32_t)r * kPlanThreads + threadIdx.x, x.rid[r], x.off[r],
                     (pair[r] & 0xFFu) | ((pair[r] >> 8 & 0x3FFu) << 16));
  cluster.barrier_wait();
}

// The groups of reads of WLO .. WTOP words out of records planned for reads of
// at most WHI: persistent blocks take one group of one tile at a time, all tiles
// of the longest reads first, in slices of per records: about a quarter of a
// block's share, a multiple of the block up to kSliceRecords.  A tile's last
// slice takes what is left.  How many slices a group needs follows from 32
// tiles, evenly spread (the same tiles for every block).  A group's slices of
// the largest shift counts of all tiles come first, so that the last items to
// end are short; up to 4 words a tile's slices follow each other, because memory
// bounds those and the slices write to the same sectors (50M pairs of 50-300 bp,
// the launch for those of up to 128: 0.81 -> 0.63 ms).
constexpr uint32_t kSliceRecords = 1024;

template <int WHI, int WLO, int WTOP>
__global__ void __launch_bounds__(kGroupThreads, WTOP <= 4 ? 8 : (WTOP <= 5 ? 6 : (WTOP <= 10 ? 4 : 2)))
    groups_kernel(const BatchArgs b, uint32_t tiles, const uint32_t *desc, uint32_t *counter) {
  constexpr uint32_t kFirst = 2 * (WHI - WTOP), kCount = 2 * (WTOP - WLO + 1);
  __shared__ uint32_t s_item, s_sum[kCount], s_slices[kCount], s_per;
  const FilterArgs &a = b.f;
  for (uint32_t g = threadIdx.x / 32; g < kCount; g += kGroupThreads / 32) {
    const uint32_t at = (uint32_t)((uint64_t)tiles * (threadIdx.x & 31u) / 32u);
    const uint32_t count = desc[(uint64_t)(kFirst + g) * tiles + at] >> 16;
    const uint32_t sum = __reduce_add_sync(0xffffffffu, count), most = __reduce_max_sync(0xffffffffu, count);
    if ((threadIdx.x & 31u) == 0) {
      s_sum[g] = sum;
      s_slices[g] = most;
    }
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    const uint32_t sum = __reduce_add_sync(0xffffffffu, threadIdx.x < kCount ? s_sum[threadIdx.x] : 0u);
    const uint32_t share = (uint32_t)min_u64(kSliceRecords, (uint64_t)sum * tiles / 32u / (4u * gridDim.x));
    const uint32_t per = max(1u, share / kGroupThreads) * kGroupThreads;
    if (threadIdx.x < kCount) s_slices[threadIdx.x] = max(1u, (s_slices[threadIdx.x] + per - 1) / per);
    if (threadIdx.x == 0) s_per = per;
  }
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) s_item = atomicAdd(counter, 1u);
    __syncthreads();
    uint32_t item = s_item, g = 0, slices = s_slices[0];
    while (g < kCount && item >= tiles * slices) {
      item -= tiles * slices;
      if (++g < kCount) slices = s_slices[g];
    }
    if (g == kCount) break;
    const uint32_t group = kFirst + g;
    const uint32_t slice = WTOP <= 4 ? item % slices : item / tiles, tile = WTOP <= 4 ? item / slices : item % tiles;
    const uint32_t d = desc[(uint64_t)group * tiles + tile];
    const uint32_t count = d >> 16, from = min(count, slice * s_per);
    const uint32_t n = (slice + 1 < slices ? min(count, from + s_per) : count) - from;
    const uint4 *recs = b.s.rec + (uint64_t)tile * kPlanPairs + (d & 0xFFFFu) + from;
    // The next pair's record is loaded while this one's words are.
    uint4 next = threadIdx.x < n ? recs[threadIdx.x] : make_uint4(0u, 0u, 0u, 0u);
    for (uint32_t j = threadIdx.x; j < n; j += kGroupThreads) {
      const uint4 rec = next;
      if (j + kGroupThreads < n) next = recs[j + kGroupThreads];
      const uint32_t e = rec.w & 0xFFFFu;
      write_count(a, rec.x, tiles_count<WHI, WLO, WTOP>(a, group, rec.y, rec.z, rec.w >> 16, e), e);
    }
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
  uint32_t *desc = b.s.km;  // 2 WHI <= 32 words per tile, out of a word per pair
  cudaLaunchAttribute cluster{};
  cluster.id = cudaLaunchAttributeClusterDimension;
  cluster.val.clusterDim.x = kPlanCluster;
  cluster.val.clusterDim.y = cluster.val.clusterDim.z = 1;
  cudaLaunchConfig_t config{};
  config.gridDim = dim3(tiles * kPlanCluster);
  config.blockDim = dim3(kPlanThreads);
  config.stream = stream;
  config.attrs = &cluster;
  config.numAttrs = 1;
  err = cudaLaunchKernelEx(&config, plan_kernel<WHI>, b, desc);
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
