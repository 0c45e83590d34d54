// k_segsort.cuh -- the local half of the hybrid radix sort (K3 / STEP-2 and
// STEP-3).  The global passes (unordered partitions, k_msd.cuh, or ordered
// onesweep passes) bring the keys into groups that share their high bits, in
// ascending order of those bits.  One CTA then finishes a run of whole groups
// in shared memory: tile t covers [bound[t], bound[t+1]), where bound[t] is
// the start of the group holding position t * TILE_T, so no group is split
// between CTAs and no run of equal keys crosses a tile boundary.
//
// A tile longer than the shared-memory capacity (it holds a group of more
// keys than that, e.g. a tandem repeat's (k+1)-mer) is "oversize": all
// oversize tiles are gathered into one buffer, which is sorted over every
// digit by the ordered global passes; the results then go back into place.
//
// Edge keys (STEP-2): k_seg_count counts a tile's copies in a hash table and
// orders the distinct keys; a tile with few copies of each key is ranked copy
// by copy (k_rank_rle); k_seg_rle, by 8-bit digit passes, takes what neither
// can.  Each writes the tile's distinct keys and multiplicities at the front
// of its own range, from where k_endpoints_tiles reads them (or k_seg_compact
// packs them).
// Node records (STEP-3): k_seg_rank ranks records within small buckets, by
// key and payload; k_seg_sort, by digit passes, takes tiles with crowded
// buckets (256 threads of 24 items, or 384 of 16 in its wide form).
#pragma once

#include "k_build.cuh"

namespace dbg {

constexpr int SEG_BLOCK = 256;

template <class K, bool HAS_VAL, int ITEMS, int BLOCK = SEG_BLOCK>
struct SegSortSmem {
  static constexpr int WARPS = BLOCK / 32;
  static constexpr int CAP = BLOCK * ITEMS;
  K keys[CAP];
  uint32_t vals[HAS_VAL ? CAP : 1];
  uint32_t whist[WARPS][RADIX];
  uint32_t match[WARPS][RADIX + 1];
  uint32_t cnt[ITEMS * WARPS + 1];
  uint32_t hpos[HAS_VAL ? 1 : CAP + 1];  // run heads' positions by rank (run-length reduce)
  uint32_t tmp[8];
  uint64_t bound[2];
  K base, range;
  uint32_t tile, passes, excl, total, span_bits;
};

// The order of records with equal keys: ascending payload << shift (the
// shift drops the side bits that a node record's payload carries on top).
// sort: they come in no particular order and payload digits take part in the
// digit passes; otherwise they come in that order and stable passes keep it.
// pb: enough bits for every (payload << shift >> shift) >> 1 of a record that
// is an edge end, with all ones left for REC_NONE.  dups: records may be equal.
struct ValOrder {
  int shift = 0;
  int sort = 0;
  int pb = 32;
  int dups = 1;
};

// bound[t] for t in [0, tiles]: the first index of the group holding
// position t * tile_keys (n for positions past the end).  The high bits are
// sorted, so a binary search finds it; it starts in the last 8192 keys
// before the position unless the group is longer.
template <class K>
__global__ void k_seg_bounds(const K *__restrict__ keys, uint64_t n, int low_bits, uint64_t tile_keys,
                             uint64_t tiles, uint64_t *__restrict__ bound) {
  for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t <= tiles; t += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t pos = t * tile_keys;
    uint64_t b;
    if (t == tiles || pos >= n) {
      b = n;
    } else if (pos == 0) {
      b = 0;
    } else {
      const K target = KeyOps<K>::shr(keys[pos], low_bits);
      uint64_t lo = pos > 8192 ? pos - 8192 : 0, hi = pos;
      if (lo > 0 && !KeyOps<K>::less(KeyOps<K>::shr(keys[lo], low_bits), target)) lo = 0;
      while (lo < hi) {  // first index whose high bits are not below target
        const uint64_t mid = lo + (hi - lo) / 2;
        if (KeyOps<K>::less(KeyOps<K>::shr(keys[mid], low_bits), target)) lo = mid + 1;
        else hi = mid;
      }
      b = lo;
    }
    bound[t] = b;
  }
}

// osize[t] = the tile's length if it exceeds cap (an oversize tile), else 0;
// those tiles' numbers in olist, their keys added up in *keys, and in *mixed
// those of tiles that do not look like the copies of one key.  If a wait of
// the global passes ran out (*err), some keys were never written: then every
// tile is made empty, so that the local kernels, which trust the keys to lie in
// their groups, read none, and the host finds the error in its next read-back.
template <class K>
__global__ void k_seg_oversize(const K *__restrict__ kin, uint64_t *__restrict__ bound, uint64_t tiles, uint32_t cap,
                               uint32_t *__restrict__ osize, uint32_t *__restrict__ olist,
                               uint32_t *__restrict__ keys, uint32_t *__restrict__ mixed,
                               uint32_t *__restrict__ count, const uint32_t *__restrict__ err) {
  for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < tiles; t += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t gave_up = *err & (ERR_TIMEOUT | ERR_INTERNAL);  // (loaded with the bounds)
    const uint64_t s = bound[t], sz = bound[t + 1] - s;
    if (gave_up) {
      bound[t] = 0;
      osize[t] = 0;
      if (t == tiles - 1) bound[tiles] = 0;
      continue;
    }
    osize[t] = sz > cap ? (uint32_t)sz : 0u;
    if (sz > cap) {
      atomicAdd(keys, (uint32_t)sz);
      if (!copies_of_one(kin, s, sz)) atomicAdd(mixed, (uint32_t)sz);
      olist[atomicAdd(count, 1u)] = (uint32_t)t;
    }
  }
}

// The gathered, sorted records back into their tiles' ranges.
template <class K>
__global__ void k_seg_place(const uint64_t *__restrict__ bound, const uint32_t *__restrict__ osize,
                            const uint64_t *__restrict__ ooff, const uint32_t *__restrict__ olist, uint32_t n,
                            const K *__restrict__ gk, const uint32_t *__restrict__ gv, K *__restrict__ kout,
                            uint32_t *__restrict__ vout) {
  for (uint32_t q = blockIdx.x; q < n; q += gridDim.x) {
    const uint32_t t = olist[q];
    const uint64_t s = bound[t], o = ooff[t];
    for (uint32_t j = threadIdx.x; j < osize[t]; j += blockDim.x) {
      kout[s + j] = gk[o + j];
      vout[s + j] = gv[o + j];
    }
  }
}

// Gathered records that come in no order are sorted by payload before the
// stable sort by key: the words (payload << shift) << 32 | index are sorted by
// their upper half, and the records follow.
static __global__ void k_val_words(const uint32_t *__restrict__ v, uint64_t n, int shift, uint64_t *__restrict__ w) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
    w[i] = (uint64_t)(v[i] << shift) << 32 | (uint32_t)i;
}
template <class K>
__global__ void k_permute(const uint64_t *__restrict__ w, uint64_t n, const K *__restrict__ kin,
                          const uint32_t *__restrict__ vin, K *__restrict__ kout, uint32_t *__restrict__ vout) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t j = (uint32_t)w[i];
    if (j >= n) continue;  // (a wait of the words' sort ran out: the host finds the error)
    kout[i] = kin[j];
    vout[i] = vin[j];
  }
}

// Copies every oversize tile to gk[ooff[t] ...] (and its payloads), in tile
// order, so that one sort of the gathered keys sorts each of them.
template <class K, bool HAS_VAL>
__global__ void k_seg_gather(const K *__restrict__ kin, const uint32_t *__restrict__ vin,
                             const uint64_t *__restrict__ bound, const uint32_t *__restrict__ osize,
                             const uint64_t *__restrict__ ooff, uint64_t tiles, K *__restrict__ gk,
                             uint32_t *__restrict__ gv) {
  for (uint64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const uint32_t sz = osize[t];
    if (sz == 0) continue;
    const uint64_t s = bound[t], o = ooff[t];
    for (uint32_t j = threadIdx.x; j < sz; j += blockDim.x) {
      gk[o + j] = kin[s + j];
      if (HAS_VAL) gv[o + j] = vin[s + j];
    }
  }
}

// The tile's range, its base (the first key with its group's low bits
// cleared: no key of the tile is below it) and, from the last key with its
// group's low bits set, the bits that key offsets span and the number of
// local passes over them, into shared memory.  There is always one pass: a
// tile of copies of one key, in a group with no bits below it, spans no bits,
// and the digit passes are also what puts the keys into shared memory.  The
// caller checks that the tile is not oversize.
template <class K, class S>
__device__ __forceinline__ void seg_setup(S &sm, const K *__restrict__ kin, const uint64_t *__restrict__ bound,
                                          uint32_t tile, LowBits lb) {
  if (threadIdx.x == 0) {
    const uint64_t s = bound[tile], e = bound[tile + 1];
    sm.bound[0] = s;
    sm.bound[1] = e;
    if (e > s) {
      const K first = kin[s], last = kin[e - 1];
      int low_first = lb.unsplit(first), low_last = lb.unsplit(last);  // (both loads in flight)
      if (lb.split) {
        low_first -= lb.taken(first, low_first);
        low_last -= lb.taken(last, low_last);
      }
      sm.base = KeyOps<K>::sub(first, KeyOps<K>::mask_low(first, low_first));
      const K range = KeyOps<K>::sub(KeyOps<K>::fill_low(last, low_last), sm.base);
      sm.span_bits = (uint32_t)KeyOps<K>::bitlen(range);
      sm.passes = max(1u, (sm.span_bits + RADIX_BITS - 1) / RADIX_BITS);
      sm.range = range;
    }
  }
  __syncthreads();
}

// first index in sorted a[0, m) whose value is >= x
__device__ __forceinline__ uint32_t lower_bound_u32(const uint32_t *__restrict__ a, uint32_t m, uint64_t x) {
  uint32_t lo = 0, hi = m;
  while (lo < hi) {
    const uint32_t mid = lo + (hi - lo) / 2;
    if ((uint64_t)a[mid] < x) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// One stable ranking step: item i of this warp gets its rank among the
// warp's equal digits so far, packed as (rank << 9) | digit, with digit
// RADIX for invalid items.  Order: item, then lane.  An item is valid if its
// index wofs + 32 i + lane is below lim.
template <int ITEMS, int RANK, class S, class Digit>
__device__ __forceinline__ void rank_digits(S &sm, uint32_t (&rank)[ITEMS], int nitems, uint32_t wofs, uint32_t lim,
                                            Digit digit) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt_mask = (1u << lane) - 1u;
#pragma unroll
  for (int i = 0; i < ITEMS; i++) {
    if (i >= nitems) break;  // warp-uniform
    const bool valid = wofs + i * 32 + lane < lim;
    const uint32_t d = valid ? digit(i) : (uint32_t)RADIX;
    unsigned peers;
    if (RANK == RANK_MATCH) {
      peers = __match_any_sync(0xffffffffu, d);
    } else if (RANK == RANK_ATOMIC) {
      atomicOr(&sm.match[warp][d], 1u << lane);
      __syncwarp();
      peers = sm.match[warp][d];
      __syncwarp();
      if (lane == __ffs(peers) - 1) sm.match[warp][d] = 0;
    } else {
      peers = 0xffffffffu;
#pragma unroll
      for (int bt = 0; bt <= RADIX_BITS; bt++) {
        const bool bit = (d >> bt) & 1u;
        const unsigned bal = __ballot_sync(0xffffffffu, bit);
        peers &= bit ? bal : ~bal;
      }
    }
    const int leader = __ffs(peers) - 1;
    uint32_t before = 0;
    if (lane == leader && valid) {
      before = sm.whist[warp][d];
      sm.whist[warp][d] = before + __popc(peers);
    }
    before = __shfl_sync(0xffffffffu, before, leader);
    rank[i] = ((before + __popc(peers & lt_mask)) << 9) | d;
    __syncwarp();
  }
}
template <class K, int ITEMS, int RANK, class S>
__device__ __forceinline__ void rank_items(S &sm, const K (&key)[ITEMS], uint32_t (&rank)[ITEMS], int nitems,
                                           uint32_t wofs, uint32_t lim, int shift) {
  rank_digits<ITEMS, RANK>(sm, rank, nitems, wofs, lim,
                           [&](int i) { return KeyOps<K>::digit(key[i], shift, RADIX_BITS); });
}

// Turns the per-warp digit counts into each warp's first position per digit
// (digit-major, then warp); returns the number of ranked keys to all threads.
template <class S>
__device__ __forceinline__ uint32_t digit_positions(S &sm) {
  const int tid = threadIdx.x;
  __syncthreads();
  uint32_t c = 0;
  if (tid < RADIX)
#pragma unroll
    for (int w = 0; w < S::WARPS; w++) c += sm.whist[w][tid];
  const uint32_t start = block_excl_scan_256(c, sm.tmp);
  if (tid < RADIX) {
    uint32_t run = start;
#pragma unroll
    for (int w = 0; w < S::WARPS; w++) {
      const uint32_t x = sm.whist[w][tid];
      sm.whist[w][tid] = run;
      run += x;
    }
    if (tid == RADIX - 1) sm.total = run;
  }
  __syncthreads();
  return sm.total;
}

template <class K, bool HAS_VAL, int ITEMS, class S>
__device__ __forceinline__ void scatter_items(S &sm, const K (&key)[ITEMS], const uint32_t (&val)[ITEMS],
                                              const uint32_t (&rank)[ITEMS], int nitems) {
  const int warp = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < ITEMS; i++) {
    if (i >= nitems) break;
    const uint32_t d = rank[i] & 0x1ffu;
    if (d < RADIX) {
      const uint32_t q = sm.whist[warp][d] + (rank[i] >> 9);
      sm.keys[q] = key[i];
      if (HAS_VAL) sm.vals[q] = val[i];
    }
  }
}

// Loads the consecutive keys [wofs, wofs + 32 * nitems) of the staging area
// (item-major; valid below lim) and zeroes the warp counters for the next
// pass.  The caller synchronises before ranking.
template <class K, bool HAS_VAL, int ITEMS, class S>
__device__ __forceinline__ void reload_items(S &sm, K (&key)[ITEMS], uint32_t (&val)[ITEMS], int nitems,
                                             uint32_t wofs, uint32_t lim) {
  const int lane = threadIdx.x & 31;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < ITEMS; i++) {
    if (i >= nitems) break;
    const uint32_t j = wofs + i * 32 + lane;
    if (j < lim) {
      key[i] = sm.keys[j];
      if (HAS_VAL) val[i] = sm.vals[j];
    }
  }
  for (int i = threadIdx.x; i < S::WARPS * RADIX; i += S::WARPS * 32) (&sm.whist[0][0])[i] = 0;
}

// Records: tile t sorted in shared memory into kout / vout at its own range;
// an oversize tile copies its slice of the gathered, globally sorted records
// (gk / gv at ooff[t]).
template <class K, int ITEMS, int RANK, int BLOCK>
__device__ __forceinline__ void seg_sort_tile(
    SegSortSmem<K, true, ITEMS, BLOCK> &sm, uint32_t tile, const K *__restrict__ kin, const uint32_t *__restrict__ vin,
    const uint64_t *__restrict__ bound, const uint32_t *__restrict__ osize, const uint64_t *__restrict__ ooff,
    const K *__restrict__ gk, const uint32_t *__restrict__ gv, K *__restrict__ kout, uint32_t *__restrict__ vout,
    LowBits lb, ValOrder vo) {
  using S = SegSortSmem<K, true, ITEMS, BLOCK>;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (osize[tile]) {
    const uint64_t s = bound[tile], o = ooff[tile];
    for (uint32_t j = tid; j < osize[tile]; j += BLOCK) {
      kout[s + j] = gk[o + j];
      vout[s + j] = gv[o + j];
    }
    return;
  }
  for (int i = tid; i < S::WARPS * RADIX; i += BLOCK) (&sm.whist[0][0])[i] = 0;
  for (int i = tid; i < S::WARPS * (RADIX + 1); i += BLOCK) (&sm.match[0][0])[i] = 0;
  seg_setup<K>(sm, kin, bound, tile, lb);
  const uint64_t s = sm.bound[0];
  const uint32_t cnt = (uint32_t)(sm.bound[1] - s);
  if (cnt == 0) return;
  const K base = sm.base;
  const int passes = (int)sm.passes;
  // the keys spread evenly over the warps: warp w holds the consecutive
  // keys [w * 32 * ipw, (w + 1) * 32 * ipw), item-major
  const int ipw = (int)((cnt + BLOCK - 1) / BLOCK);
  const uint32_t wofs = (uint32_t)warp * 32u * ipw;
  K key[ITEMS];
  uint32_t val[ITEMS];
  uint32_t rank[ITEMS];
#pragma unroll
  for (int i = 0; i < ITEMS; i++) {
    const uint32_t j = wofs + i * 32 + lane;
    const bool in = i < ipw && j < cnt;
    key[i] = in ? KeyOps<K>::sub(kin[s + j], base) : KeyOps<K>::zero();
    val[i] = in ? vin[s + j] : 0u;
  }
  // records that come in no order: their payloads' digits first
  const int vpasses = vo.sort ? 4 : 0;
  for (int p = 0; p < vpasses + passes; p++) {
    if (p > 0) {
      reload_items<K, true, ITEMS>(sm, key, val, ipw, wofs, cnt);
      __syncthreads();
    }
    if (p < vpasses)
      rank_digits<ITEMS, RANK>(sm, rank, ipw, wofs, cnt,
                               [&](int i) { return ((val[i] << vo.shift) >> (p * RADIX_BITS)) & 0xffu; });
    else
      rank_items<K, ITEMS, RANK>(sm, key, rank, ipw, wofs, cnt, (p - vpasses) * RADIX_BITS);
    digit_positions(sm);
    scatter_items<K, true, ITEMS>(sm, key, val, rank, ipw);
  }
  __syncthreads();
  for (uint32_t j = tid; j < cnt; j += BLOCK) {
    kout[s + j] = KeyOps<K>::add(sm.keys[j], base);
    vout[s + j] = sm.vals[j];
  }
}

// One CTA per tile; or, with a tile list, a grid of CTAs that take the
// *list_count listed tiles in turn.
template <class K, int ITEMS, int RANK, int BLOCK = SEG_BLOCK>
__global__ __launch_bounds__(BLOCK, 2) void k_seg_sort(
    const K *__restrict__ kin, const uint32_t *__restrict__ vin, const uint64_t *__restrict__ bound,
    const uint32_t *__restrict__ osize, const uint64_t *__restrict__ ooff, const K *__restrict__ gk,
    const uint32_t *__restrict__ gv, K *__restrict__ kout, uint32_t *__restrict__ vout, LowBits lb, ValOrder vo,
    const uint32_t *__restrict__ tile_list = nullptr, const uint32_t *__restrict__ list_count = nullptr) {
  using S = SegSortSmem<K, true, ITEMS, BLOCK>;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  S &sm = *reinterpret_cast<S *>(smem_raw);
  if (!tile_list) {
    seg_sort_tile<K, ITEMS, RANK, BLOCK>(sm, blockIdx.x, kin, vin, bound, osize, ooff, gk, gv, kout, vout, lb, vo);
    return;
  }
  const uint32_t n = *list_count;
  for (uint32_t q = blockIdx.x; q < n; q += gridDim.x) {
    seg_sort_tile<K, ITEMS, RANK, BLOCK>(sm, tile_list[q], kin, vin, bound, osize, ooff, gk, gv, kout, vout,
                                         lb, vo);
    __syncthreads();
  }
}

// Records by ranking within small buckets.  The tile's records are spread
// over 8192 buckets (4096 for 128-bit keys, whose tiles are half as long) by
// the top bits of their key offsets (a counting sort in
// shared memory: one atomic add per record, a scan, one scatter), and a
// record's place in the sorted tile is its bucket's start plus the number of
// the bucket's records that precede it: those with a smaller key, or an
// equal key and a smaller payload.  A bucket holds a node's own records and
// seldom another node's, so that is a few comparisons per record, and they
// need no particular order on arrival.  A tile with a bucket longer than
// RANK_GROUP_MAX is listed in fb_list for the digit-pass kernel instead.
//
// Bound by instruction issue.  Where a record's bits below its bucket's and
// its payload's upper bits fit 64 bits (vo.pb of them; nearly every tile of
// 64-bit keys), they form one word that a single comparison orders; the
// bucket, the payload's lowest bit (an edge end's role: the tie-break where it
// has no room in the word) and its side bits are in 16 bits beside it.  Two CTAs of 512 threads per SM.
//
// FUSED (STEP-3's node records): instead of the sorted keys, the tile's
// distinct keys go to the front of its own range of kout, with their number
// in tcount, and a bit per record that starts a node to `heads` -- record j
// of tile t at bit j % 32 of word (first record of t) / 32 + t + j / 32.
constexpr int RANK_BLOCK = 512;
constexpr uint32_t RANK_GROUP_MAX = 512;

__device__ __forceinline__ uint32_t *head_words(uint32_t *heads, uint64_t first, uint32_t tile) {
  return heads + (first >> 5) + tile;
}

template <class K>
struct SegRankSmem {
  static constexpr int CAP = SEG_BLOCK * (sizeof(K) == 8 ? 24 : 12);  // the digit-pass kernel's capacity
  static constexpr int ITEMS = CAP / RANK_BLOCK;
  static constexpr int TBITS = sizeof(K) == 8 ? 13 : 12, NB = 1 << TBITS, PER = NB / 2 / RANK_BLOCK;
  union {
    struct {
      K key[CAP];  // offsets from base
      uint32_t val[CAP];
    } g;
    struct {
      uint64_t word[CAP];
      uint16_t ord[CAP];
    } n;
  };
  uint32_t start2[NB / 2 + 1];  // 16 bits per bucket: its records, then its first position
  uint32_t wsum[RANK_BLOCK / 32];
  uint32_t cnt[ITEMS * (RANK_BLOCK / 32) + 1];
  uint64_t bound[2];
  K base, range;
  uint32_t passes, span_bits, maxg;
};

template <class K, bool FUSED>
__global__ __launch_bounds__(RANK_BLOCK, 2) void k_seg_rank(
    const K *__restrict__ kin, const uint32_t *__restrict__ vin, const uint64_t *__restrict__ bound,
    const uint32_t *__restrict__ osize, const uint64_t *__restrict__ ooff, const K *__restrict__ gk,
    const uint32_t *__restrict__ gv, K *__restrict__ kout, uint32_t *__restrict__ vout, LowBits lb, ValOrder vo,
    uint32_t *__restrict__ fb_list, uint32_t *__restrict__ fb_count, uint32_t *__restrict__ heads,
    uint32_t *__restrict__ tcount) {
  using S = SegRankSmem<K>;
  constexpr int ITEMS = S::ITEMS, PER = S::PER;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  S &sm = *reinterpret_cast<S *>(smem_raw);
  uint16_t *const start = reinterpret_cast<uint16_t *>(sm.start2);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t tile = blockIdx.x;
  const uint64_t s = bound[tile];
  if (osize[tile]) {
    if (FUSED) {  // (later: k_seg_place, k_tile_heads)
      if (tid == 0) tcount[tile] = 0;
      return;
    }
    const uint64_t o = ooff[tile];
    for (uint32_t j = tid; j < osize[tile]; j += RANK_BLOCK) {
      kout[s + j] = gk[o + j];
      vout[s + j] = gv[o + j];
    }
    return;
  }
  const uint32_t cnt = (uint32_t)(bound[tile + 1] - s);
  if (cnt == 0) {
    if (FUSED && tid == 0) tcount[tile] = 0;
    return;
  }
  const int items = (int)((cnt + RANK_BLOCK - 1) / RANK_BLOCK);  // of each thread
  K key[ITEMS];
  uint32_t val[ITEMS], oa[ITEMS];  // bucket, place on arrival << 13
#pragma unroll
  for (int i = 0; i < ITEMS; i++) {
    if (i >= items) break;
    const uint32_t j = (uint32_t)i * RANK_BLOCK + tid;
    if (j < cnt) {
      key[i] = kin[s + j];
      val[i] = vin[s + j];
    }
  }
  for (int j = tid; j <= S::NB / 2; j += RANK_BLOCK) sm.start2[j] = 0;
  if (tid == 0) sm.maxg = 0;
  seg_setup<K>(sm, kin, bound, tile, lb);  // synchronises
  const K base = sm.base;
  const int bshift = (int)sm.span_bits > S::TBITS ? (int)sm.span_bits - S::TBITS : 0;
  const bool narrow = sizeof(K) == 8 && bshift + vo.pb <= 64;
#pragma unroll
  for (int i = 0; i < ITEMS; i++) {
    if (i >= items) break;
    if ((uint32_t)i * RANK_BLOCK + tid < cnt) {
      key[i] = KeyOps<K>::sub(key[i], base);
      const uint32_t o = (uint32_t)KeyOps<K>::words_lo(KeyOps<K>::shr(key[i], bshift)), h = 16 * (o & 1u);
      oa[i] = o | ((atomicAdd(&sm.start2[o >> 1], 1u << h) >> h) & 0xffffu) << S::TBITS;
    }
  }
  __syncthreads();
  // exclusive scan, 2 PER consecutive buckets per thread
  uint32_t c[PER], sum = 0, mx = 0;
#pragma unroll
  for (int j = 0; j < PER; j++) {
    c[j] = sm.start2[tid * PER + j];
    const uint32_t c0 = c[j] & 0xffffu, c1 = c[j] >> 16;
    sum += c0 + c1;
    mx = max(mx, max(c0, c1));
  }
  const uint32_t incl = warp_incl_scan(sum);
  if (lane == 31) sm.wsum[warp] = incl;
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0 && mx > RANK_GROUP_MAX) sm.maxg = mx;
  __syncthreads();
  if (sm.maxg) {
    if (tid == 0) {
      fb_list[atomicAdd(fb_count, 1u)] = tile;
      if (FUSED) tcount[tile] = 0;
    }
    return;
  }
  uint32_t run = incl - sum;
  for (int w = 0; w < warp; w++) run += sm.wsum[w];
#pragma unroll
  for (int j = 0; j < PER; j++) {
    const uint32_t c0 = c[j] & 0xffffu, c1 = c[j] >> 16;
    sm.start2[tid * PER + j] = run | (run + c0) << 16;
    run += c0 + c1;
  }
  if (tid == RANK_BLOCK - 1) sm.start2[S::NB / 2] = run;
  __syncthreads();
  // the output, from the sorted tile in shared memory
  auto write_out = [&](auto key_at, auto val_at, auto is_head) {
    if (FUSED) {
      unsigned hb[ITEMS];
#pragma unroll
      for (int i = 0; i < ITEMS; i++) {
        if (i >= items) break;
        const uint32_t j = (uint32_t)i * RANK_BLOCK + tid;
        hb[i] = __ballot_sync(0xffffffffu, j < cnt && is_head(j));
        if (lane == 0) {
          sm.cnt[i * (RANK_BLOCK / 32) + warp] = __popc(hb[i]);
          if (j < cnt) head_words(heads, s, tile)[j >> 5] = hb[i];
        }
      }
      __syncthreads();
      // heads before each warp's 32 records: scanned by one warp
      if (warp == 0) {
        constexpr int NW = ITEMS * (RANK_BLOCK / 32), EACH = (NW + 31) / 32;
        const int nw = items * (RANK_BLOCK / 32);
        uint32_t x[EACH], sum = 0;
#pragma unroll
        for (int j = 0; j < EACH; j++) {
          x[j] = lane * EACH + j < nw ? sm.cnt[lane * EACH + j] : 0u;
          sum += x[j];
        }
        const uint32_t incl = warp_incl_scan(sum);
        uint32_t run = incl - sum;
#pragma unroll
        for (int j = 0; j < EACH; j++) {
          if (lane * EACH + j < nw) sm.cnt[lane * EACH + j] = run;
          run += x[j];
        }
        if (lane == 31) tcount[tile] = incl;
      }
      __syncthreads();
#pragma unroll
      for (int i = 0; i < ITEMS; i++) {
        if (i >= items) break;
        const uint32_t j = (uint32_t)i * RANK_BLOCK + tid;
        if (j < cnt) vout[s + j] = val_at(j);
        if (hb[i] >> lane & 1u)
          kout[s + sm.cnt[i * (RANK_BLOCK / 32) + warp] + __popc(hb[i] & ((1u << lane) - 1u))] = key_at(j);
      }
    } else {
      for (uint32_t j = tid; j < cnt; j += RANK_BLOCK) {
        kout[s + j] = key_at(j);
        vout[s + j] = val_at(j);
      }
    }
  };
  if constexpr (sizeof(K) == 8) {
    if (narrow) {
      // word: the bits below the bucket's at the top, the payload's upper pb
      // bits -- and its lowest, where there is room -- at the bottom
      const int up = 64 - bshift;                      // (64: no bit below the bucket's)
      const int role = up > vo.pb ? 1 : 0;
      const int pbits = vo.pb + role;
      const uint32_t pmask = pbits >= 32 ? 0xffffffffu : (1u << pbits) - 1u, obits = S::NB - 1;
#pragma unroll
      for (int i = 0; i < ITEMS; i++) {
        if (i >= items) break;
        if ((uint32_t)i * RANK_BLOCK + tid < cnt) {
          const uint32_t o = oa[i] & obits, q = start[o] + (oa[i] >> S::TBITS);
          const uint32_t p = val[i] << vo.shift >> vo.shift;
          const uint64_t low = bshift ? key[i] << up : 0ull;
          sm.n.word[q] = low | min(p >> (1 - role), pmask);  // (no edge: all ones, last)
          sm.n.ord[q] = (uint16_t)(o | (p & 1u) << 13 | (vo.shift ? val[i] >> 30 : 0u) << 14);
        }
      }
      __syncthreads();
      const bool ties = vo.dups || !role;
      uint64_t wd[ITEMS];
      uint32_t po[ITEMS];
#pragma unroll
      for (int i = 0; i < ITEMS; i++) {
        if (i >= items) break;
        const uint32_t q = (uint32_t)i * RANK_BLOCK + tid;
        if (q < cnt) {
          const uint64_t d = sm.n.word[q];
          const uint32_t od = sm.n.ord[q], o = od & obits, a = start[o], b = start[o + 1];
          uint32_t r = a;
          if (!ties) {
#pragma unroll 2
            for (uint32_t t = a; t < b; t++) r += sm.n.word[t] < d ? 1u : 0u;
          } else {
            for (uint32_t t = a; t < b; t++) {
              const uint64_t y = sm.n.word[t];
              r += y < d ? 1u : 0u;
              if (y == d && t != q) {  // one edge's two ends at a node, or equal records
                const uint32_t bt = sm.n.ord[t] >> 13 & 1u, bq = od >> 13 & 1u;
                r += bt < bq || (bt == bq && t < q) ? 1u : 0u;
              }
            }
          }
          wd[i] = d;
          po[i] = od | r << 16;
        }
      }
      __syncthreads();
#pragma unroll
      for (int i = 0; i < ITEMS; i++) {
        if (i >= items) break;
        if ((uint32_t)i * RANK_BLOCK + tid < cnt) {
          sm.n.word[po[i] >> 16] = wd[i];
          sm.n.ord[po[i] >> 16] = (uint16_t)po[i];
        }
      }
      __syncthreads();
      write_out(
          [&](uint32_t j) {
            return base + ((uint64_t)(sm.n.ord[j] & obits) << bshift | (bshift ? sm.n.word[j] >> up : 0ull));
          },
          [&](uint32_t j) {
            const uint32_t e = (uint32_t)sm.n.word[j] & pmask, od = sm.n.ord[j];
            const uint32_t v = (role ? e : e << 1 | (od >> 13 & 1u)) | (vo.shift ? (od >> 14) << 30 : 0u);
            return e == pmask ? REC_NONE : v;
          },
          [&](uint32_t j) {
            if (j == 0) return true;
            const uint64_t x = sm.n.word[j] ^ sm.n.word[j - 1];
            return ((uint32_t)(x >> 32) | ((uint32_t)x & ~pmask) |
                    ((uint32_t)(sm.n.ord[j] ^ sm.n.ord[j - 1]) & obits)) != 0;
          });
      return;
    }
  }
#pragma unroll
  for (int i = 0; i < ITEMS; i++)
    if ((uint32_t)i * RANK_BLOCK + tid < cnt) {
      const uint32_t q = start[oa[i] & (S::NB - 1)] + (oa[i] >> S::TBITS);
      sm.g.key[q] = key[i];
      sm.g.val[q] = val[i];
    }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < ITEMS; i++) {
    const uint32_t q = (uint32_t)i * RANK_BLOCK + tid;
    if (q < cnt) {
      const K d = sm.g.key[q];
      const uint32_t v = sm.g.val[q], o = (uint32_t)KeyOps<K>::words_lo(KeyOps<K>::shr(d, bshift));
      const uint32_t a = start[o], b = start[o + 1];
      uint32_t r = a;
      for (uint32_t t = a; t < b; t++) {
        const K y = sm.g.key[t];
        bool before = KeyOps<K>::less(y, d);
        if (KeyOps<K>::eq(y, d)) {
          const uint32_t w = sm.g.val[t] << vo.shift, mine = v << vo.shift;
          before = w < mine || (w == mine && t < q);
        }
        r += before ? 1u : 0u;
      }
      key[i] = d;
      val[i] = v;
      oa[i] = r;
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < ITEMS; i++)
    if ((uint32_t)i * RANK_BLOCK + tid < cnt) {
      sm.g.key[oa[i]] = key[i];
      sm.g.val[oa[i]] = val[i];
    }
  __syncthreads();
  write_out([&](uint32_t j) { return KeyOps<K>::add(sm.g.key[j], base); }, [&](uint32_t j) { return sm.g.val[j]; },
            [&](uint32_t j) { return j == 0 || !KeyOps<K>::eq(sm.g.key[j], sm.g.key[j - 1]); });
}

// FUSED's outputs for tiles that other kernels sorted into keys / vals (the
// n_fb of fb_list and the n_over oversize ones of olist): the heads, their number,
// and the distinct keys moved to the front of the tile.  One CTA per tile at a
// time; a chunk's keys are all in registers before its distinct ones, which
// lie at or before them, are written.
template <class K>
__global__ __launch_bounds__(RANK_BLOCK) void k_tile_heads(K *__restrict__ keys, const uint64_t *__restrict__ bound,
                                                           const uint32_t *__restrict__ fb_list, uint32_t n_fb,
                                                           const uint32_t *__restrict__ olist, uint32_t n_over,
                                                           uint32_t *__restrict__ heads,
                                                           uint32_t *__restrict__ tcount) {
  constexpr int ITEMS = 8;
  constexpr uint32_t CHUNK = RANK_BLOCK * ITEMS;
  __shared__ uint32_t s_cnt[ITEMS * (RANK_BLOCK / 32) + 1];
  __shared__ K s_last;
  const int tid = threadIdx.x, lane = tid & 31;
  for (uint32_t q = blockIdx.x; q < n_fb + n_over; q += gridDim.x) {
    const uint32_t tile = q < n_fb ? fb_list[q] : olist[q - n_fb];
    const uint64_t s = bound[tile], n = bound[tile + 1] - s;
    uint32_t *hw = head_words(heads, s, tile);
    uint64_t out = 0;
    for (uint64_t c = 0; c < n; c += CHUNK) {
      K k[ITEMS];
      bool head[ITEMS];
      uint32_t rk[ITEMS];
#pragma unroll
      for (int i = 0; i < ITEMS; i++) {
        const uint64_t j = c + (uint64_t)i * RANK_BLOCK + tid;
        head[i] = false;
        if (j < n) {
          k[i] = keys[s + j];
          head[i] = j == 0 || !KeyOps<K>::eq(k[i], j == c ? s_last : keys[s + j - 1]);
        }
        const unsigned b = __ballot_sync(0xffffffffu, head[i]);
        if (lane == 0 && j < n) hw[j >> 5] = b;
      }
      const uint32_t count = tile_flag_ranks<RANK_BLOCK, ITEMS>(head, rk, s_cnt);  // synchronises
      if (c + CHUNK - 1 < n && tid == RANK_BLOCK - 1) s_last = k[ITEMS - 1];
#pragma unroll
      for (int i = 0; i < ITEMS; i++)
        if (head[i]) keys[s + out + rk[i]] = k[i];
      out += count;
      __syncthreads();
    }
    if (tid == 0) tcount[tile] = (uint32_t)out;
  }
}

// STEP-3 / STEP-4 from FUSED's outputs: tile t's records, hoff[t] the ID of
// its first node, (ISO) eoff[t] the adjacency slot of its first edge end --
// without reads of exactly k bases every record is an edge end, and a record's
// slot is its own index.  Writes the tile's node keys and row starts, the
// adjacency entries, and the edge ends partitioned by edge range (see
// k_write_nodes).  Reads 4 bytes and a bit per record and 8 or 16 per node.
// Launched with a CTA per tile, so that what the chip writes at one time lies
// together: 2.6 ms for 380 M records (a resident grid that takes every 456th
// tile: 2.9; without the loop the compiler's code is 3 to 6 % slower).
template <class K, bool ISO>
__global__ __launch_bounds__(RANK_BLOCK, ISO ? 2 : 3) void k_node_tiles(
    const uint64_t *__restrict__ bound, uint32_t tiles, const K *__restrict__ ukeys, const uint32_t *__restrict__ vals,
    const uint32_t *__restrict__ heads, const uint32_t *__restrict__ tcount, const uint64_t *__restrict__ hoff,
    const uint64_t *__restrict__ eoff, K *__restrict__ node_keys, uint64_t *__restrict__ row_ptr,
    uint32_t *__restrict__ adj_edge, uint8_t *__restrict__ adj_role, uint8_t *__restrict__ adj_side,
    uint64_t *__restrict__ ends, uint32_t *__restrict__ bucket_fill, int bshift) {
  constexpr int ITEMS = 12, WARPS = RANK_BLOCK / 32;
  constexpr uint32_t CHUNK = RANK_BLOCK * ITEMS;
  __shared__ uint32_t s_word[ITEMS * WARPS], s_pre[ITEMS * WARPS + 1], s_cnt[ISO ? ITEMS * WARPS + 1 : 1];
  __shared__ uint32_t s_bcnt[256], s_bbase[256], s_w[WARPS];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (uint32_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const uint64_t s = bound[tile], n = bound[tile + 1] - s;
    const uint32_t *hw = heads + (s >> 5) + tile;
    uint64_t id0 = hoff[tile], slot0 = ISO ? eoff[tile] : s;
    for (uint32_t u = tid; u < tcount[tile]; u += RANK_BLOCK) node_keys[id0 + u] = ukeys[s + u];
    for (uint64_t c = 0; c < n; c += CHUNK) {
      const uint32_t cnt = (uint32_t)min((uint64_t)CHUNK, n - c);
      const int items = (int)((cnt + RANK_BLOCK - 1) / RANK_BLOCK);
      uint32_t val[ITEMS];
#pragma unroll
      for (int i = 0; i < ITEMS; i++) {
        const uint32_t j = (uint32_t)i * RANK_BLOCK + tid;
        val[i] = j < cnt ? vals[s + c + j] : REC_NONE;
      }
      // heads before each word of 32 records
      uint32_t w = 0, pc = 0;
      if (tid < ITEMS * WARPS) {
        w = (uint32_t)tid * 32 < cnt ? hw[(c >> 5) + tid] : 0u;
        pc = __popc(w);
        s_word[tid] = w;
      }
      if (tid < 256) s_bcnt[tid] = 0;
      const uint32_t incl = warp_incl_scan(pc);
      if (lane == 31) s_w[warp] = incl;
      __syncthreads();
      uint32_t pre = incl - pc;
      for (int x = 0; x < warp; x++) pre += s_w[x];
      if (tid < ITEMS * WARPS) s_pre[tid] = pre;
      if (tid == ITEMS * WARPS - 1) s_pre[ITEMS * WARPS] = pre + pc;
      uint32_t rk[ITEMS];  // an edge end's slot, then its rank in its bucket
      uint32_t n_end = cnt;
      if (ISO) {
        bool end[ITEMS];
#pragma unroll
        for (int i = 0; i < ITEMS; i++) end[i] = val[i] != REC_NONE;
        n_end = tile_flag_ranks<RANK_BLOCK, ITEMS>(end, rk, s_cnt);  // synchronises
      } else {
        __syncthreads();
      }
      auto id_of = [&](int i, uint32_t hb) {
        return (uint32_t)id0 + s_pre[i * WARPS + warp] + __popc(hb & (0xffffffffu >> (31 - lane))) - 1u;
      };
#pragma unroll
      for (int i = 0; i < ITEMS; i++) {
        if (i >= items) break;
        const uint32_t j = (uint32_t)i * RANK_BLOCK + tid;
        if (j < cnt) {
          const uint32_t hb = s_word[i * WARPS + warp];
          const uint64_t slot = slot0 + (ISO ? rk[i] : j);
          if (hb >> lane & 1u) row_ptr[id_of(i, hb)] = slot;
          if (!ISO || val[i] != REC_NONE) {
            if (adj_side) {  // the two side bits on top of the payload
              adj_side[slot] = (uint8_t)(val[i] >> 30);
              val[i] &= 0x3fffffffu;
            }
            adj_edge[slot] = val[i] >> 1;
            adj_role[slot] = (uint8_t)(val[i] & 1u);
            rk[i] = atomicAdd(&s_bcnt[val[i] >> 1 >> bshift], 1u);
          }
        }
      }
      __syncthreads();
      if (tid < 256 && s_bcnt[tid]) s_bbase[tid] = atomicAdd(bucket_fill + tid, s_bcnt[tid]);
      __syncthreads();
#pragma unroll
      for (int i = 0; i < ITEMS; i++) {
        if (i >= items) break;
        if ((uint32_t)i * RANK_BLOCK + tid < cnt && (!ISO || val[i] != REC_NONE)) {
          const uint32_t bk = val[i] >> 1 >> bshift;
          ends[((uint64_t)bk << (bshift + 1)) + s_bbase[bk] + rk[i]] =
              (uint64_t)val[i] << 32 | id_of(i, s_word[i * WARPS + warp]);
        }
      }
      id0 += s_pre[ITEMS * WARPS];
      slot0 += n_end;
      __syncthreads();
    }
    if (tile == tiles - 1 && tid == 0) row_ptr[id0] = slot0;
  }
}

// Edge ends (records that are not REC_NONE) of each tile.
static __global__ __launch_bounds__(256) void k_tile_ends(const uint64_t *__restrict__ bound, uint32_t tiles,
                                                          const uint32_t *__restrict__ vals,
                                                          uint32_t *__restrict__ ecount) {
  __shared__ uint32_t s_sum;
  for (uint32_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    if (threadIdx.x == 0) s_sum = 0;
    __syncthreads();
    uint32_t c = 0;
    for (uint64_t j = bound[tile] + threadIdx.x; j < bound[tile + 1]; j += 256) c += vals[j] != REC_NONE;
    c = __reduce_add_sync(0xffffffffu, c);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(&s_sum, c);
    __syncthreads();
    if (threadIdx.x == 0) ecount[tile] = s_sum;
  }
}

// Edge keys (STEP-2's local pass).  Tile t writes its distinct keys and
// their multiplicities at the start of its own range, ustage / mstage[bound[t]
// ...], and their number to tcount[t]; a scan of tcount and k_seg_compact
// then make the dense edge list.  No tile waits for another.

// The distinct keys of an oversize tile, from the gathered, globally sorted
// and reduced keys (guniq, run heads gheads at the positions of the gathered
// buffer, H runs in all, gheads[H] = its length).
template <class K>
__device__ __forceinline__ void seg_rle_gathered(uint32_t tile, const uint64_t *__restrict__ bound,
                                                 const uint32_t *__restrict__ osize, const uint64_t *__restrict__ ooff,
                                                 const K *__restrict__ guniq, const uint32_t *__restrict__ gheads,
                                                 uint32_t H, K *__restrict__ ustage, uint32_t *__restrict__ mstage,
                                                 uint32_t *__restrict__ tcount) {
  const uint64_t o = ooff[tile], s = bound[tile];
  const uint32_t h0 = lower_bound_u32(gheads, H, o), h1 = lower_bound_u32(gheads, H, o + osize[tile]);
  for (uint32_t r = threadIdx.x; r < h1 - h0; r += blockDim.x) {
    ustage[s + r] = guniq[h0 + r];
    mstage[s + r] = gheads[h0 + r + 1] - gheads[h0 + r];
  }
  if (threadIdx.x == 0) tcount[tile] = h1 - h0;
}

// Block radix local sort + RLE: one CTA per tile (every tile, or the tiles of
// tile_list when it is not null), or a grid of CTAs that take the *list_count
// listed tiles in turn.
template <class K, int ITEMS, int RANK>
__global__ __launch_bounds__(SEG_BLOCK, 2) void k_seg_rle(
    const K *__restrict__ kin, const uint64_t *__restrict__ bound, const uint32_t *__restrict__ osize,
    const uint64_t *__restrict__ ooff, const K *__restrict__ guniq, const uint32_t *__restrict__ gheads, uint32_t H,
    K *__restrict__ ustage, uint32_t *__restrict__ mstage, uint32_t *__restrict__ tcount, LowBits lb,
    const uint32_t *__restrict__ tile_list, const uint32_t *__restrict__ list_count) {
  using S = SegSortSmem<K, false, ITEMS>;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  S &sm = *reinterpret_cast<S *>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t todo = list_count ? *list_count : gridDim.x;
  for (uint32_t q = blockIdx.x; q < todo; q += gridDim.x) {
    const uint32_t tile = tile_list ? tile_list[q] : q;
    if (osize[tile]) {
      seg_rle_gathered<K>(tile, bound, osize, ooff, guniq, gheads, H, ustage, mstage, tcount);
      continue;
    }
    __syncthreads();  // the previous tile's shared memory is read
    for (int i = tid; i < S::WARPS * RADIX; i += SEG_BLOCK) (&sm.whist[0][0])[i] = 0;
    for (int i = tid; i < S::WARPS * (RADIX + 1); i += SEG_BLOCK) (&sm.match[0][0])[i] = 0;
    seg_setup<K>(sm, kin, bound, tile, lb);
    const uint64_t s = sm.bound[0];
    const uint32_t cnt = (uint32_t)(sm.bound[1] - s);
    const K base = sm.base;
    uint32_t rank[ITEMS];
    if (cnt > 0) {
      const int passes = (int)sm.passes;
      const int ipw = (int)((cnt + SEG_BLOCK - 1) / SEG_BLOCK);
      const uint32_t wofs = (uint32_t)warp * 32u * ipw;
      K key[ITEMS];
      uint32_t none[ITEMS];
#pragma unroll
      for (int i = 0; i < ITEMS; i++) {
        const uint32_t j = wofs + i * 32 + lane;
        key[i] = (i < ipw && j < cnt) ? KeyOps<K>::sub(kin[s + j], base) : KeyOps<K>::zero();
      }
      for (int p = 0; p < passes; p++) {
        if (p > 0) {
          reload_items<K, false, ITEMS>(sm, key, none, ipw, wofs, cnt);
          __syncthreads();
        }
        rank_items<K, ITEMS, RANK>(sm, key, rank, ipw, wofs, cnt, p * RADIX_BITS);
        digit_positions(sm);
        scatter_items<K, false, ITEMS>(sm, key, none, rank, ipw);
      }
    }
    __syncthreads();
    // distinct keys: the first key of each run; a run's length is the
    // distance to the next run's first key
    bool head[ITEMS];
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
      const uint32_t j = (uint32_t)i * SEG_BLOCK + tid;
      head[i] = j < cnt && (j == 0 || !KeyOps<K>::eq(sm.keys[j], sm.keys[j - 1]));
    }
    const uint32_t count = tile_flag_ranks<SEG_BLOCK, ITEMS>(head, rank, sm.cnt);
#pragma unroll
    for (int i = 0; i < ITEMS; i++)
      if (head[i]) sm.hpos[rank[i]] = (uint32_t)i * SEG_BLOCK + tid;
    if (tid == 0) sm.hpos[count] = cnt;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
      if (head[i]) {
        const uint32_t j = (uint32_t)i * SEG_BLOCK + tid;
        ustage[s + rank[i]] = KeyOps<K>::add(sm.keys[j], base);
        mstage[s + rank[i]] = sm.hpos[rank[i] + 1] - j;
      }
    }
    if (tid == 0) tcount[tile] = count;
  }
}

// Edge keys, counted before they are sorted.  A tile of the local pass
// holds every copy of each of its keys, and at read coverage c a tile of n
// keys holds about n / c distinct ones, so k_seg_count counts the copies
// first, in a shared-memory hash table of TBL slots (linear probing; a slot
// is claimed by compare-and-swap and counted by atomic add), packs the
// occupied slots to the front of the table in slot order, and then orders
// only the distinct keys.  The output is that of k_seg_rle: each distinct
// key once, in order, with its multiplicity (STEP-2), staged in the tile's
// own range.  The table is small so that several CTAs share an SM; a tile
// whose keys do not fit (a probe longer than PROBES slots), or would not, is
// listed in over_list and ordered copy by copy instead (k_rank_rle, or
// k_seg_rle without rank_groups).
//
// Ordering the distinct keys.  With rank_groups set, the distinct keys are
// bucketed by the top 11 bits of their offset from the tile's base (2048
// buckets for a few hundred to 1500 keys, so that most hold one or none),
// and each key goes to its bucket's start plus the number of the bucket's
// keys below it; a tile with a bucket of more than COUNT_GROUP_MAX distinct
// keys is radix-sorted by the 8-bit passes instead (and counted in rank_fb).
// (Packing a 64-bit key's offset and its count into one slot word, counted
// by 64-bit shared atomic adds, measured 1.9x slower: the hot slots of a
// 30x-covered key serialise.)
constexpr uint32_t COUNT_GROUP_MAX = 256;

// Of the first 256 keys of a tile of n with c copies each, about
// 1 - 128 c / n are the first of their key: 96 % (64-bit keys, n = 4096) or
// 92 % (128-bit, n = 2048) at c = 1.3, 50 % and 25 % at c = 30, and 40 to 60 %
// where half a percent of errors adds its own keys.  At 1.3 copies of 28.5 M
// 128-bit keys every tile passes 65 %, and the edge list's local pass takes
// 0.89 ms; at 80 % 12143 of 13923 do, 0.98; at 90 % 6448, 1.27; without the
// sample, sorting the 6465 tiles that overflow by digits, 2.17.  At 30 copies
// the sample itself costs 1 % (1.035 G keys: 7.87 -> 7.97 ms).
constexpr int COUNT_FRESH_PCT = 65;

// Hash-table slots of the counting pass.  The empty mark is the all-ones
// key, which no key offset reaches: an offset is key - base <= key, and the
// all-ones key (T repeated) is never canonical, its reverse complement (A
// repeated) being smaller.
template <class K>
struct SlotOps;

// claim(p, d) returns the slot's key, having stored d there if it was empty
// (then it returns empty): the caller has found d's slot when it gets empty
// or d, and probes on otherwise.
template <>
struct SlotOps<uint64_t> {
  __device__ static uint64_t empty() { return ~0ull; }
  // Fibonacci hashing: the high 32 bits of d times 2^64 / golden ratio
  __device__ static uint32_t hash(uint64_t d) { return (uint32_t)((d * 0x9e3779b97f4a7c15ull) >> 32); }
  __device__ static uint64_t claim(uint64_t *p, uint64_t d) {
    // a 64-bit load is single-copy atomic, so it settles most probes
    // without an atomic operation
    const uint64_t cur = *reinterpret_cast<const volatile uint64_t *>(p);
    if (cur != ~0ull) return cur;
    return atomicCAS(reinterpret_cast<unsigned long long *>(p), ~0ull, d);
  }
};

template <>
struct SlotOps<Key128> {
  __device__ static Key128 empty() { return Key128{~0ull, ~0ull}; }
  __device__ static uint32_t hash(Key128 d) {
    return (uint32_t)(((d.lo ^ (d.hi * 0x9e3779b97f4a7c15ull)) * 0xc2b2ae3d27d4eb4full) >> 32);
  }
  // every probe is a 128-bit compare-and-swap, which also reads the slot
  // whole (two 64-bit loads could see a slot half written; trusting halves
  // that are not empty's and swapping only otherwise was slower, 2.4 instead of
  // 1.0 ms for 9 M keys nearly all distinct and no gain at 30x coverage)
  __device__ static Key128 claim(Key128 *p, Key128 d) {
    Key128 old;
    asm volatile(
        "{\n .reg .b128 c, n, o;\n mov.b128 c, {%2, %3};\n mov.b128 n, {%4, %5};\n"
        " atom.shared.cas.b128 o, [%6], c, n;\n mov.b128 {%0, %1}, o;\n}"
        : "=l"(old.hi), "=l"(old.lo)
        : "l"(~0ull), "l"(~0ull), "l"(d.hi), "l"(d.lo), "r"(smem_u32(p))
        : "memory");
    return old;
  }
};

template <class K, int RANK>
struct SegCountSmem {
  static constexpr int WARPS = SEG_BLOCK / 32;
  static constexpr int TBL = 2048;                // hash slots
  static constexpr int TBITS = 11;                // log2(TBL)
  static constexpr int ITEMS = TBL / SEG_BLOCK;   // distinct keys per thread in the sort
  static constexpr int LOAD = 8;                  // keys per thread per load batch
  static constexpr uint32_t PROBES = 64;          // longest probe before the tile overflows
  static_assert((1 << TBITS) == TBL, "table size");
  K keys[TBL];         // hash slots; then the distinct keys, packed and sorted
  uint32_t vals[TBL];  // copies per slot; then per distinct key
  uint16_t perm[TBL];  // distinct keys bucketed by group
  uint32_t gst[TBL];   // distinct keys per group, then where each group ends
  uint32_t whist[WARPS][RADIX];
  uint32_t match[RANK == RANK_ATOMIC ? WARPS : 1][RADIX + 1];
  uint32_t cnt[ITEMS * WARPS + 1];
  uint32_t tmp[8];
  uint64_t bound[2];
  K base, range;
  uint32_t tile, passes, excl, total, span_bits, overflow, fresh, maxg;
};

// high bits of a key offset, as a bucket index within the tile
template <class K>
__device__ __forceinline__ uint32_t group_of(K d, int bshift) {
  return (uint32_t)KeyOps<K>::words_lo(KeyOps<K>::shr(d, bshift));
}

template <class K, int RANK>
__global__ __launch_bounds__(SEG_BLOCK, 4) void k_seg_count(
    const K *__restrict__ kin, const uint64_t *__restrict__ bound, const uint32_t *__restrict__ osize,
    K *__restrict__ ustage, uint32_t *__restrict__ mstage, uint32_t *__restrict__ tcount,
    uint32_t *__restrict__ over_list, uint32_t *__restrict__ over_count, LowBits lb, int rank_groups, uint32_t *__restrict__ rank_fb) {
  using S = SegCountSmem<K, RANK>;
  using O = SlotOps<K>;
  constexpr int ITEMS = S::ITEMS;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  S &sm = *reinterpret_cast<S *>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t tile = blockIdx.x;
  if (osize[tile]) {  // (later: k_seg_rle, from the gathered keys)
    if (tid == 0) tcount[tile] = 0;
    return;
  }
  for (int j = tid; j < S::TBL; j += SEG_BLOCK) {
    sm.keys[j] = O::empty();
    sm.vals[j] = 0;
  }
  if (tid == 0) sm.overflow = sm.fresh = 0;
  seg_setup<K>(sm, kin, bound, tile, lb);  // synchronises
  const uint64_t s = sm.bound[0];
  const uint32_t cnt = (uint32_t)(sm.bound[1] - s);
  const K base = sm.base;
  // the tile's path (uniform): ranked by buckets of groups
  const bool by_groups = rank_groups && cnt > 0;
  const int bshift = (int)sm.span_bits > S::TBITS ? (int)sm.span_bits - S::TBITS : 0;
  // count: each key into its slot, LOAD keys per thread at a time.  A tile
  // that could fill more than half the table and whose first keys are nearly
  // all distinct (see COUNT_FRESH_PCT) is listed at once.
  bool sample = rank_groups && cnt > S::TBL / 2;
  for (uint32_t j0 = 0; j0 < cnt; j0 += S::LOAD * SEG_BLOCK) {
    K d[S::LOAD];
#pragma unroll
    for (int i = 0; i < S::LOAD; i++) {
      const uint32_t j = j0 + (uint32_t)i * SEG_BLOCK + tid;
      d[i] = j < cnt ? KeyOps<K>::sub(kin[s + j], base) : O::empty();
    }
    // (not in the first batch: another warp may set the flag between two lanes'
    // reads of it, and the sample below counts with all lanes of the warp)
    if (j0 > 0 && *reinterpret_cast<volatile uint32_t *>(&sm.overflow)) break;
#pragma unroll
    for (int i = 0; i < S::LOAD; i++) {
      // (128-bit tiles are one batch long; in 64-bit ones, of two, a test here
      // costs every tile 8 %)
      if (sizeof(K) == 16 && i == 2 && *reinterpret_cast<volatile uint32_t *>(&sm.overflow)) break;
      uint32_t fresh = 0;
      if (!KeyOps<K>::eq(d[i], O::empty())) {
        uint32_t h = O::hash(d[i]) >> (32 - S::TBITS);
        bool done = false;
        for (uint32_t probe = 0; probe < S::PROBES; probe++) {
          const K cur = O::claim(&sm.keys[h], d[i]);
          if (KeyOps<K>::eq(cur, O::empty()) || KeyOps<K>::eq(cur, d[i])) {
            atomicAdd(&sm.vals[h], 1u);
            if (i == 0) fresh = KeyOps<K>::eq(cur, d[i]) ? 0 : 1;
            done = true;
            break;
          }
          h = (h + 1) & (S::TBL - 1);
        }
        if (!done) sm.overflow = 1;
      }
      if (i == 0 && sample) {
        const uint32_t f = __popc(__ballot_sync(0xffffffffu, fresh));
        if (lane == 0 && atomicAdd(&sm.fresh, f) + f > SEG_BLOCK * COUNT_FRESH_PCT / 100) sm.overflow = 1;
        sample = false;
      }
    }
  }
  __syncthreads();
  if (sm.overflow) {
    if (tid == 0) {
      over_list[atomicAdd(over_count, 1u)] = tile;
      tcount[tile] = 0;
    }
    return;
  }
  // pack the occupied slots to the front in slot order: a slot moves to its
  // rank among the occupied slots (at most its own index) once every slot
  // has been read
  uint32_t D;
  {
    K pk[ITEMS];
    uint32_t pc[ITEMS], pr[ITEMS];
    bool occ[ITEMS];
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
      const uint32_t j = (uint32_t)i * SEG_BLOCK + tid;
      pk[i] = sm.keys[j];
      pc[i] = sm.vals[j];
      occ[i] = !KeyOps<K>::eq(pk[i], O::empty());
    }
    D = tile_flag_ranks<SEG_BLOCK, ITEMS>(occ, pr, sm.cnt);
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
      if (occ[i]) {
        sm.keys[pr[i]] = pk[i];
        sm.vals[pr[i]] = pc[i];
      }
    }
  }
  __syncthreads();
  bool ranked = false;
  if (by_groups && D > 0) {
    // bucket the distinct keys: counts, exclusive scan (ITEMS consecutive
    // buckets per thread), then placement
    const uint32_t G = cnt > 0 ? group_of<K>(sm.range, bshift) + 1u : 0u;
    for (uint32_t o = tid; o < G; o += SEG_BLOCK) sm.gst[o] = 0;
    if (tid == 0) sm.maxg = 0;
    __syncthreads();
    for (uint32_t r = tid; r < D; r += SEG_BLOCK) atomicAdd(&sm.gst[group_of<K>(sm.keys[r], bshift)], 1u);
    __syncthreads();
    uint32_t gc[ITEMS], sum = 0, mx = 0;
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
      const uint32_t o = (uint32_t)tid * ITEMS + i;
      gc[i] = o < G ? sm.gst[o] : 0u;
      sum += gc[i];
      mx = max(mx, gc[i]);
    }
    uint32_t run = block_excl_scan_256(sum, sm.tmp);
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
      const uint32_t o = (uint32_t)tid * ITEMS + i;
      if (o < G) sm.gst[o] = run;
      run += gc[i];
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0 && mx) atomicMax(&sm.maxg, mx);
    __syncthreads();
    if (sm.maxg <= COUNT_GROUP_MAX) {
      for (uint32_t r = tid; r < D; r += SEG_BLOCK)
        sm.perm[atomicAdd(&sm.gst[group_of<K>(sm.keys[r], bshift)], 1u)] = (uint16_t)r;
      __syncthreads();
      // bucket o now spans [gst[o - 1], gst[o]) (from 0 for o = 0)
      for (uint32_t q = tid; q < D; q += SEG_BLOCK) {
        const uint32_t r = sm.perm[q], o = group_of<K>(sm.keys[r], bshift);
        const uint32_t a = o ? sm.gst[o - 1] : 0u, b = sm.gst[o];
        const K x = sm.keys[r];
        uint32_t below = 0;
        for (uint32_t t = a; t < b; t++) below += KeyOps<K>::less(sm.keys[sm.perm[t]], x) ? 1u : 0u;
        ustage[s + a + below] = KeyOps<K>::add(x, base);
        mstage[s + a + below] = sm.vals[r];
      }
      ranked = true;
    }
  }
  if (!ranked && D > 0) {
    if (rank_groups && tid == 0) atomicAdd(rank_fb, 1u);
    // sort the D distinct keys (with their counts) by their offset bits
    for (int i = tid; i < S::WARPS * RADIX; i += SEG_BLOCK) (&sm.whist[0][0])[i] = 0;
    if (RANK == RANK_ATOMIC)
      for (int i = tid; i < S::WARPS * (RADIX + 1); i += SEG_BLOCK) (&sm.match[0][0])[i] = 0;
    __syncthreads();
    const int passes = (int)sm.passes;
    const int ipw = (int)((D + SEG_BLOCK - 1) / SEG_BLOCK);
    const uint32_t wofs = (uint32_t)warp * 32u * ipw;
    K key[ITEMS];
    uint32_t val[ITEMS], rank[ITEMS];
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
      const uint32_t j = wofs + i * 32 + lane;
      const bool in = i < ipw && j < D;
      key[i] = in ? sm.keys[j] : KeyOps<K>::zero();
      val[i] = in ? sm.vals[j] : 0u;
    }
    for (int p = 0; p < passes; p++) {
      if (p > 0) {
        reload_items<K, true, ITEMS>(sm, key, val, ipw, wofs, D);
        __syncthreads();
      }
      rank_items<K, ITEMS, RANK>(sm, key, rank, ipw, wofs, D, p * RADIX_BITS);
      digit_positions(sm);
      scatter_items<K, true, ITEMS>(sm, key, val, rank, ipw);
    }
    __syncthreads();
    for (uint32_t r = tid; r < D; r += SEG_BLOCK) {
      ustage[s + r] = KeyOps<K>::add(sm.keys[r], base);
      mstage[s + r] = sm.vals[r];
    }
  }
  if (tid == 0) tcount[tile] = D;
}

// Moves every tile's distinct keys from its staging range to the dense
// edge list (toff = exclusive scan of tcount).
template <class K>
__global__ void k_seg_compact(const uint64_t *__restrict__ bound, const uint32_t *__restrict__ tcount,
                              const uint64_t *__restrict__ toff, uint64_t tiles, const K *__restrict__ ustage,
                              const uint32_t *__restrict__ mstage, K *__restrict__ uniq, uint32_t *__restrict__ mult) {
  for (uint64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const uint64_t s = bound[t], o = toff[t];
    const uint32_t c = tcount[t];
    for (uint32_t r = threadIdx.x; r < c; r += blockDim.x) {
      uniq[o + r] = ustage[s + r];
      mult[o + r] = mstage[s + r];
    }
  }
}

// The multiplicities alone.
static __global__ void k_mult_compact(const uint64_t *__restrict__ bound, const uint32_t *__restrict__ tcount,
                                      const uint64_t *__restrict__ toff, uint64_t tiles,
                                      const uint32_t *__restrict__ mstage, uint32_t *__restrict__ mult) {
  for (uint64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const uint64_t s = bound[t], o = toff[t];
    for (uint32_t r = threadIdx.x; r < tcount[t]; r += blockDim.x) mult[o + r] = mstage[s + r];
  }
}

// Edge keys of a tile with few copies each: every copy is ranked, as the
// records are by k_seg_rank, by a counting sort over buckets of the top bits
// of the key offsets and comparisons within the bucket; then the runs of equal
// keys are counted.  Bound by instruction issue: 0.27 ms for 6448 tiles of 2048
// 128-bit keys, where k_seg_rle's digit passes take 0.89.
// A grid of CTAs takes the *list_count tiles of `list` in turn (two of 512
// threads per SM); a tile with a bucket longer than RANK_GROUP_MAX goes to
// fb_list, for k_seg_rle.
template <class K>
struct RankRleSmem {
  static constexpr int CAP = SegRankSmem<K>::CAP, ITEMS = SegRankSmem<K>::ITEMS;
  static constexpr int TBITS = SegRankSmem<K>::TBITS, NB = 1 << TBITS, PER = NB / 2 / RANK_BLOCK;
  static_assert(NB > CAP, "the run starts take the buckets' place");
  K key[CAP];                   // offsets from base
  uint32_t start2[NB / 2 + 1];  // 16 bits per bucket: its keys, then its first position; then where each run starts
  uint32_t wsum[RANK_BLOCK / 32];
  uint32_t cnt[ITEMS * (RANK_BLOCK / 32) + 1], head[ITEMS * (RANK_BLOCK / 32)];
  uint64_t bound[2];
  K base, range;
  uint32_t passes, span_bits, maxg, distinct;
};

template <class K>
__global__ __launch_bounds__(RANK_BLOCK, 2) void k_rank_rle(
    const K *__restrict__ kin, const uint64_t *__restrict__ bound, K *__restrict__ ustage,
    uint32_t *__restrict__ mstage, uint32_t *__restrict__ tcount, LowBits lb, const uint32_t *__restrict__ list,
    const uint32_t *__restrict__ list_count, uint32_t *__restrict__ fb_list, uint32_t *__restrict__ fb_count) {
  using S = RankRleSmem<K>;
  constexpr int ITEMS = S::ITEMS, PER = S::PER;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  S &sm = *reinterpret_cast<S *>(smem_raw);
  uint16_t *const start = reinterpret_cast<uint16_t *>(sm.start2);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t todo = *list_count;
  for (uint32_t next = blockIdx.x; next < todo; next += gridDim.x) {
    const uint32_t tile = list[next];
    __syncthreads();  // the previous tile's shared memory is read
    for (int j = tid; j <= S::NB / 2; j += RANK_BLOCK) sm.start2[j] = 0;
    if (tid == 0) sm.maxg = 0;
    seg_setup<K>(sm, kin, bound, tile, lb);  // synchronises
    const uint64_t s = sm.bound[0];
    const uint32_t cnt = (uint32_t)(sm.bound[1] - s);
    const int items = (int)((cnt + RANK_BLOCK - 1) / RANK_BLOCK);  // of each thread
    const K base = sm.base;
    const int bshift = (int)sm.span_bits > S::TBITS ? (int)sm.span_bits - S::TBITS : 0;
    K key[ITEMS];
    uint32_t oa[ITEMS];  // bucket, place on arrival << 13; then place
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
      if (i >= items) break;
      const uint32_t j = (uint32_t)i * RANK_BLOCK + tid;
      if (j < cnt) key[i] = KeyOps<K>::sub(kin[s + j], base);
    }
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
      if (i >= items) break;
      if ((uint32_t)i * RANK_BLOCK + tid < cnt) {
        const uint32_t o = group_of<K>(key[i], bshift), h = 16 * (o & 1u);
        oa[i] = o | ((atomicAdd(&sm.start2[o >> 1], 1u << h) >> h) & 0xffffu) << S::TBITS;
      }
    }
    __syncthreads();
    // exclusive scan, 2 PER consecutive buckets per thread
    uint32_t c[PER], sum = 0, mx = 0;
#pragma unroll
    for (int j = 0; j < PER; j++) {
      c[j] = sm.start2[tid * PER + j];
      const uint32_t c0 = c[j] & 0xffffu, c1 = c[j] >> 16;
      sum += c0 + c1;
      mx = max(mx, max(c0, c1));
    }
    const uint32_t incl = warp_incl_scan(sum);
    if (lane == 31) sm.wsum[warp] = incl;
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0 && mx > RANK_GROUP_MAX) sm.maxg = mx;
    __syncthreads();
    if (sm.maxg) {  // (tcount is 0 from the listing)
      if (tid == 0) fb_list[atomicAdd(fb_count, 1u)] = tile;
      continue;
    }
    uint32_t run = incl - sum;
    for (int w = 0; w < warp; w++) run += sm.wsum[w];
#pragma unroll
    for (int j = 0; j < PER; j++) {
      const uint32_t c0 = c[j] & 0xffffu, c1 = c[j] >> 16;
      sm.start2[tid * PER + j] = run | (run + c0) << 16;
      run += c0 + c1;
    }
    if (tid == RANK_BLOCK - 1) sm.start2[S::NB / 2] = run;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
      if (i >= items) break;
      if ((uint32_t)i * RANK_BLOCK + tid < cnt) {
        oa[i] = start[oa[i] & (S::NB - 1)] + (oa[i] >> S::TBITS);
        sm.key[oa[i]] = key[i];
      }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
      if (i >= items) break;
      if ((uint32_t)i * RANK_BLOCK + tid < cnt) {
        // place: the bucket's smaller keys, and its equal ones before this
        const uint32_t q = oa[i], o = group_of<K>(key[i], bshift), a = start[o], b = start[o + 1];
        uint32_t r = a;
#pragma unroll 1
        for (uint32_t t = a; t < q; t++) r += KeyOps<K>::less(key[i], sm.key[t]) ? 0u : 1u;
#pragma unroll 1
        for (uint32_t t = q + 1; t < b; t++) r += KeyOps<K>::less(sm.key[t], key[i]) ? 1u : 0u;
        oa[i] = r;
      }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
      if (i >= items) break;
      if ((uint32_t)i * RANK_BLOCK + tid < cnt) sm.key[oa[i]] = key[i];
    }
    __syncthreads();
    // the runs' first positions, in the buckets' place
    for (int i = 0; i < items; i++) {
      const uint32_t j = (uint32_t)i * RANK_BLOCK + tid;
      const unsigned hb = __ballot_sync(0xffffffffu, j < cnt && (j == 0 || !KeyOps<K>::eq(sm.key[j], sm.key[j - 1])));
      if (lane == 0) {
        sm.head[i * (RANK_BLOCK / 32) + warp] = hb;
        sm.cnt[i * (RANK_BLOCK / 32) + warp] = __popc(hb);
      }
    }
    __syncthreads();
    if (warp == 0) {
      constexpr int NW = ITEMS * (RANK_BLOCK / 32), EACH = (NW + 31) / 32;
      const int nw = items * (RANK_BLOCK / 32);
      uint32_t x[EACH], sum = 0;
#pragma unroll
      for (int j = 0; j < EACH; j++) {
        x[j] = lane * EACH + j < nw ? sm.cnt[lane * EACH + j] : 0u;
        sum += x[j];
      }
      const uint32_t incl = warp_incl_scan(sum);
      uint32_t run = incl - sum;
#pragma unroll
      for (int j = 0; j < EACH; j++) {
        if (lane * EACH + j < nw) sm.cnt[lane * EACH + j] = run;
        run += x[j];
      }
      if (lane == 31) {
        sm.distinct = incl;
        start[incl] = (uint16_t)cnt;
        tcount[tile] = incl;
      }
    }
    __syncthreads();
    for (int i = 0; i < items; i++) {
      const int w = i * (RANK_BLOCK / 32) + warp;
      if (sm.head[w] >> lane & 1u)
        start[sm.cnt[w] + __popc(sm.head[w] & ((1u << lane) - 1u))] = (uint16_t)(i * RANK_BLOCK + tid);
    }
    __syncthreads();
    for (uint32_t r = tid; r < sm.distinct; r += RANK_BLOCK) {
      ustage[s + r] = KeyOps<K>::add(sm.key[start[r]], base);
      mstage[s + r] = (uint32_t)start[r + 1] - start[r];
    }
  }
}

}  // namespace dbg
