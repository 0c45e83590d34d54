// k_msd.cuh -- the global half of the hybrid sort (K3 / STEP-2, STEP-3), most
// significant digit first: at most two partition passes put the keys into
// groups -- the keys that share their high bits -- in ascending order of
// those bits, and the local pass (k_segsort.cuh) finishes runs of whole
// groups in shared memory.
//
// Why this way round.  A least-significant-first sort has to keep the order
// of equal digits in every pass but its first, so each tile waits for the
// tiles before it (look-back) and ranks its keys in order.  Most significant
// first, a pass only has to bring keys to their bucket: a tile ranks its keys
// by shared-memory atomic adds and reserves its part of every bucket with one
// global atomic add per digit.  No order, no wait, and a digit of up to 12
// bits where the ordered pass takes 8, so two passes give the groups that
// took three.  What is lost -- the order of equal keys -- the local pass
// restores where it matters, by comparing payloads too.
//
//   plan    W = 2^w1 buckets by the top w1 bits, counted by the producer of
//           the keys.  A bucket of m keys gets w2 = ceil(log2(m / mean)) more
//           bits (at most two more than the average bucket), so that groups
//           hold about `mean` keys where the keys lie evenly within buckets
//           (canonical keys are twice as dense at the low end as on average).
//           One pass is enough when W groups are.
//   pass 1  k_msd_part over the keys as they come.
//   count   k_msd_count: the sizes of each bucket's 2^w2 groups; their scan
//           gives every group's place.
//   pass 2  k_msd_part again, tile by tile of each bucket.
//   split   only when the local pass met many keys in groups too long for it
//           (an uneven base composition: at 20 % GC a group of AT-rich
//           prefixes holds ten times the mean): k_msd_split lists those
//           groups, and they alone are counted and partitioned once more by
//           as many bits as each takes.  Groups of copies of one key are left
//           out: no digit divides them.
#pragma once

#include "k_build.cuh"

namespace dbg {

constexpr int MSD_MAX_BITS = 12;  // of one digit
constexpr size_t MSD_PAD = 32;    // bytes behind the end of arrays that bulk copies read (see k_msd_part)

// Tile shapes of a partition pass.  The run of a digit in a tile is what a
// CTA writes in one piece, and the digits are what it scans and reserves, so
// digits of 10 bits and up want the largest tile that shared memory holds
// twice (one CTA per SM); below that, two CTAs per SM overlap one's ranking
// with the other's write-out.  Per 2^27 64-bit keys: 8 bits 0.471 ms (512 x
// 12) and 0.499 (768 x 16), 10 bits 0.587 and 0.571, 11 bits 0.763 and 0.637,
// 12 bits 1.394 (one CTA of it fits) and 0.794.
template <class K, bool HAS_VAL, bool WIDE> struct MsdShape {
  static constexpr int BLOCK = WIDE ? 768 : 512, MINB = WIDE ? 1 : 2;
  static constexpr int ITEMS = sizeof(K) == 8 ? (HAS_VAL ? (WIDE ? 11 : 8) : (WIDE ? 16 : 12))
                                              : (HAS_VAL ? (WIDE ? 6 : 4) : (WIDE ? 8 : 6));
  static constexpr uint32_t TILE = BLOCK * ITEMS;
};

// The buckets of pass 1 and, for two passes, their groups and tiles; or the
// groups that are split, in no order, as the buckets of that pass.
struct MsdTables {
  uint64_t *start;         // [W + 1] first key of each bucket
  uint64_t *end;           // [W] its end (start + 1, unless groups are split)
  uint32_t *gfirst;        // [W + 1] first group of each bucket
  uint32_t *tfirst;        // [W + 1] first tile of each bucket
  uint32_t *ntiles;        // the tiles' number
  uint8_t *w2;             // [W] bits of the bucket's second digit
  uint8_t *low;            // [W] bits below the bucket's groups
  uint32_t *tmap;          // [tiles] bucket of each tile
};

// One block.  Bucket starts from the producer's histogram; with two passes
// also each bucket's second digit, groups and tiles.
static __global__ __launch_bounds__(1024) void k_msd_plan(const unsigned long long *__restrict__ hist, int w1,
                                                          int shift1, int two, uint32_t mean, int max_w2,
                                                          uint32_t tile, MsdTables tb,
                                                          uint32_t *__restrict__ cursor) {
  __shared__ uint64_t s_sum[32];
  __shared__ uint32_t s_g[32], s_t[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t W = 1u << w1;
  const uint32_t per = (W + 1023) / 1024;  // consecutive buckets of this thread (at most 4)
  const uint32_t b0 = (uint32_t)tid * per;
  uint64_t sum = 0;
  uint32_t groups = 0, tiles = 0;
  for (uint32_t j = 0; j < per && b0 + j < W; j++) {
    const uint64_t c = hist[b0 + j];
    sum += c;
    if (two) {
      int w = 0;
      while (w < max_w2 && ((uint64_t)mean << w) < c) w++;
      tb.w2[b0 + j] = (uint8_t)w;
      tb.low[b0 + j] = (uint8_t)(shift1 - w);
      groups += 1u << w;
      tiles += (uint32_t)((c + tile - 1) / tile);
    }
  }
  uint64_t is = warp_incl_scan(sum);
  uint32_t ig = warp_incl_scan(groups), it = warp_incl_scan(tiles);
  if (lane == 31) {
    s_sum[warp] = is;
    s_g[warp] = ig;
    s_t[warp] = it;
  }
  __syncthreads();
  if (warp == 0) {
    const uint64_t a = s_sum[lane], ai = warp_incl_scan(a);
    const uint32_t g = s_g[lane], gi = warp_incl_scan(g);
    const uint32_t t = s_t[lane], ti = warp_incl_scan(t);
    s_sum[lane] = ai - a;
    s_g[lane] = gi - g;
    s_t[lane] = ti - t;
  }
  __syncthreads();
  uint64_t at = s_sum[warp] + is - sum;
  uint32_t g = s_g[warp] + ig - groups, t = s_t[warp] + it - tiles;
  for (uint32_t j = 0; j < per && b0 + j < W; j++) {
    const uint32_t b = b0 + j;
    const uint64_t c = hist[b];
    tb.start[b] = at;
    cursor[b] = (uint32_t)at;
    at += c;
    if (two) {
      tb.gfirst[b] = g;
      tb.tfirst[b] = t;
      g += 1u << tb.w2[b];
      const uint32_t nt = (uint32_t)((c + tile - 1) / tile);
      for (uint32_t q = 0; q < nt; q++) tb.tmap[t + q] = b;
      t += nt;
    }
    if (b == W - 1) {
      tb.start[W] = at;
      if (two) {
        tb.gfirst[W] = g;
        tb.tfirst[W] = t;
      }
    }
  }
}

// Sizes of the groups of pass 1's buckets.  Each CTA takes consecutive tiles,
// so its shared-memory counters go to global memory only when the bucket
// changes (every 60 to 120 tiles for a thousand-key group size).  A read of
// every key and one shared-memory atomic add per key: HBM-bound.
constexpr int MSD_BLOCK = 512;

template <class K>
__global__ __launch_bounds__(MSD_BLOCK) void k_msd_count(const K *__restrict__ keys, uint32_t TILE, MsdTables tb,
                                                         uint32_t *__restrict__ gcount) {
  constexpr int ITEMS = 8;
  extern __shared__ uint32_t s_h[];
  const int tid = threadIdx.x;
  const uint32_t NT = *tb.ntiles;
  const uint32_t per = (NT + gridDim.x - 1) / gridDim.x;
  const uint32_t t0 = min(NT, blockIdx.x * per), t1 = min(NT, t0 + per);
  uint32_t cur = 0xffffffffu, ways = 0;
  int low = 0;
  auto flush = [&]() {
    __syncthreads();
    for (uint32_t i = tid; i < ways; i += MSD_BLOCK)
      if (s_h[i]) atomicAdd(gcount + tb.gfirst[cur] + i, s_h[i]);
    __syncthreads();
  };
  for (uint32_t t = t0; t < t1; t++) {
    const uint32_t b = tb.tmap[t];
    if (b != cur) {
      if (cur != 0xffffffffu) flush();
      cur = b;
      ways = 1u << tb.w2[b];
      low = tb.low[b];
      for (uint32_t i = tid; i < ways; i += MSD_BLOCK) s_h[i] = 0;
      __syncthreads();
    }
    const uint64_t base = tb.start[b] + (uint64_t)(t - tb.tfirst[b]) * TILE;
    const uint64_t end = min(base + TILE, tb.end[b]);
    for (uint64_t p = base + tid; p < end; p += (uint64_t)MSD_BLOCK * ITEMS) {
      K k[ITEMS];
#pragma unroll
      for (int i = 0; i < ITEMS; i++) {
        const uint64_t q = p + (uint64_t)i * MSD_BLOCK;
        k[i] = q < end ? keys[q] : KeyOps<K>::zero();
      }
#pragma unroll
      for (int i = 0; i < ITEMS; i++)
        if (p + (uint64_t)i * MSD_BLOCK < end)
          atomicAdd(&s_h[(uint32_t)KeyOps<K>::words_lo(KeyOps<K>::shr(k[i], low)) & (ways - 1)], 1u);
    }
  }
  if (cur != 0xffffffffu) flush();
}

// One partition pass, persistent CTAs.  Pass 1 (`two` false): tile t is keys
// [t TILE, ...), the digit the `bits` bits from `shift` up.  Pass 2: tile t
// is part of bucket tmap[t], the digit that bucket's.  cursor[d] (pass 2:
// [gfirst + d]) is the next free place of digit d.
//
// A tile arrives by bulk copies while the one before it is ranked and
// written; its keys are ranked by shared-memory atomic adds, staged in digit
// order in their own buffer, and written out run by run.  The tile's parts of
// the digits' runs are reserved (neighbouring lanes, neighbouring digits:
// whole sectors of cursors) while the keys are staged.  A bulk copy starts on
// a 16-byte boundary at or before the tile's first key and may read up to 15
// bytes past its last, so the arrays carry MSD_PAD bytes behind their end.
template <class K, bool HAS_VAL, int BLOCK, int ITEMS>
struct MsdSmem {
  static constexpr uint32_t TILE = BLOCK * ITEMS;
  static constexpr uint32_t KA = sizeof(K) >= 16 ? 1 : 16 / sizeof(K), VA = 4;  // elements in 16 bytes
  static constexpr uint32_t KSLOTS = TILE + KA, VSLOTS = HAS_VAL ? TILE + 2 * VA : 0;
  static_assert(KSLOTS * sizeof(K) % 16 == 0 && VSLOTS % 4 == 0, "buffers stay 16-byte aligned");
  static constexpr size_t BUF = (size_t)KSLOTS * sizeof(K) + (size_t)VSLOTS * 4;
  static constexpr size_t bytes(int ways) { return 2 * BUF + (size_t)ways * 8 + 16; }
};

template <class K, bool HAS_VAL, int BLOCK, int ITEMS, int MINB>
__global__ __launch_bounds__(BLOCK, MINB) void k_msd_part(const K *__restrict__ kin, K *__restrict__ kout,
                                                          const uint32_t *__restrict__ vin,
                                                          uint32_t *__restrict__ vout, uint64_t n, int shift,
                                                          int bits, MsdTables tb, int two,
                                                          uint32_t *__restrict__ cursor, uint32_t max_ways,
                                                          uint32_t spin_limit, uint32_t *__restrict__ err) {
  using S = MsdSmem<K, HAS_VAL, BLOCK, ITEMS>;
  constexpr uint32_t TILE = S::TILE;
  constexpr int WARPS = BLOCK / 32;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  auto kbuf = [&](int b) { return reinterpret_cast<K *>(smem_raw + b * S::BUF); };
  auto vbuf = [&](int b) { return reinterpret_cast<uint32_t *>(smem_raw + b * S::BUF + S::KSLOTS * sizeof(K)); };
  uint32_t *s_delta = reinterpret_cast<uint32_t *>(smem_raw + 2 * S::BUF);  // modulo 2^32: n <= 2^32
  uint32_t *s_off = s_delta + max_ways;                                    // max_ways + 1 entries
  __shared__ uint32_t s_w[WARPS];
  __shared__ uint64_t s_bar[2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t NT = two ? *tb.ntiles : (uint32_t)((n + TILE - 1) / TILE);
  const bool bulk = ((reinterpret_cast<uintptr_t>(kin) | (HAS_VAL ? reinterpret_cast<uintptr_t>(vin) : 0)) & 15) == 0;
  auto base_of = [&](uint32_t t, uint32_t b) {
    return two ? tb.start[b] + (uint64_t)(t - tb.tfirst[b]) * TILE : (uint64_t)t * TILE;
  };
  auto count_of = [&](uint64_t base, uint32_t b) {
    return (uint32_t)min((uint64_t)TILE, (two ? tb.end[b] : n) - base);
  };
  // (one thread) tile t into buffer q
  auto issue = [&](uint32_t t, int q) {
    const uint32_t b = two ? tb.tmap[t] : 0;
    const uint64_t base = base_of(t, b);
    const uint32_t c = count_of(base, b);
    const uint32_t ko = (uint32_t)(base & (S::KA - 1)), vo = (uint32_t)(base & (S::VA - 1));
    const uint32_t kb = (ko + c + S::KA - 1) / S::KA * S::KA * (uint32_t)sizeof(K);
    const uint32_t vb = HAS_VAL ? (vo + c + S::VA - 1) / S::VA * S::VA * 4u : 0u;
    mbar_expect_tx(&s_bar[q], kb + vb);
    tma_load_bulk(kbuf(q), kin + (base - ko), kb, &s_bar[q]);
    if (HAS_VAL) tma_load_bulk(vbuf(q), vin + (base - vo), vb, &s_bar[q]);
  };
  auto digit_of = [](const K &k, int sh, uint32_t mask) {
    return (uint32_t)KeyOps<K>::words_lo(KeyOps<K>::shr(k, sh)) & mask;
  };
  if (tid == 0) {
    mbar_init(&s_bar[0], 1);
    mbar_init(&s_bar[1], 1);
    mbar_init_fence();
  }
  __syncthreads();
  uint32_t t = blockIdx.x;
  if (tid == 0 && bulk && t < NT) issue(t, 0);
  uint32_t phase = 0;  // bit q: parity of buffer q's next completion
  for (int it = 0; t < NT; t += gridDim.x, it++) {
    const int q = it & 1;
    const uint32_t tn = t + gridDim.x;
    if (tid == 0 && bulk && tn < NT) issue(tn, q ^ 1);
    const uint32_t b = two ? tb.tmap[t] : 0;
    const uint64_t base = base_of(t, b);
    const uint32_t count = count_of(base, b);
    const uint32_t ways = 1u << (two ? (int)tb.w2[b] : bits), mask = ways - 1;
    const int sh = two ? (int)tb.low[b] : shift;
    uint32_t *cur = cursor + (two ? tb.gfirst[b] : 0u);
    for (uint32_t i = tid; i < ways; i += BLOCK) s_off[i] = 0;
    if (bulk) {
      const bool ok = __syncthreads_and(mbar_wait(&s_bar[q], (phase >> q) & 1u, spin_limit));
      phase ^= 1u << q;
      if (!ok) {
        // give up on this launch; first let the copies in flight land
        if (tid == 0) atomicOr(err, ERR_TIMEOUT);
        mbar_wait(&s_bar[q], ((phase >> q) & 1u) ^ 1u, spin_limit);
        if (tn < NT) mbar_wait(&s_bar[q ^ 1], (phase >> (q ^ 1)) & 1u, spin_limit);
        return;
      }
    } else {
      __syncthreads();
    }
    K *const sk = kbuf(q);
    uint32_t *const sv = vbuf(q);
    const uint32_t ko = (uint32_t)(base & (S::KA - 1)), vo = (uint32_t)(base & (S::VA - 1));
    K key[ITEMS];
    uint32_t val[HAS_VAL ? ITEMS : 1];
    uint32_t rank[ITEMS];
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
      const uint32_t j = (uint32_t)i * BLOCK + tid;
      if (j < count) {
        key[i] = bulk ? sk[ko + j] : kin[base + j];
        if (HAS_VAL) val[i] = bulk ? sv[vo + j] : vin[base + j];
        rank[i] = atomicAdd(&s_off[digit_of(key[i], sh, mask)], 1u);
      }
    }
    __syncthreads();
    // the digits' places in the staged tile: `per` consecutive digits per thread
    const uint32_t per = (ways + BLOCK - 1) / BLOCK, d0 = (uint32_t)tid * per;
    uint32_t sum = 0;
    for (uint32_t j = 0; j < per; j++) sum += d0 + j < ways ? s_off[d0 + j] : 0u;
    const uint32_t incl = warp_incl_scan(sum);
    if (lane == 31) s_w[warp] = incl;
    __syncthreads();
    uint32_t run = incl - sum;
    for (int w = 0; w < warp; w++) run += s_w[w];
    for (uint32_t j = 0; j < per; j++)
      if (d0 + j < ways) {
        const uint32_t c = s_off[d0 + j];
        s_off[d0 + j] = run;
        run += c;
      }
    if (tid == 0) s_off[ways] = count;
    __syncthreads();
    // reserve the runs (the answers are needed only after the staging)
    constexpr int PER = 4096 / BLOCK > 4 ? 4 : 4096 / BLOCK;
    uint32_t g[PER];
#pragma unroll
    for (int j = 0; j < PER; j++) {
      const uint32_t d = (uint32_t)j * BLOCK + tid;
      if (d < ways) {
        const uint32_t o = s_off[d], c = s_off[d + 1] - o;
        g[j] = c ? atomicAdd(cur + d, c) - o : 0u;
      }
    }
#pragma unroll
    for (int i = 0; i < ITEMS; i++)
      if ((uint32_t)i * BLOCK + tid < count) {
        const uint32_t p = s_off[digit_of(key[i], sh, mask)] + rank[i];
        sk[p] = key[i];
        if (HAS_VAL) sv[p] = val[i];
      }
#pragma unroll
    for (int j = 0; j < PER; j++) {
      const uint32_t d = (uint32_t)j * BLOCK + tid;
      if (d < ways) s_delta[d] = g[j];
    }
    for (uint32_t d = (uint32_t)PER * BLOCK + tid; d < ways; d += BLOCK) {
      const uint32_t o = s_off[d], c = s_off[d + 1] - o;
      if (c) s_delta[d] = atomicAdd(cur + d, c) - o;
    }
    __syncthreads();
#pragma unroll 4
    for (uint32_t p = tid; p < count; p += BLOCK) {
      const K k = sk[p];
      const uint32_t dst = s_delta[digit_of(k, sh, mask)] + p;
      if (dst < n) {
        kout[dst] = k;
        if (HAS_VAL) vout[dst] = sv[p];
      } else {  // only reachable if the digit counts were inconsistent
        atomicOr(err, ERR_INTERNAL);
      }
    }
    // this buffer's next use is a bulk copy (async proxy) after these
    // generic-proxy accesses
    fence_proxy_async_smem();
    __syncthreads();
  }
}

// bound[t] = the first key of the group that holds key t * tile_keys, from
// the groups' places (goff[g] .. goff[g + 1]); bound[tiles] = n.  cursor[g],
// if given, = goff[g].  Groups that split (their bits, or 0) says to be split
// are left to k_split_bounds.
__device__ __forceinline__ void tile_bounds(uint64_t s, uint64_t e, uint64_t tile_keys, uint64_t *bound) {
  for (uint64_t t = (s + tile_keys - 1) / tile_keys; t * tile_keys < e; t++) bound[t] = s;  // (empty: no tile)
}

static __global__ void k_msd_bounds(const uint64_t *__restrict__ goff, const uint32_t *__restrict__ groups_of,
                                    uint32_t groups, uint64_t n, uint64_t tile_keys, uint64_t tiles,
                                    uint64_t *__restrict__ bound, uint32_t *__restrict__ cursor,
                                    const uint8_t *__restrict__ split) {
  const uint32_t NG = groups_of ? *groups_of : groups;
  for (uint32_t g = blockIdx.x * blockDim.x + threadIdx.x; g < NG; g += gridDim.x * blockDim.x) {
    const uint64_t s = goff[g], e = goff[g + 1];
    if (cursor) cursor[g] = (uint32_t)s;
    if (!split || !split[g]) tile_bounds(s, e, tile_keys, bound);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) bound[tiles] = n;
}

// ---------------------------------------------------------------------------
// Splitting long groups.  made[0 .. 3]: groups listed, their parts, their
// tiles, their keys.
// ---------------------------------------------------------------------------
constexpr int MSD_SPLIT_BITS = 11;

// Lists the groups of more than `longest` keys as buckets of tb, each with as
// many bits as bring its parts to `mean` keys; groups of copies of one key are
// left out.
template <class K>
__global__ void k_msd_split(const K *__restrict__ keys, const uint64_t *__restrict__ goff,
                            const uint32_t *__restrict__ groups_of, uint32_t groups, LowBits lb, uint32_t longest,
                            uint32_t mean, uint32_t tile, MsdTables tb, uint8_t *__restrict__ split,
                            uint32_t *__restrict__ made) {
  const uint32_t NG = groups_of ? *groups_of : groups;
  for (uint32_t g = blockIdx.x * blockDim.x + threadIdx.x; g < NG; g += gridDim.x * blockDim.x) {
    const uint64_t s = goff[g], e = goff[g + 1], c = e - s;
    if (c <= longest) continue;
    const int low = lb.unsplit(keys[s]);
    if (low == 0 || copies_of_one(keys, s, c)) continue;
    int w = 0;
    while (w < min(MSD_SPLIT_BITS, low) && ((uint64_t)mean << w) < c) w++;
    const uint32_t nt = (uint32_t)((c + tile - 1) / tile);
    const uint32_t b = atomicAdd(made, 1u), part = atomicAdd(made + 1, 1u << w), t = atomicAdd(made + 2, nt);
    atomicAdd(made + 3, (uint32_t)c);
    split[g] = (uint8_t)w;
    tb.start[b] = s;
    tb.end[b] = e;
    tb.gfirst[b] = part;
    tb.tfirst[b] = t;
    tb.w2[b] = (uint8_t)w;
    tb.low[b] = (uint8_t)(low - w);
    for (uint32_t q = 0; q < nt; q++) tb.tmap[t + q] = b;
  }
}

// From the scan of the parts' sizes (poff): where each part lies, as the
// partition's cursors, and the tiles' bounds.
static __global__ void k_split_bounds(MsdTables tb, uint32_t listed, const uint64_t *__restrict__ poff,
                                      uint64_t tile_keys, uint64_t *__restrict__ bound,
                                      uint32_t *__restrict__ cursor) {
  for (uint32_t b = blockIdx.x; b < listed; b += gridDim.x) {
    const uint32_t p0 = tb.gfirst[b], parts = 1u << tb.w2[b];
    const uint64_t at = tb.start[b] - poff[p0];  // (modulo 2^64)
    for (uint32_t j = p0 + threadIdx.x; j < p0 + parts; j += blockDim.x) {
      const uint64_t s = at + poff[j], e = at + poff[j + 1];
      cursor[j] = (uint32_t)s;
      tile_bounds(s, e, tile_keys, bound);
    }
  }
}

// The listed groups' keys (and payloads) back from the partition's output.
template <class K, bool HAS_VAL>
__global__ void k_split_back(MsdTables tb, uint32_t tile, const K *__restrict__ kin, K *__restrict__ kout,
                             const uint32_t *__restrict__ vin, uint32_t *__restrict__ vout) {
  const uint32_t NT = *tb.ntiles;
  for (uint32_t t = blockIdx.x; t < NT; t += gridDim.x) {
    const uint32_t b = tb.tmap[t];
    const uint64_t base = tb.start[b] + (uint64_t)(t - tb.tfirst[b]) * tile;
    const uint32_t c = (uint32_t)min((uint64_t)tile, tb.end[b] - base);
    for (uint32_t j = threadIdx.x; j < c; j += blockDim.x) {
      kout[base + j] = kin[base + j];
      if (HAS_VAL) vout[base + j] = vin[base + j];
    }
  }
}

}  // namespace dbg
