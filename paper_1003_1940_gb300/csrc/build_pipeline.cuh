// build_pipeline.cuh -- host side of dbg_build for one key width: plans the
// buffers, launches STEP-1..4 on the context's stream, and fills the graph.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "k_build.cuh"
#include "k_msd.cuh"
#include "k_segsort.cuh"

namespace dbg {

inline int passes_for_bits(int bits) { return (bits + RADIX_BITS - 1) / RADIX_BITS; }

// items per thread of the build's run-length reduce and node-ID scans
constexpr int BUILD_SCAN_ITEMS = 8;
constexpr int BUILD_SCAN_TILE = SCAN_BLOCK * BUILD_SCAN_ITEMS;

// ---------------------------------------------------------------------------
// Radix sort variants.  Every compiled onesweep configuration of a key kind
// sorts identically; they differ in tile shape, load path and ranking
// method.  The context keeps one choice per kind (default, set by the
// caller, or picked by dbg_autotune).
// ---------------------------------------------------------------------------
using SortLaunchFn = void (*)(dbg_ctx *ctx, const void *kin, void *kout, const uint32_t *vin, uint32_t *vout,
                              uint64_t n, int shift, const uint64_t *digit_base, uint32_t epoch);

struct SortVariant {
  const char *name;
  int tile;
  SortLaunchFn launch;
};

template <class K, bool V, int BLOCK, int ITEMS, int RANK, bool TMA, int MINB, bool EARLY, bool DIRECT = false,
          int LB = 1>
void launch_onesweep(dbg_ctx *ctx, const void *kin, void *kout, const uint32_t *vin, uint32_t *vout, uint64_t n,
                     int shift, const uint64_t *digit_base, uint32_t epoch) {
  auto kern = k_onesweep<K, V, BLOCK, ITEMS, RANK, TMA, MINB, EARLY, DIRECT, LB>;
  constexpr size_t smem = sizeof(OnesweepSmem<K, V, BLOCK, ITEMS>);
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
  const uint64_t tiles = (n + BLOCK * ITEMS - 1) / (BLOCK * ITEMS);
  kern<<<(unsigned)tiles, BLOCK, smem, ctx->stream>>>(static_cast<const K *>(kin), static_cast<K *>(kout), vin,
                                                      vout, n, shift, digit_base, ctx->d_status, ctx->d_counters,
                                                      epoch, ctx->spin_limit, ctx->d_err);
}

template <class K, bool V, int BLOCK, int ITEMS, int RANK, int MINB, int LB, int HB = 4, bool BULK = false>
void launch_onesweep_p(dbg_ctx *ctx, const void *kin, void *kout, const uint32_t *vin, uint32_t *vout, uint64_t n,
                       int shift, const uint64_t *digit_base, uint32_t epoch) {
  auto kern = k_onesweep_p<K, V, BLOCK, ITEMS, RANK, MINB, LB, HB, BULK>;
  constexpr size_t smem = sizeof(OnesweepPSmem<K, V, BLOCK, ITEMS, RANK, HB, BULK>);
  static_assert(smem <= 227 * 1024, "onesweep variant exceeds the shared memory of a CTA");
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
  const uint64_t tiles = (n + BLOCK * ITEMS - 1) / (BLOCK * ITEMS);
  const unsigned grid = (unsigned)std::min<uint64_t>(tiles, (uint64_t)MINB * (uint64_t)ctx->num_sms);
  kern<<<grid, BLOCK, smem, ctx->stream>>>(static_cast<const K *>(kin), static_cast<K *>(kout), vin, vout, n, shift,
                                           digit_base, ctx->d_status, ctx->d_counters, epoch, ctx->spin_limit,
                                           ctx->d_err);
}

#define DBG_SVP(K, V, B, I, R, M, L, NAME) \
  SortVariant { NAME, (B) * (I), &launch_onesweep_p<K, V, B, I, R, M, L> }
#define DBG_SVH(K, V, B, I, R, M, L, NAME) \
  SortVariant { NAME, (B) * (I), &launch_onesweep_p<K, V, B, I, R, M, L, 2> }
#define DBG_SVB(K, V, B, I, R, M, L, NAME) \
  SortVariant { NAME, (B) * (I), &launch_onesweep_p<K, V, B, I, R, M, L, 2, true> }
#define DBG_SV(K, V, B, I, R, T, M, NAME) \
  SortVariant { NAME, (B) * (I), &launch_onesweep<K, V, B, I, R, T, M, false> }
#define DBG_SVE(K, V, B, I, R, T, M, NAME) \
  SortVariant { NAME, (B) * (I), &launch_onesweep<K, V, B, I, R, T, M, true> }
#define DBG_SVL(K, V, B, I, R, T, M, E, L, NAME) \
  SortVariant { NAME, (B) * (I), &launch_onesweep<K, V, B, I, R, T, M, E, false, L> }
#define DBG_SVD(K, V, B, I, R, T, M, E, NAME) \
  SortVariant { NAME, (B) * (I), &launch_onesweep<K, V, B, I, R, T, M, E, true> }

// kinds: 0 = 64-bit keys, 1 = 64-bit keys + payload, 2 = 128-bit keys,
// 3 = 128-bit keys + payload
template <class K, bool V> struct SortKind;
template <> struct SortKind<uint64_t, false> {
  static constexpr int kind = 0;
  static const SortVariant *table(int *count) {
    static const SortVariant t[] = {
        DBG_SV(uint64_t, false, 256, 16, RANK_BALLOT, false, 1, "256x16 ballot ldg"),
        DBG_SV(uint64_t, false, 256, 16, RANK_MATCH, false, 1, "256x16 match ldg"),
        DBG_SV(uint64_t, false, 256, 16, RANK_MATCH, true, 1, "256x16 match tma"),
        DBG_SV(uint64_t, false, 256, 12, RANK_MATCH, true, 3, "256x12 match tma occ3"),
        DBG_SV(uint64_t, false, 256, 12, RANK_ATOMIC, true, 3, "256x12 atomic tma occ3"),
        DBG_SV(uint64_t, false, 256, 8, RANK_MATCH, true, 4, "256x8 match tma occ4"),
        DBG_SV(uint64_t, false, 512, 8, RANK_MATCH, true, 2, "512x8 match tma occ2"),
        DBG_SVE(uint64_t, false, 256, 12, RANK_ATOMIC, true, 3, "256x12 atomic tma occ3 early"),
        DBG_SVE(uint64_t, false, 256, 12, RANK_MATCH, true, 3, "256x12 match tma occ3 early"),
        DBG_SVE(uint64_t, false, 256, 8, RANK_ATOMIC, true, 4, "256x8 atomic tma occ4 early"),
        DBG_SVE(uint64_t, false, 256, 16, RANK_ATOMIC, true, 2, "256x16 atomic tma occ2 early"),
        DBG_SV(uint64_t, false, 256, 8, RANK_ATOMIC, true, 4, "256x8 atomic tma occ4"),
        DBG_SV(uint64_t, false, 256, 10, RANK_ATOMIC, true, 3, "256x10 atomic tma occ3"),
        DBG_SV(uint64_t, false, 384, 8, RANK_ATOMIC, true, 2, "384x8 atomic tma occ2"),
        DBG_SV(uint64_t, false, 512, 6, RANK_ATOMIC, true, 2, "512x6 atomic tma occ2"),
        DBG_SVD(uint64_t, false, 256, 12, RANK_ATOMIC, true, 3, false, "256x12 atomic tma occ3 direct"),
        DBG_SVD(uint64_t, false, 256, 12, RANK_ATOMIC, false, 3, false, "256x12 atomic ldg occ3 direct"),
        DBG_SVD(uint64_t, false, 256, 16, RANK_ATOMIC, false, 2, false, "256x16 atomic ldg occ2 direct"),
        DBG_SVD(uint64_t, false, 256, 12, RANK_ATOMIC, true, 3, true, "256x12 atomic tma occ3 early direct"),
        DBG_SVL(uint64_t, false, 256, 12, RANK_ATOMIC, true, 3, false, 4, "256x12 atomic tma occ3 lb4"),
        DBG_SVL(uint64_t, false, 256, 12, RANK_ATOMIC, true, 3, true, 4, "256x12 atomic tma occ3 early lb4"),
        DBG_SVL(uint64_t, false, 256, 12, RANK_ATOMIC, true, 3, true, 8, "256x12 atomic tma occ3 early lb8"),
        DBG_SVL(uint64_t, false, 256, 16, RANK_ATOMIC, true, 2, true, 8, "256x16 atomic tma occ2 early lb8"),
        DBG_SVL(uint64_t, false, 256, 12, RANK_ATOMIC, true, 3, false, 8, "256x12 atomic tma occ3 lb8"),
        DBG_SVL(uint64_t, false, 256, 12, RANK_ATOMIC, true, 3, false, 16, "256x12 atomic tma occ3 lb16"),
        DBG_SVL(uint64_t, false, 256, 16, RANK_ATOMIC, true, 2, false, 4, "256x16 atomic tma occ2 lb4"),
        DBG_SVL(uint64_t, false, 256, 8, RANK_ATOMIC, true, 4, false, 4, "256x8 atomic tma occ4 lb4"),
        DBG_SVL(uint64_t, false, 256, 10, RANK_ATOMIC, true, 3, false, 8, "256x10 atomic tma occ3 lb8"),
        DBG_SVP(uint64_t, false, 256, 12, RANK_ATOMIC, 3, 4, "256x12 atomic persistent occ3 lb4"),
        DBG_SVP(uint64_t, false, 256, 12, RANK_ATOMIC, 3, 8, "256x12 atomic persistent occ3 lb8"),
        DBG_SVP(uint64_t, false, 256, 8, RANK_ATOMIC, 4, 4, "256x8 atomic persistent occ4 lb4"),
        DBG_SVP(uint64_t, false, 256, 12, RANK_MATCH, 3, 4, "256x12 match persistent occ3 lb4"),
        DBG_SVP(uint64_t, false, 256, 16, RANK_ATOMIC, 2, 4, "256x16 atomic persistent occ2 lb4"),
        DBG_SVP(uint64_t, false, 512, 8, RANK_ATOMIC, 2, 4, "512x8 atomic persistent occ2 lb4"),
        DBG_SVP(uint64_t, false, 1024, 8, RANK_ATOMIC, 1, 4, "1024x8 atomic persistent occ1 lb4"),
        DBG_SVP(uint64_t, false, 1024, 8, RANK_ATOMIC, 1, 8, "1024x8 atomic persistent occ1 lb8"),
        DBG_SVP(uint64_t, false, 768, 8, RANK_ATOMIC, 1, 4, "768x8 atomic persistent occ1 lb4"),
        DBG_SVP(uint64_t, false, 1024, 10, RANK_ATOMIC, 1, 8, "1024x10 atomic persistent occ1 lb8"),
        DBG_SVP(uint64_t, false, 1024, 9, RANK_ATOMIC, 1, 8, "1024x9 atomic persistent occ1 lb8"),
        DBG_SVH(uint64_t, false, 1024, 10, RANK_ATOMIC, 1, 8, "1024x10 atomic persistent occ1 lb8 h16"),
        DBG_SVH(uint64_t, false, 1024, 11, RANK_ATOMIC, 1, 8, "1024x11 atomic persistent occ1 lb8 h16"),
        DBG_SVH(uint64_t, false, 1024, 12, RANK_MATCH, 1, 8, "1024x12 match persistent occ1 lb8 h16"),
        DBG_SVB(uint64_t, false, 1024, 10, RANK_ATOMIC, 1, 8, "1024x10 atomic persistent occ1 lb8 h16 bulk"),
        DBG_SVB(uint64_t, false, 1024, 11, RANK_MATCH, 1, 8, "1024x11 match persistent occ1 lb8 h16 bulk"),
        DBG_SVB(uint64_t, false, 1024, 12, RANK_MATCH, 1, 8, "1024x12 match persistent occ1 lb8 h16 bulk"),
    };
    *count = sizeof(t) / sizeof(t[0]);
    return t;
  }
};
template <> struct SortKind<uint64_t, true> {
  static constexpr int kind = 1;
  static const SortVariant *table(int *count) {
    static const SortVariant t[] = {
        DBG_SV(uint64_t, true, 256, 12, RANK_BALLOT, false, 1, "256x12 ballot ldg"),
        DBG_SV(uint64_t, true, 256, 12, RANK_MATCH, true, 1, "256x12 match tma"),
        DBG_SV(uint64_t, true, 256, 8, RANK_MATCH, true, 3, "256x8 match tma occ3"),
        DBG_SV(uint64_t, true, 256, 8, RANK_ATOMIC, true, 3, "256x8 atomic tma occ3"),
        DBG_SVE(uint64_t, true, 256, 8, RANK_ATOMIC, true, 3, "256x8 atomic tma occ3 early"),
        DBG_SVE(uint64_t, true, 256, 12, RANK_ATOMIC, true, 2, "256x12 atomic tma occ2 early"),
        DBG_SV(uint64_t, true, 256, 10, RANK_ATOMIC, true, 3, "256x10 atomic tma occ3"),
        DBG_SV(uint64_t, true, 384, 8, RANK_ATOMIC, true, 2, "384x8 atomic tma occ2"),
        DBG_SVD(uint64_t, true, 256, 10, RANK_ATOMIC, true, 3, false, "256x10 atomic tma occ3 direct"),
        DBG_SVD(uint64_t, true, 256, 8, RANK_ATOMIC, false, 3, false, "256x8 atomic ldg occ3 direct"),
        DBG_SVL(uint64_t, true, 256, 10, RANK_ATOMIC, true, 3, true, 4, "256x10 atomic tma occ3 early lb4"),
        DBG_SVL(uint64_t, true, 256, 10, RANK_ATOMIC, true, 3, false, 4, "256x10 atomic tma occ3 lb4"),
        DBG_SVL(uint64_t, true, 256, 10, RANK_ATOMIC, true, 3, false, 8, "256x10 atomic tma occ3 lb8"),
        DBG_SVL(uint64_t, true, 256, 8, RANK_ATOMIC, true, 3, false, 8, "256x8 atomic tma occ3 lb8"),
        DBG_SVP(uint64_t, true, 256, 8, RANK_ATOMIC, 3, 4, "256x8 atomic persistent occ3 lb4"),
        DBG_SVP(uint64_t, true, 256, 10, RANK_ATOMIC, 2, 4, "256x10 atomic persistent occ2 lb4"),
        DBG_SVP(uint64_t, true, 256, 6, RANK_ATOMIC, 4, 4, "256x6 atomic persistent occ4 lb4"),
        DBG_SVP(uint64_t, true, 1024, 6, RANK_ATOMIC, 1, 4, "1024x6 atomic persistent occ1 lb4"),
        DBG_SVP(uint64_t, true, 1024, 6, RANK_ATOMIC, 1, 8, "1024x6 atomic persistent occ1 lb8"),
        DBG_SVH(uint64_t, true, 1024, 7, RANK_ATOMIC, 1, 8, "1024x7 atomic persistent occ1 lb8 h16"),
        DBG_SVB(uint64_t, true, 1024, 6, RANK_ATOMIC, 1, 8, "1024x6 atomic persistent occ1 lb8 h16 bulk"),
        DBG_SVB(uint64_t, true, 1024, 7, RANK_MATCH, 1, 8, "1024x7 match persistent occ1 lb8 h16 bulk"),
    };
    *count = sizeof(t) / sizeof(t[0]);
    return t;
  }
};
template <> struct SortKind<Key128, false> {
  static constexpr int kind = 2;
  static const SortVariant *table(int *count) {
    static const SortVariant t[] = {
        DBG_SV(Key128, false, 256, 8, RANK_BALLOT, false, 1, "256x8 ballot ldg"),
        DBG_SV(Key128, false, 256, 8, RANK_MATCH, true, 1, "256x8 match tma"),
        DBG_SV(Key128, false, 256, 6, RANK_MATCH, true, 3, "256x6 match tma occ3"),
        DBG_SVE(Key128, false, 256, 6, RANK_ATOMIC, true, 3, "256x6 atomic tma occ3 early"),
        DBG_SVE(Key128, false, 256, 8, RANK_ATOMIC, true, 2, "256x8 atomic tma occ2 early"),
        DBG_SVD(Key128, false, 256, 8, RANK_ATOMIC, true, 2, true, "256x8 atomic tma occ2 early direct"),
        DBG_SVL(Key128, false, 256, 8, RANK_ATOMIC, true, 2, true, 4, "256x8 atomic tma occ2 early lb4"),
        DBG_SVL(Key128, false, 256, 8, RANK_ATOMIC, true, 2, false, 8, "256x8 atomic tma occ2 lb8"),
        DBG_SVL(Key128, false, 256, 6, RANK_ATOMIC, true, 3, false, 8, "256x6 atomic tma occ3 lb8"),
        DBG_SVP(Key128, false, 256, 6, RANK_ATOMIC, 3, 4, "256x6 atomic persistent occ3 lb4"),
        DBG_SVP(Key128, false, 256, 8, RANK_ATOMIC, 2, 4, "256x8 atomic persistent occ2 lb4"),
        DBG_SVP(Key128, false, 1024, 4, RANK_ATOMIC, 1, 4, "1024x4 atomic persistent occ1 lb4"),
        DBG_SVP(Key128, false, 1024, 5, RANK_ATOMIC, 1, 8, "1024x5 atomic persistent occ1 lb8"),
        DBG_SVH(Key128, false, 1024, 6, RANK_MATCH, 1, 8, "1024x6 match persistent occ1 lb8 h16"),
        DBG_SVB(Key128, false, 1024, 5, RANK_ATOMIC, 1, 8, "1024x5 atomic persistent occ1 lb8 h16 bulk"),
    };
    *count = sizeof(t) / sizeof(t[0]);
    return t;
  }
};
template <> struct SortKind<Key128, true> {
  static constexpr int kind = 3;
  static const SortVariant *table(int *count) {
    static const SortVariant t[] = {
        DBG_SV(Key128, true, 256, 8, RANK_BALLOT, false, 1, "256x8 ballot ldg"),
        DBG_SV(Key128, true, 256, 8, RANK_MATCH, true, 1, "256x8 match tma"),
        DBG_SV(Key128, true, 256, 6, RANK_MATCH, true, 3, "256x6 match tma occ3"),
        DBG_SVE(Key128, true, 256, 6, RANK_ATOMIC, true, 3, "256x6 atomic tma occ3 early"),
        DBG_SVD(Key128, true, 256, 6, RANK_ATOMIC, true, 3, true, "256x6 atomic tma occ3 early direct"),
        DBG_SVL(Key128, true, 256, 6, RANK_ATOMIC, true, 3, true, 4, "256x6 atomic tma occ3 early lb4"),
        DBG_SVL(Key128, true, 256, 6, RANK_ATOMIC, true, 3, false, 8, "256x6 atomic tma occ3 lb8"),
        DBG_SVP(Key128, true, 256, 6, RANK_ATOMIC, 2, 4, "256x6 atomic persistent occ2 lb4"),
        DBG_SVP(Key128, true, 1024, 3, RANK_ATOMIC, 1, 4, "1024x3 atomic persistent occ1 lb4"),
        DBG_SVB(Key128, true, 1024, 3, RANK_ATOMIC, 1, 8, "1024x3 atomic persistent occ1 lb8 h16 bulk"),
    };
    *count = sizeof(t) / sizeof(t[0]);
    return t;
  }
};
#undef DBG_SV
#undef DBG_SVP
#undef DBG_SVH
#undef DBG_SVB
#undef DBG_SVE
#undef DBG_SVD
#undef DBG_SVL

template <class K, bool V>
const SortVariant &chosen_variant(dbg_ctx *ctx) {
  int count = 0;
  const SortVariant *t = SortKind<K, V>::table(&count);
  int v = ctx->sort_variant[SortKind<K, V>::kind];
  if (v < 0 || v >= count) v = 0;
  return t[v];
}

template <class F>
inline void set_smem_attrs(F kern, size_t smem) {
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
}

// Ascending LSD radix sort of n keys (with optional u32 payloads) whose
// significant bits are the low `bits`.  `hist` holds the per-pass digit
// histograms (passes x 256), already accumulated by the producer kernel.
// Passes below first_pass are skipped: the keys are then sorted by their
// bits from 8 * first_pass - adj up (stably; for keys without payload, with
// the partition-first switch on, keys equal in those bits end in no
// particular order).  Pass p takes the 8 bits from 8 p - adj up: adj > 0
// aligns the top pass with the top of a key of 8 P - adj bits, so that the
// passes from first_pass up resolve whole bytes of it.  On return the data is in *keys / *vals (the buffers may have
// been swapped with *alt_keys / *alt_vals).
template <class K, bool HAS_VAL>
dbg_status radix_sort(dbg_ctx *ctx, K **keys, K **alt_keys, uint32_t **vals, uint32_t **alt_vals, uint64_t n,
                      int bits, const unsigned long long *d_hist, uint64_t *d_digit_base, int first_pass = 0,
                      int adj = 0) {
  if (n <= 1) return DBG_OK;
  const SortVariant &sv = chosen_variant<K, HAS_VAL>(ctx);
  const int passes = passes_for_bits(bits);
  const uint64_t tiles = (n + sv.tile - 1) / sv.tile;
  if (tiles > 0x7fffffffull) return DBG_EOVERFLOW;
  DBG_TRY(ensure_status(ctx, (size_t)tiles * RADIX));
  cudaStream_t s = ctx->stream;
  DBG_LAUNCH(ctx, HAS_VAL ? ST_SORT_NODES : ST_SORT_EDGES, 0.0,
             k_digit_base<<<passes, RADIX, 0, s>>>(d_hist, d_digit_base));
  int p = first_pass;
  if (!HAS_VAL && ctx->partition_first && p < passes) {
    // the first pass of keys without payload as a partition (no look-back)
    constexpr int tile = PART_BLOCK * PartShape<K>::ITEMS;
    constexpr size_t smem = sizeof(PartSmem<K>);
    set_smem_attrs(k_partition<K>, smem);
    const uint64_t tiles = (n + tile - 1) / tile;
    const unsigned grid = (unsigned)std::min<uint64_t>(tiles, 3ull * (uint64_t)ctx->num_sms);
    DBG_LAUNCH(ctx, ST_PARTITION_EDGES, 2.0 * (double)n * (double)sizeof(K),
               k_partition<K><<<grid, PART_BLOCK, smem, s>>>(
                   *keys, *alt_keys, n, p * RADIX_BITS - adj,
                   reinterpret_cast<unsigned long long *>(d_digit_base + p * RADIX), ctx->spin_limit, ctx->d_err));
    std::swap(*keys, *alt_keys);
    p++;
  }
  for (; p < passes; p++) {
    uint32_t epoch;
    DBG_TRY(next_epoch(ctx, &epoch));
    DBG_CUDA_TRY(cudaMemsetAsync(ctx->d_counters, 0, sizeof(uint32_t), s));
    DBG_LAUNCH(ctx, HAS_VAL ? ST_SORT_NODES : ST_SORT_EDGES,
               2.0 * (double)n * (double)(sizeof(K) + (HAS_VAL ? sizeof(uint32_t) : 0)),
               sv.launch(ctx, *keys, *alt_keys, HAS_VAL ? *vals : nullptr, HAS_VAL ? *alt_vals : nullptr, n,
                         p * RADIX_BITS - adj, d_digit_base + p * RADIX, epoch));
    std::swap(*keys, *alt_keys);
    if (HAS_VAL) std::swap(*vals, *alt_vals);
  }
  DBG_CUDA_TRY(cudaGetLastError());
  return DBG_OK;
}

// ---------------------------------------------------------------------------
// Hybrid sort: global onesweep passes over the high digits, then one local
// pass (k_seg_sort) that finishes each group-aligned tile in shared memory.
// ---------------------------------------------------------------------------
template <class K> struct SegShape;
template <> struct SegShape<uint64_t> {
  static constexpr int ITEMS = 24, TILE = 4096;  // capacity 6144: groups of up to 2048 keys
  static constexpr double MAX_MEAN = 128.0;
};
template <> struct SegShape<Key128> {
  static constexpr int ITEMS = 12, TILE = 2048;  // capacity 3072: groups of up to 1024 keys
  static constexpr double MAX_MEAN = 64.0;
};

// The first global pass of the hybrid sort of n keys of `bits` bits: the
// largest p >= 2 for which keys sharing their bits from 8p up form groups of
// at most MAX_MEAN keys on average, for keys `density` times as dense as
// uniform ones; 0 = no hybrid.
template <class K>
int hybrid_first_pass(uint64_t n, int bits, double density = 1.0) {
  const int P = passes_for_bits(bits);
  for (int p = P; p >= 2; p--) {
    const int hi = bits - RADIX_BITS * p;
    if (hi <= 0) {
      if (n <= (uint64_t)SegShape<K>::TILE) return p;  // one tile holds every key
      continue;
    }
    if ((double)n * density <= SegShape<K>::MAX_MEAN * std::ldexp(1.0, hi)) return p;
  }
  return 0;
}

// ---------------------------------------------------------------------------
// How a sort of n keys of `bits` bits goes: MSD (k_msd.cuh: up to two
// partition passes, then the local pass), the least-significant-first hybrid
// (first_pass > 0, or one local tile), or every digit globally.
// ---------------------------------------------------------------------------
// Mean group size the MSD passes aim at: a tile of TILE keys stretched to
// group boundaries holds at most SegShape's capacity as long as groups stay
// below TILE / 2, and a bucket's groups hold half to all of the mean.
template <class K> constexpr uint32_t msd_mean() { return SegShape<K>::TILE / 4; }

template <class K>
struct SortPlan {
  bool msd = false;
  uint32_t mean = msd_mean<K>();  // MSD: the groups' size aimed at
  int first_pass = 0, adj = 0;  // least significant first
  int bits = 0;                 // key bits
  int need = 0;                 // MSD: bits that groups of the mean size take,
  int w1 = 0, passes = 0;       // bits of the first digit, passes
  int shift1() const { return bits - w1; }
  DigitSpec digits() const {
    DigitSpec d;
    if (msd) {
      d.first = shift1();
      d.wide = w1;  // 0 (no pass): nothing is counted
    } else {
      d.first = first_pass;
      d.passes = passes_for_bits(bits);
      d.adj = adj;
    }
    return d;
  }
  bool local() const { return msd || first_pass > 0; }
};

// MSD where unordered passes are allowed (the partition switch) and leave
// groups that end above the lowest bits: at most one key value per group in
// four would be needed, so that the copies of one key alone seldom fill a
// group.  Up to 2^10 groups in one pass; above, two digits of equal width
// (the second then varies by bucket).  density > 1, for the offsets of one
// key range: how many times denser than over all values of `bits` bits the keys
// lie where they are.  Their groups are planned at a quarter of the mean: the
// range ends anywhere in its last bucket, whose keys may lie in an eighth of
// it.
template <class K>
SortPlan<K> plan_sort(const dbg_ctx *ctx, uint64_t n, int bits, bool unordered, double density = 1.0) {
  const double dense = (double)n * density;
  SortPlan<K> p;
  if (density > 1.0) p.mean /= 4;
  p.bits = bits;
  if (!ctx->hybrid_sort) return p;
  if (unordered && n <= 0xffffffffull) {
    int need = 0;
    if (n > (uint64_t)SegShape<K>::TILE)
      while (std::ldexp((double)p.mean, need) < dense) need++;
    if (need + (need ? 2 : 0) <= bits && need <= 24) {
      p.msd = true;
      p.passes = need == 0 ? 0 : need <= 10 ? 1 : 2;
      p.need = need;
      p.w1 = p.passes == 2 ? std::min(need / 2, MSD_MAX_BITS - 1) : need;  // (records take one bit less)
      return p;
    }
  }
  p.first_pass = hybrid_first_pass<K>(n, bits, density);
  return p;
}

// ranking method of the local sort, by variant number (kinds 4 and 5)
inline int local_rank_method(dbg_ctx *ctx, bool wide) {
  static const int methods[] = {RANK_MATCH, RANK_ATOMIC, RANK_BALLOT};
  const int v = ctx->sort_variant[wide ? 5 : 4];
  return methods[(v >= 0 && v < 6) ? v % 3 : 0];
}

inline unsigned grid_for(uint64_t n, int per_block) {
  uint64_t g = (n + per_block - 1) / per_block;
  return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(g, 0x7fffffffull));
}

// Exclusive scan of n u32 values into n + 1 u64 (the last is the total, which
// also goes to counter `total`).
inline dbg_status scan_u32_async(dbg_ctx *ctx, const uint32_t *in, uint64_t n, uint64_t *out, int stage,
                                 int total = 1) {
  cudaStream_t s = ctx->stream;
  const uint64_t tiles = (n + SCAN_TILE - 1) / SCAN_TILE;
  DBG_TRY(ensure_status(ctx, tiles));
  uint32_t epoch;
  DBG_TRY(next_epoch(ctx, &epoch));
  DBG_CUDA_TRY(cudaMemsetAsync(ctx->d_counters, 0, 2 * sizeof(uint32_t), s));
  DBG_LAUNCH(ctx, stage, 12.0 * n,
             k_scan_excl<<<(unsigned)tiles, SCAN_BLOCK, 0, s>>>(in, n, out, ctx->d_status, ctx->d_counters, epoch,
                                                                ctx->spin_limit, ctx->d_err, ctx->d_counters + total));
  DBG_CUDA_TRY(cudaGetLastError());
  return DBG_OK;
}
inline dbg_status scan_u32(dbg_ctx *ctx, const uint32_t *in, uint64_t n, uint64_t *out, uint32_t *total, int stage) {
  DBG_TRY(scan_u32_async(ctx, in, n, out, stage));
  return read_small(ctx, ctx->d_counters + 1, sizeof(uint32_t), total);
}

// K4 by reduce-then-scan: unique keys into `uniq`, run heads into headpos
// (E + 1 entries, the last = n); returns E.
template <class K>
dbg_status run_length_reduce(dbg_ctx *ctx, const K *sorted, uint64_t n, K *uniq, uint32_t *headpos, uint64_t *E) {
  cudaStream_t s = ctx->stream;
  const uint64_t tiles = (n + RS_TILE - 1) / RS_TILE;
  DevBuf counts, toff;
  DBG_TRY(alloc_tmp(ctx, counts, tiles * 4));
  DBG_TRY(alloc_tmp(ctx, toff, (tiles + 1) * 8));
  DBG_LAUNCH(ctx, ST_RLE, (double)n * sizeof(K),
             k_count_heads<K><<<(unsigned)tiles, SCAN_BLOCK, 0, s>>>(sorted, nullptr, n, counts.as<uint32_t>(),
                                                                   nullptr));
  uint32_t total = 0;
  DBG_TRY(scan_u32(ctx, counts.as<uint32_t>(), tiles, toff.as<uint64_t>(), &total, ST_RLE));
  DBG_LAUNCH(ctx, ST_RLE, (double)n * sizeof(K) + (double)total * (sizeof(K) + 4),
             k_write_heads<K><<<(unsigned)tiles, SCAN_BLOCK, 0, s>>>(sorted, n, toff.as<uint64_t>(), uniq, headpos));
  DBG_CUDA_TRY(cudaGetLastError());
  *E = total;
  return DBG_OK;
}

// The groups that the global passes left: where each key's low bits start,
// and, after MSD passes, the tables that say where each group lies.
struct Groups {
  LowBits lb;
  DevBuf tables, goff;                  // MSD: bucket tables; the groups' places
  DevBuf bound;                         // the local pass's tile bounds, once known
  DevBuf split;                         // bits by which each group was split since (or none was)
  const uint32_t *ng_dev = nullptr;     // the groups' number (two passes), or
  uint32_t ng = 0;                      // their number (one pass)
  uint32_t ng_max = 0;                  // at most that many (0: no MSD pass)
};

inline const uint64_t *group_places(const Groups &gr) {
  return gr.ng ? gr.tables.as<uint64_t>() : gr.goff.as<uint64_t>();
}

// The local pass's tile bounds from the places of the groups (but those that
// are split), which are copied to `cursor` (if given).
template <class K>
dbg_status msd_bounds(dbg_ctx *ctx, Groups &gr, uint64_t n, uint32_t *cursor, int stage) {
  constexpr uint64_t T = SegShape<K>::TILE;
  const uint64_t tiles = (n + T - 1) / T;
  DBG_TRY(alloc_tmp(ctx, gr.bound, (tiles + 1) * 8));
  const uint64_t *places = group_places(gr);
  DBG_LAUNCH(ctx, stage, 0.0,
             k_msd_bounds<<<std::min(grid_for(gr.ng_max, 256), 152u * 8), 256, 0, ctx->stream>>>(
                 places, gr.ng_dev, gr.ng, n, T, tiles, gr.bound.as<uint64_t>(), cursor, gr.split.as<uint8_t>()));
  return DBG_OK;
}

// One partition pass (k_msd_part) in its shape for digits of up to max_bits.
template <class K, bool HAS_VAL, bool WIDE>
dbg_status launch_msd_part(dbg_ctx *ctx, const K *kin, K *kout, const uint32_t *vin, uint32_t *vout, uint64_t n, int shift,
                     int bits, const MsdTables &tb, bool two, uint32_t *cursor, int max_bits,
                     uint64_t tiles) {
  using Sh = MsdShape<K, HAS_VAL, WIDE>;
  using S = MsdSmem<K, HAS_VAL, Sh::BLOCK, Sh::ITEMS>;
  // the attribute is the kernel's, shared by every context: always the most
  // that any launch of this shape asks for
  constexpr size_t most = S::bytes(1 << (WIDE && !(HAS_VAL && sizeof(K) == 8) ? MSD_MAX_BITS : 11));
  static_assert(Sh::MINB * (most + 1024) <= 228 * 1024, "MINB CTAs per SM");
  auto kern = k_msd_part<K, HAS_VAL, Sh::BLOCK, Sh::ITEMS, Sh::MINB>;
  const size_t smem = S::bytes(1 << max_bits);
  if (smem > most) {
    set_error("partition digit of %d bits", max_bits);
    return DBG_EINTERNAL;
  }
  set_smem_attrs(kern, most);
  const uint64_t slots = (uint64_t)Sh::MINB * (uint64_t)std::max(1, ctx->num_sms);
  kern<<<(unsigned)std::min(tiles, slots), Sh::BLOCK, smem, ctx->stream>>>(
      kin, kout, vin, vout, n, shift, bits, tb, two ? 1 : 0, cursor, 1u << max_bits, ctx->spin_limit, ctx->d_err);
  return DBG_OK;
}

// The MSD passes of plan p over n keys (and payloads) whose first digit the
// producer counted in d_hist.  On return the data is in *keys / *vals.  All
// four arrays have MSD_PAD bytes behind their n entries.
template <class K, bool HAS_VAL>
dbg_status msd_sort(dbg_ctx *ctx, K **keys, K **alt_keys, uint32_t **vals, uint32_t **alt_vals, uint64_t n,
                    const SortPlan<K> &p, const unsigned long long *d_hist, Groups &gr) {
  cudaStream_t s = ctx->stream;
  gr.lb.fixed = p.shift1();
  if (p.passes == 0) return DBG_OK;
  const uint32_t W = 1u << p.w1;
  const bool two = p.passes == 2;
  const bool wide1 = p.w1 >= 10, wide2 = p.need - p.w1 >= 10;
  const uint32_t tile1 = wide1 ? MsdShape<K, HAS_VAL, true>::TILE : MsdShape<K, HAS_VAL, false>::TILE;
  const uint32_t tile2 = wide2 ? MsdShape<K, HAS_VAL, true>::TILE : MsdShape<K, HAS_VAL, false>::TILE;
  const uint64_t tiles1 = (n + tile1 - 1) / tile1;
  const uint64_t tiles2 = n / tile2 + W;  // at most: every bucket's last tile may be partial
  if (std::max(tiles1, tiles2) > 0x7fffffffull) return DBG_EOVERFLOW;
  const int stage = HAS_VAL ? ST_SORT_NODES : ST_SORT_EDGES;
  // the second digit of a bucket four times the average size, if it fits
  const int max_w2 = std::min({HAS_VAL ? 11 : MSD_MAX_BITS, p.shift1(), p.need - p.w1 + 2});
  // every bucket has at most max(1, 2 n_b / mean) groups
  gr.ng_max = two ? (uint32_t)(2 * (n / p.mean) + W) : W;
  // [start: W + 1] u64, [cursor: W][gfirst: W + 1][tfirst: W + 1] u32, [tmap] u32, [w2][low] u8
  const size_t bytes = (size_t)(W + 1) * 8 + (size_t)(3 * W + 2) * 4 + (two ? tiles2 * 4 : 0) + 2 * (size_t)W + 16;
  DBG_TRY(alloc_tmp(ctx, gr.tables, bytes));
  MsdTables tb{};
  tb.start = gr.tables.as<uint64_t>();
  tb.end = tb.start + 1;
  uint32_t *cursor = reinterpret_cast<uint32_t *>(tb.start + W + 1);
  tb.gfirst = cursor + W;
  tb.tfirst = tb.gfirst + W + 1;
  tb.ntiles = tb.tfirst + W;
  tb.tmap = tb.tfirst + W + 1;
  tb.w2 = reinterpret_cast<uint8_t *>(tb.tmap + (two ? tiles2 : 0));
  tb.low = tb.w2 + W;
  DBG_LAUNCH(ctx, stage, 0.0,
             k_msd_plan<<<1, 1024, 0, s>>>(d_hist, p.w1, p.shift1(), two ? 1 : 0, p.mean, max_w2, tile2, tb,
                                           cursor));
  const double bytes_pass = 2.0 * (double)n * (double)(sizeof(K) + (HAS_VAL ? 4 : 0));
  auto swap = [&]() {
    std::swap(*keys, *alt_keys);
    if (HAS_VAL) std::swap(*vals, *alt_vals);
  };
  const uint32_t *vi = HAS_VAL ? *vals : nullptr;
  uint32_t *vt = HAS_VAL ? *alt_vals : nullptr;
  DBG_LAUNCH(ctx, HAS_VAL ? ST_SORT_NODES : ST_PARTITION_EDGES, bytes_pass,
             DBG_TRY((wide1 ? launch_msd_part<K, HAS_VAL, true>(ctx, *keys, *alt_keys, vi, vt, n, p.shift1(), p.w1,
                                                                tb, false, cursor, p.w1, tiles1)
                            : launch_msd_part<K, HAS_VAL, false>(ctx, *keys, *alt_keys, vi, vt, n, p.shift1(), p.w1,
                                                                 tb, false, cursor, p.w1, tiles1))));
  swap();
  if (!two) {
    gr.ng = W;
    DBG_CUDA_TRY(cudaGetLastError());
    return DBG_OK;
  }
  // the groups' sizes, their places, and the second pass
  DevBuf gcount;
  const uint64_t NG = gr.ng_max;
  DBG_TRY(alloc_tmp(ctx, gcount, NG * 4));
  DBG_TRY(alloc_tmp(ctx, gr.goff, (NG + 1) * 8));
  DBG_CUDA_TRY(cudaMemsetAsync(gcount.p, 0, NG * 4, s));
  DBG_LAUNCH(ctx, stage, (double)n * sizeof(K),
             k_msd_count<K><<<(unsigned)std::min<uint64_t>(tiles2, 4ull * std::max(1, ctx->num_sms)), MSD_BLOCK,
                              (size_t)4 << max_w2, s>>>(*keys, tile2, tb, gcount.as<uint32_t>()));
  DBG_TRY(scan_u32_async(ctx, gcount.as<uint32_t>(), NG, gr.goff.as<uint64_t>(), stage));
  gr.lb.low = tb.low;
  gr.lb.shift1 = p.shift1();
  gr.lb.gfirst = tb.gfirst;
  gr.ng_dev = tb.gfirst + W;
  // the counts' memory now takes the second pass's cursors (the places stay)
  DBG_TRY(msd_bounds<K>(ctx, gr, n, gcount.as<uint32_t>(), stage));
  vi = HAS_VAL ? *vals : nullptr;
  vt = HAS_VAL ? *alt_vals : nullptr;
  DBG_LAUNCH(ctx, stage, bytes_pass,
             DBG_TRY((wide2 ? launch_msd_part<K, HAS_VAL, true>(ctx, *keys, *alt_keys, vi, vt, n, 0, 0, tb, true,
                                                                gcount.as<uint32_t>(), max_w2, tiles2)
                            : launch_msd_part<K, HAS_VAL, false>(ctx, *keys, *alt_keys, vi, vt, n, 0, 0, tb, true,
                                                                 gcount.as<uint32_t>(), max_w2, tiles2))));
  swap();
  DBG_CUDA_TRY(cudaGetLastError());
  return DBG_OK;
}

// Whether the keys in oversize tiles (counters c) are worth a split of the long
// groups.  Gathering them costs some 30 launches and ten passes over them; a
// split, 13 launches and the local pass over all keys once more.  So few keys
// are worth it where launches count, and one in 24 beyond (builds at 31 bases,
// all gathered against split: 0.64 M instances at 33 % GC 0.69 ms and 0.47, at
// 20 % 0.78 and 0.48; 27.6 M at 33 %, where one key in 40 is in such tiles,
// 2.03 and 2.17, at 20 %, one in 3, 4.08 and 2.28; 276 M 15.9 and 16.7, and
// 37.7 and 17.3).
inline bool worth_split(const uint32_t *c, uint64_t n) {
  return c[CT_MIXED] > n / (n <= 1u << 22 ? 256 : 24) && c[CT_MIXED] >= c[CT_GATHERED] / 4;
}

// Splits the groups that are too long for the local pass, in place: they are
// partitioned by their next bits into alt_keys / alt_vals and copied back.
// On return, if *done, gr describes the parts; otherwise (no MSD passes, few
// keys in oversize tiles, or most of those copies of one key) nothing has
// changed.  Waits for the stream; the tiles' counts are in the counters.
template <class K, bool HAS_VAL>
dbg_status msd_split(dbg_ctx *ctx, K *keys, K *alt_keys, uint32_t *vals, uint32_t *alt_vals, uint64_t n, Groups &gr,
                     int stage, bool *done) {
  using Sh = MsdShape<K, HAS_VAL, false>;
  cudaStream_t s = ctx->stream;
  *done = false;
  if (gr.ng_max == 0 || gr.split.p) return DBG_OK;
  constexpr uint32_t longest = SegShape<K>::TILE / 2, mean = SegShape<K>::TILE / 16;
  const uint64_t L = n / longest + 1, tiles = n / Sh::TILE + L;
  if (tiles > 0x7fffffffull) return DBG_OK;
  DevBuf tables, split;
  DBG_TRY(alloc_tmp(ctx, split, gr.ng_max));
  DBG_TRY(alloc_tmp(ctx, tables, L * (8 + 8 + 4 + 4 + 1 + 1) + tiles * 4));
  MsdTables tb{};
  tb.start = tables.as<uint64_t>();
  tb.end = tb.start + L;
  tb.gfirst = reinterpret_cast<uint32_t *>(tb.end + L);
  tb.tfirst = tb.gfirst + L;
  tb.tmap = tb.tfirst + L;
  tb.w2 = reinterpret_cast<uint8_t *>(tb.tmap + tiles);
  tb.low = tb.w2 + L;
  uint32_t *made = ctx->d_counters + CT_SPLIT;
  tb.ntiles = made + 2;
  DBG_CUDA_TRY(cudaMemsetAsync(split.p, 0, gr.ng_max, s));
  DBG_CUDA_TRY(cudaMemsetAsync(made, 0, 4 * sizeof(uint32_t), s));
  DBG_LAUNCH(ctx, stage, 0.0,
             k_msd_split<K><<<std::min(grid_for(gr.ng_max, 256), 152u * 8), 256, 0, s>>>(
                 keys, group_places(gr), gr.ng_dev, gr.ng, gr.lb, longest, mean, Sh::TILE, tb, split.as<uint8_t>(),
                 made));
  DBG_CUDA_TRY(cudaGetLastError());
  uint32_t c[CT_LAST + 1];
  DBG_TRY(read_counters(ctx, c));
  const uint32_t listed = c[CT_SPLIT], parts = c[CT_SPLIT + 1], ntiles = c[CT_SPLIT + 2], moved = c[CT_SPLIT + 3];
  if (!worth_split(c, n) || moved < c[CT_GATHERED] / 4) return DBG_OK;
  DevBuf pcount, poff;
  DBG_TRY(alloc_tmp(ctx, pcount, (uint64_t)parts * 4));
  DBG_TRY(alloc_tmp(ctx, poff, ((uint64_t)parts + 1) * 8));
  DBG_CUDA_TRY(cudaMemsetAsync(pcount.p, 0, (uint64_t)parts * 4, s));
  DBG_LAUNCH(ctx, stage, (double)moved * sizeof(K),
             k_msd_count<K><<<(unsigned)std::min<uint64_t>(ntiles, 4ull * std::max(1, ctx->num_sms)), MSD_BLOCK,
                              (size_t)4 << MSD_SPLIT_BITS, s>>>(keys, Sh::TILE, tb, pcount.as<uint32_t>()));
  DBG_TRY(scan_u32_async(ctx, pcount.as<uint32_t>(), parts, poff.as<uint64_t>(), stage));
  gr.split = std::move(split);
  DBG_TRY(msd_bounds<K>(ctx, gr, n, nullptr, stage));
  DBG_LAUNCH(ctx, stage, 0.0,
             k_split_bounds<<<std::min(listed, 152u * 8), 256, 0, s>>>(tb, listed, poff.as<uint64_t>(),
                                                                       SegShape<K>::TILE, gr.bound.as<uint64_t>(),
                                                                       pcount.as<uint32_t>()));
  const double bytes = 2.0 * (double)moved * (double)(sizeof(K) + (HAS_VAL ? 4 : 0));
  DBG_LAUNCH(ctx, stage, bytes,
             DBG_TRY((launch_msd_part<K, HAS_VAL, false>(ctx, keys, alt_keys, vals, alt_vals, n, 0, 0, tb, true,
                                                         pcount.as<uint32_t>(), MSD_SPLIT_BITS, ntiles))));
  DBG_LAUNCH(ctx, stage, bytes,
             (k_split_back<K, HAS_VAL><<<std::min(ntiles, 152u * 8), 512, 0, s>>>(tb, Sh::TILE, alt_keys, keys,
                                                                                 alt_vals, vals)));
  DBG_CUDA_TRY(cudaGetLastError());
  gr.lb.split = gr.split.as<uint8_t>();
  *done = true;
  return DBG_OK;
}

// The local pass's tiles and, sorted over every digit, the keys of the
// oversize ones.
struct TileSet {
  uint64_t tiles = 0;
  uint32_t gathered = 0;         // keys in oversize tiles, once known
  uint32_t oversize = 0;         // and those tiles' number,
  DevBuf bound, osize, olist;    // which olist lists
  DevBuf ooff, gk, gv;           // (seg_gather)
};

// The records' order by payload: *out = n words whose low halves list the
// records by ascending payload << shift.  (64-bit keys' sort: build_u64.cu.)
dbg_status order_by_payload(dbg_ctx *ctx, const uint32_t *v, uint64_t n, int shift, DevBuf &buf,
                            const uint64_t **out);

// Tile bounds of the local pass over n keys in the groups gr (sorted by
// their bits from gr.lb up), and the oversize tiles (longer than the
// shared-memory capacity): their sizes, a list of them, and in the counters
// their keys and number.
template <class K>
dbg_status seg_tiles(dbg_ctx *ctx, const K *kin, uint64_t n, Groups &gr, TileSet &ts, int stage) {
  using Sh = SegShape<K>;
  cudaStream_t s = ctx->stream;
  const uint64_t tiles = (n + Sh::TILE - 1) / Sh::TILE;
  if (tiles > 0x7fffffffull) return DBG_EOVERFLOW;
  ts.tiles = tiles;
  DBG_TRY(alloc_tmp(ctx, ts.osize, tiles * 4));
  DBG_TRY(alloc_tmp(ctx, ts.olist, tiles * 4));
  if (gr.ng && !gr.bound.p) DBG_TRY(msd_bounds<K>(ctx, gr, n, nullptr, stage));
  if (gr.bound.p) {
    ts.bound = std::move(gr.bound);
  } else {
    DBG_TRY(alloc_tmp(ctx, ts.bound, (tiles + 1) * 8));
    DBG_LAUNCH(ctx, stage, 0.0,
               k_seg_bounds<K><<<grid_for(tiles + 1, 256), 256, 0, s>>>(kin, n, gr.lb.fixed, Sh::TILE, tiles,
                                                                       ts.bound.as<uint64_t>()));
  }
  DBG_CUDA_TRY(cudaMemsetAsync(ctx->d_counters + CT_GATHERED, 0, (CT_MIXED - CT_GATHERED + 1) * 4, s));
  DBG_LAUNCH(ctx, stage, 0.0,
             k_seg_oversize<K><<<grid_for(tiles, 256), 256, 0, s>>>(
                 kin, ts.bound.as<uint64_t>(), tiles, (uint32_t)(SEG_BLOCK * Sh::ITEMS), ts.osize.as<uint32_t>(),
                 ts.olist.as<uint32_t>(), ctx->d_counters + CT_GATHERED, ctx->d_counters + CT_MIXED,
                 ctx->d_counters + CT_OVERSIZE, ctx->d_err));
  DBG_CUDA_TRY(cudaGetLastError());
  return DBG_OK;
}

// The keys (and payloads) of the oversize tiles, gathered and sorted over
// every digit, once ts.gathered says that there are some.
template <class K, bool HAS_VAL>
dbg_status seg_gather(dbg_ctx *ctx, const K *kin, const uint32_t *vin, ValOrder vo, int key_bits, TileSet &ts,
                      int stage) {
  if (ts.gathered == 0) return DBG_OK;
  cudaStream_t s = ctx->stream;
  const uint64_t tiles = ts.tiles;
  const uint32_t *G = &ts.gathered;
  DevBuf &bound = ts.bound, &osize = ts.osize, &ooff = ts.ooff, &gk = ts.gk, &gv = ts.gv;
  DBG_TRY(alloc_tmp(ctx, ooff, (tiles + 1) * 8));
  DBG_TRY(scan_u32_async(ctx, osize.as<uint32_t>(), tiles, ooff.as<uint64_t>(), stage));
  // the oversize tiles, gathered in order and sorted over every digit
  const uint64_t g = *G;
  DevBuf galt, gvalt, small;
  DBG_TRY(alloc_tmp(ctx, gk, g * sizeof(K)));
  if (HAS_VAL) DBG_TRY(alloc_tmp(ctx, gv, g * 4));
  DBG_TRY(alloc_tmp(ctx, small, MAX_PASSES * RADIX * 16));
  unsigned long long *hist = small.as<unsigned long long>();
  uint64_t *dbase = reinterpret_cast<uint64_t *>(hist + MAX_PASSES * RADIX);
  const int passes = passes_for_bits(key_bits);
  DBG_LAUNCH(ctx, stage, 2.0 * g * (sizeof(K) + (HAS_VAL ? 4 : 0)),
             k_seg_gather<K, HAS_VAL><<<(unsigned)std::min<uint64_t>(tiles, 152ull * 8), 256, 0, s>>>(
                 kin, vin, bound.as<uint64_t>(), osize.as<uint32_t>(), ooff.as<uint64_t>(), tiles, gk.as<K>(),
                 HAS_VAL ? gv.as<uint32_t>() : nullptr));
  DevBuf order;  // for records in no order: the words that order them by payload
  const uint64_t *words = nullptr;
  if (HAS_VAL && vo.sort) DBG_TRY(order_by_payload(ctx, gv.as<uint32_t>(), g, vo.shift, order, &words));
  DBG_TRY(alloc_tmp(ctx, galt, g * sizeof(K)));
  if (HAS_VAL) DBG_TRY(alloc_tmp(ctx, gvalt, g * 4));
  if (words) {
    DBG_LAUNCH(ctx, stage, 2.0 * g * (sizeof(K) + 4),
               k_permute<K><<<grid_for(g, 256 * 8), 256, 0, s>>>(words, g, gk.as<K>(), gv.as<uint32_t>(),
                                                                 galt.as<K>(), gvalt.as<uint32_t>()));
    std::swap(gk, galt);
    std::swap(gv, gvalt);
    order.release();
  }
  DBG_CUDA_TRY(cudaMemsetAsync(hist, 0, MAX_PASSES * RADIX * 8, s));
  DBG_LAUNCH(ctx, stage, (double)g * sizeof(K),
             k_digit_hist<K><<<std::min(grid_for(g, 256 * 16), 152u * 8), 256, 0, s>>>(gk.as<K>(), g, 0, passes,
                                                                                       hist));
  K *kp = gk.as<K>(), *ka = galt.as<K>();
  uint32_t *vp = HAS_VAL ? gv.as<uint32_t>() : nullptr, *va = HAS_VAL ? gvalt.as<uint32_t>() : nullptr;
  DBG_TRY((radix_sort<K, HAS_VAL>(ctx, &kp, &ka, &vp, &va, g, key_bits, hist, dbase)));
  if (kp != gk.as<K>()) std::swap(gk, galt);
  if (HAS_VAL && vp != gv.as<uint32_t>()) std::swap(gv, gvalt);
  ctx->local_sort_fallbacks++;
  return DBG_OK;
}

// The listed tiles of k_seg_rank, sorted by the digit passes.
template <class K>
dbg_status seg_sort_listed(dbg_ctx *ctx, const K *kin, const uint32_t *vin, K *kout, uint32_t *vout, Groups &gr,
                           ValOrder vo, TileSet &ts, const uint32_t *fb_list, const uint32_t *fb_count,
                           uint32_t nfb) {
  using Sh = SegShape<K>;
  const int rank = local_rank_method(ctx, sizeof(K) == 16);
  auto kern = rank == RANK_MATCH    ? k_seg_sort<K, Sh::ITEMS, RANK_MATCH>
              : rank == RANK_ATOMIC ? k_seg_sort<K, Sh::ITEMS, RANK_ATOMIC>
                                    : k_seg_sort<K, Sh::ITEMS, RANK_BALLOT>;
  constexpr size_t smem = sizeof(SegSortSmem<K, true, Sh::ITEMS>);
  set_smem_attrs(kern, smem);
  const unsigned grid = (unsigned)std::min<uint64_t>(nfb, 2ull * (uint64_t)std::max(1, ctx->num_sms));
  DBG_LAUNCH(ctx, ST_LOCAL_SORT_NODES, 0.0,
             kern<<<grid, SEG_BLOCK, smem, ctx->stream>>>(
                 kin, vin, ts.bound.as<uint64_t>(), ts.osize.as<uint32_t>(), ts.ooff.as<uint64_t>(), ts.gk.as<K>(),
                 ts.gv.as<uint32_t>(), kout, vout, gr.lb, vo, fb_list, fb_count));
  DBG_CUDA_TRY(cudaGetLastError());
  return DBG_OK;
}

// k_seg_rank over every tile, then the digit passes for the tiles that it
// listed: the sorted records.
template <class K>
dbg_status seg_rank_tiles(dbg_ctx *ctx, const K *kin, const uint32_t *vin, K *kout, uint32_t *vout, uint64_t n,
                          Groups &gr, ValOrder vo, TileSet &ts) {
  auto kern = k_seg_rank<K, false>;
  set_smem_attrs(kern, sizeof(SegRankSmem<K>));
  DevBuf fb;
  DBG_TRY(alloc_tmp(ctx, fb, ts.tiles * 4));
  uint32_t *nlisted = ctx->d_counters + CT_LISTED;
  DBG_CUDA_TRY(cudaMemsetAsync(nlisted, 0, 4, ctx->stream));
  DBG_LAUNCH(ctx, ST_LOCAL_SORT_NODES, 2.0 * (double)n * (sizeof(K) + 4),
             kern<<<(unsigned)ts.tiles, RANK_BLOCK, sizeof(SegRankSmem<K>), ctx->stream>>>(
                 kin, vin, ts.bound.as<uint64_t>(), ts.osize.as<uint32_t>(), ts.ooff.as<uint64_t>(), ts.gk.as<K>(),
                 ts.gv.as<uint32_t>(), kout, vout, gr.lb, vo, fb.as<uint32_t>(), nlisted, nullptr, nullptr));
  DBG_CUDA_TRY(cudaGetLastError());
  uint32_t c[CT_LAST + 1];
  DBG_TRY(read_counters(ctx, c));
  ctx->rank_fallback_tiles += c[CT_LISTED];
  if (c[CT_LISTED])
    DBG_TRY(seg_sort_listed<K>(ctx, kin, vin, kout, vout, gr, vo, ts, fb.as<uint32_t>(), nlisted, c[CT_LISTED]));
  return DBG_OK;
}

// The local pass over records in the groups gr: the fully sorted records
// (equal keys by payload, in the order vo) to kout / vout.
template <class K>
dbg_status seg_sort_records(dbg_ctx *ctx, const K *kin, const uint32_t *vin, K *kout, uint32_t *vout, uint64_t n,
                            Groups &gr, ValOrder vo, TileSet &ts) {
  using Sh = SegShape<K>;
  if (ctx->seg_rank)
    return seg_rank_tiles<K>(ctx, kin, vin, kout, vout, n, gr, vo, ts);
  const int rank = local_rank_method(ctx, sizeof(K) == 16);
  const uint64_t tiles = ts.tiles;
  const DevBuf &bound = ts.bound, &osize = ts.osize, &ooff = ts.ooff, &gk = ts.gk, &gv = ts.gv;
  const int v = ctx->sort_variant[sizeof(K) == 16 ? 5 : 4];
  if (v >= 3) {
    // the wide form: 384 threads x (2/3 of the items), the same capacity
    constexpr int WB = 384, WI = Sh::ITEMS * SEG_BLOCK / WB;
    static_assert(WB * WI == SEG_BLOCK * Sh::ITEMS, "same tile capacity");
    auto kern = rank == RANK_MATCH    ? k_seg_sort<K, WI, RANK_MATCH, WB>
                : rank == RANK_ATOMIC ? k_seg_sort<K, WI, RANK_ATOMIC, WB>
                                      : k_seg_sort<K, WI, RANK_BALLOT, WB>;
    constexpr size_t smem = sizeof(SegSortSmem<K, true, WI, WB>);
    set_smem_attrs(kern, smem);
    DBG_LAUNCH(ctx, ST_LOCAL_SORT_NODES, 2.0 * (double)n * (sizeof(K) + 4),
               kern<<<(unsigned)tiles, WB, smem, ctx->stream>>>(
                   kin, vin, bound.as<uint64_t>(), osize.as<uint32_t>(), ooff.as<uint64_t>(), gk.as<K>(),
                   gv.as<uint32_t>(), kout, vout, gr.lb, vo, nullptr, nullptr));
    DBG_CUDA_TRY(cudaGetLastError());
    return DBG_OK;
  }
  auto kern = rank == RANK_MATCH    ? k_seg_sort<K, Sh::ITEMS, RANK_MATCH>
              : rank == RANK_ATOMIC ? k_seg_sort<K, Sh::ITEMS, RANK_ATOMIC>
                                    : k_seg_sort<K, Sh::ITEMS, RANK_BALLOT>;
  constexpr size_t smem = sizeof(SegSortSmem<K, true, Sh::ITEMS>);
  set_smem_attrs(kern, smem);
  DBG_LAUNCH(ctx, ST_LOCAL_SORT_NODES, 2.0 * (double)n * (sizeof(K) + 4),
             kern<<<(unsigned)tiles, SEG_BLOCK, smem, ctx->stream>>>(
                 kin, vin, bound.as<uint64_t>(), osize.as<uint32_t>(), ooff.as<uint64_t>(), gk.as<K>(),
                 gv.as<uint32_t>(), kout, vout, gr.lb, vo, nullptr, nullptr));
  DBG_CUDA_TRY(cudaGetLastError());
  return DBG_OK;
}

// The tiles of STEP-2's local pass: tile t's tcount[t] distinct keys start at
// bound[t] of the key buffer that they were staged in, their multiplicities
// there in mult; toff numbers them.
struct EdgeTiles {
  uint64_t tiles = 0;
  DevBuf bound, tcount, toff, mult;
  bool uneven = false;  // the sort split long groups
  bool dense = false;   // mult holds one per edge, in edge order
  void release() {
    for (DevBuf *b : {&bound, &tcount, &toff, &mult}) b->release();
  }
};

// The local pass of STEP-2 over n edge keys in the groups gr.  Leaves the E
// distinct keys in kin[0, E) and their multiplicities in mult_out (allocated
// here), kstage (n keys) being scratch; or, with `staged`, in kstage by tiles.
template <class K>
dbg_status seg_rle(dbg_ctx *ctx, K *kin, K *kstage, uint64_t n, Groups &gr, int key_bits, DevBuf *mult_out,
                   EdgeTiles *staged, uint64_t *E) {
  using Sh = SegShape<K>;
  cudaStream_t s = ctx->stream;
  TileSet ts;
  DevBuf gheads, guniq, mstage, tcount, toff, over, crowded;
  uint64_t H = 0;
  DBG_TRY(seg_tiles<K>(ctx, kin, n, gr, ts, ST_LOCAL_SORT_EDGES));
  const uint64_t tiles = ts.tiles;
  uint32_t c[CT_LAST + 1];
  // the tiles again once long groups have been split
  auto split = [&](bool *done) -> dbg_status {
    *done = false;
    if (!worth_split(c, n)) return DBG_OK;
    DBG_TRY((msd_split<K, false>(ctx, kin, kstage, nullptr, nullptr, n, gr, ST_SORT_EDGES, done)));
    if (*done) DBG_TRY(seg_tiles<K>(ctx, kin, n, gr, ts, ST_LOCAL_SORT_EDGES));
    return DBG_OK;
  };
  DBG_TRY(alloc_tmp(ctx, mstage, n * 4));
  DBG_TRY(alloc_tmp(ctx, tcount, tiles * 4));
  DBG_TRY(alloc_tmp(ctx, toff, (tiles + 1) * 8));
  const int rank = local_rank_method(ctx, sizeof(K) == 16);
  // the radix-sorting kernel over `count` tiles: all of them, those of a
  // list, or as many of the list as the device has counted in *dcount
  auto sort_tiles = [&](uint64_t count, const uint32_t *list, const uint32_t *dcount, double bytes) -> dbg_status {
    auto radix = rank == RANK_MATCH    ? k_seg_rle<K, Sh::ITEMS, RANK_MATCH>
                 : rank == RANK_ATOMIC ? k_seg_rle<K, Sh::ITEMS, RANK_ATOMIC>
                                       : k_seg_rle<K, Sh::ITEMS, RANK_BALLOT>;
    constexpr size_t rsmem = sizeof(SegSortSmem<K, false, Sh::ITEMS>);
    set_smem_attrs(radix, rsmem);
    if (count == 0) return DBG_OK;
    if (dcount) count = std::min<uint64_t>(count, 2ull * (uint64_t)std::max(1, ctx->num_sms));
    DBG_LAUNCH(ctx, ST_LOCAL_SORT_EDGES, bytes,
               radix<<<(unsigned)count, SEG_BLOCK, rsmem, s>>>(
                   kin, ts.bound.as<uint64_t>(), ts.osize.as<uint32_t>(), ts.ooff.as<uint64_t>(), guniq.as<K>(),
                   gheads.as<uint32_t>(), (uint32_t)H, kstage, mstage.as<uint32_t>(), tcount.as<uint32_t>(), gr.lb,
                   list, dcount));
    DBG_CUDA_TRY(cudaGetLastError());
    return DBG_OK;
  };
  auto gather = [&]() -> dbg_status {
    if (ts.gathered == 0) return DBG_OK;
    DBG_TRY((seg_gather<K, false>(ctx, kin, nullptr, ValOrder{}, key_bits, ts, ST_LOCAL_SORT_EDGES)));
    DBG_TRY(alloc_tmp(ctx, guniq, (uint64_t)ts.gathered * sizeof(K)));
    DBG_TRY(alloc_tmp(ctx, gheads, ((uint64_t)ts.gathered + 1) * 4));
    return run_length_reduce<K>(ctx, ts.gk.as<K>(), ts.gathered, guniq.as<K>(), gheads.as<uint32_t>(), &H);
  };
  bool final = false;  // the scan below covers every tile
  if (ctx->count_first) {
    // count-first; the tiles that overflow their table, or would, are listed
    // and ordered copy by copy.  Those with crowded buckets (by digits) and the
    // oversize ones follow if one read-back, with the total that holds
    // otherwise, says that there are some.
    auto count = rank == RANK_MATCH    ? k_seg_count<K, RANK_MATCH>
                 : rank == RANK_ATOMIC ? k_seg_count<K, RANK_ATOMIC>
                                       : k_seg_count<K, RANK_BALLOT>;
    const size_t csmem = rank == RANK_MATCH    ? sizeof(SegCountSmem<K, RANK_MATCH>)
                         : rank == RANK_ATOMIC ? sizeof(SegCountSmem<K, RANK_ATOMIC>)
                                               : sizeof(SegCountSmem<K, RANK_BALLOT>);
    set_smem_attrs(count, csmem);
    DBG_TRY(alloc_tmp(ctx, over, tiles * 4));
    for (bool again = true; again;) {
      DBG_LAUNCH(ctx, ST_LOCAL_SORT_EDGES, (double)n * sizeof(K),
                 count<<<(unsigned)tiles, SEG_BLOCK, csmem, s>>>(
                     kin, ts.bound.as<uint64_t>(), ts.osize.as<uint32_t>(), kstage, mstage.as<uint32_t>(),
                     tcount.as<uint32_t>(), over.as<uint32_t>(), ctx->d_counters + CT_LISTED, gr.lb, ctx->seg_rank,
                     ctx->d_counters + CT_LONG));
      DBG_CUDA_TRY(cudaGetLastError());
      uint32_t *listed = ctx->d_counters + CT_LISTED;
      if (ctx->seg_rank) {
        DBG_TRY(alloc_tmp(ctx, crowded, tiles * 4));
        set_smem_attrs(k_rank_rle<K>, sizeof(RankRleSmem<K>));
        DBG_LAUNCH(ctx, ST_LOCAL_SORT_EDGES, 0.0,
                   k_rank_rle<K><<<(unsigned)std::min<uint64_t>(tiles, 2ull * (uint64_t)std::max(1, ctx->num_sms)),
                                   RANK_BLOCK, sizeof(RankRleSmem<K>), s>>>(
                       kin, ts.bound.as<uint64_t>(), kstage, mstage.as<uint32_t>(), tcount.as<uint32_t>(), gr.lb,
                       over.as<uint32_t>(), listed, crowded.as<uint32_t>(), ctx->d_counters + CT_CROWDED));
        DBG_CUDA_TRY(cudaGetLastError());
      } else {
        DBG_TRY(sort_tiles(tiles, over.as<uint32_t>(), listed, 0.0));
      }
      DBG_TRY(scan_u32_async(ctx, tcount.as<uint32_t>(), tiles, toff.as<uint64_t>(), ST_LOCAL_SORT_EDGES, CT_TOTAL));
      DBG_TRY(read_counters(ctx, c));
      ts.gathered = c[CT_GATHERED];
      ts.oversize = c[CT_OVERSIZE];
      const uint32_t met[3] = {c[CT_LISTED], c[CT_LONG], c[CT_CROWDED]};
      DBG_TRY(split(&again));
      if (again) continue;
      ctx->count_overflow_tiles += met[0];
      ctx->rank_fallback_tiles += met[1] + met[2];
      final = ts.oversize == 0 && c[CT_CROWDED] == 0;
      if (!final) {
        const uint32_t n_crowded = c[CT_CROWDED];
        DBG_TRY(gather());
        DBG_TRY(sort_tiles(n_crowded, crowded.as<uint32_t>(), nullptr, 0.0));
        DBG_TRY(sort_tiles(ts.oversize, ts.olist.as<uint32_t>(), nullptr, 0.0));
      }
    }
  } else {
    DBG_TRY(read_counters(ctx, c));
    ts.gathered = c[CT_GATHERED];
    bool again = false;
    DBG_TRY(split(&again));
    if (again) {
      DBG_TRY(read_counters(ctx, c));
      ts.gathered = c[CT_GATHERED];
    }
    DBG_TRY(gather());
    DBG_TRY(sort_tiles(tiles, nullptr, nullptr, (double)n * sizeof(K)));
  }
  if (!final) {
    DBG_TRY(scan_u32_async(ctx, tcount.as<uint32_t>(), tiles, toff.as<uint64_t>(), ST_LOCAL_SORT_EDGES, CT_TOTAL));
    DBG_TRY(read_counters(ctx, c));
  }
  const uint32_t total = c[CT_TOTAL];
  const DevBuf &bound = ts.bound;
  *E = total;
  if (staged) {
    staged->tiles = tiles;
    staged->bound = std::move(ts.bound);
    staged->tcount = std::move(tcount);
    staged->toff = std::move(toff);
    staged->mult = std::move(mstage);
    staged->uneven = gr.split.p != nullptr;
    return DBG_OK;
  }
  DBG_TRY(alloc_buf(ctx, *mult_out, std::max<uint64_t>(1, total) * 4));
  DBG_LAUNCH(ctx, ST_LOCAL_SORT_EDGES, 2.0 * total * (sizeof(K) + 4),
             k_seg_compact<K><<<(unsigned)std::min<uint64_t>(tiles, 152ull * 16), 256, 0, s>>>(
                 bound.as<uint64_t>(), tcount.as<uint32_t>(), toff.as<uint64_t>(), tiles, kstage,
                 mstage.as<uint32_t>(), kin, mult_out->as<uint32_t>()));
  DBG_CUDA_TRY(cudaGetLastError());
  return DBG_OK;
}

// STEP-2 over n edge keys by plan p (p.local()): the global passes, then the
// local pass with the run-length reduce.  The E distinct keys end in *alt,
// their multiplicities in *mult, or (mult == nullptr) both as *staged tells.
template <class K>
dbg_status sort_count_keys(dbg_ctx *ctx, K **kp, K **alt, uint64_t n, const SortPlan<K> &p,
                           const unsigned long long *d_hist, uint64_t *d_digit_base, DevBuf *mult, EdgeTiles *staged,
                           uint64_t *E) {
  uint32_t *vn = nullptr, *van = nullptr;
  Groups gr;
  if (p.msd) {
    DBG_TRY((msd_sort<K, false>(ctx, kp, alt, &vn, &van, n, p, d_hist, gr)));
  } else {
    DBG_TRY((radix_sort<K, false>(ctx, kp, alt, &vn, &van, n, p.bits, d_hist, d_digit_base, p.first_pass)));
    gr.lb.fixed = RADIX_BITS * p.first_pass;
  }
  DBG_TRY(seg_rle<K>(ctx, *kp, *alt, n, gr, p.bits, mult, staged, E));
  if (!staged) std::swap(*kp, *alt);
  return DBG_OK;
}

// STEP-3's sort of R records by key, equal keys by payload, by plan p: the
// global passes and the local pass's tiles (p.local()).  The records come in
// payload order, which the least-significant-first passes keep and the local
// pass restores after the MSD passes.
template <class K>
dbg_status sort_records_global(dbg_ctx *ctx, K **rk, K **rk_alt, uint32_t **rv, uint32_t **rv_alt, uint64_t R,
                               const SortPlan<K> &p, ValOrder &vo, unsigned long long *d_hist,
                               uint64_t *d_digit_base, Groups &gr, TileSet &ts) {
  if (p.msd) {
    DBG_TRY((msd_sort<K, true>(ctx, rk, rk_alt, rv, rv_alt, R, p, d_hist, gr)));
    vo.sort = p.passes > 0;
  } else {
    DBG_TRY((radix_sort<K, true>(ctx, rk, rk_alt, rv, rv_alt, R, p.bits, d_hist, d_digit_base, p.first_pass, p.adj)));
    gr.lb.fixed = RADIX_BITS * p.first_pass - p.adj;
  }
  return seg_tiles<K>(ctx, *rk, R, gr, ts, ST_LOCAL_SORT_NODES);
}

// The whole sort, the sorted records in *rk / *rv.
template <class K>
dbg_status sort_records(dbg_ctx *ctx, K **rk, K **rk_alt, uint32_t **rv, uint32_t **rv_alt, uint64_t R,
                        const SortPlan<K> &p, ValOrder vo, unsigned long long *d_hist, uint64_t *d_digit_base) {
  if (!p.local() || R <= 1) return radix_sort<K, true>(ctx, rk, rk_alt, rv, rv_alt, R, p.bits, d_hist, d_digit_base);
  Groups gr;
  TileSet ts;
  DBG_TRY(sort_records_global<K>(ctx, rk, rk_alt, rv, rv_alt, R, p, vo, d_hist, d_digit_base, gr, ts));
  uint32_t c[CT_LAST + 1];
  DBG_TRY(read_counters(ctx, c));
  ts.gathered = c[CT_GATHERED];
  bool again = false;
  if (worth_split(c, R))
    DBG_TRY((msd_split<K, true>(ctx, *rk, *rk_alt, *rv, *rv_alt, R, gr, ST_SORT_NODES, &again)));
  if (again) {
    DBG_TRY(seg_tiles<K>(ctx, *rk, R, gr, ts, ST_LOCAL_SORT_NODES));
    DBG_TRY(read_counters(ctx, c));
    ts.gathered = c[CT_GATHERED];
  }
  ts.oversize = c[CT_OVERSIZE];
  DBG_TRY((seg_gather<K, true>(ctx, *rk, *rv, vo, p.bits, ts, ST_LOCAL_SORT_NODES)));
  DBG_TRY(seg_sort_records<K>(ctx, *rk, *rv, *rk_alt, *rv_alt, R, gr, vo, ts));
  std::swap(*rk, *rk_alt);
  std::swap(*rv, *rv_alt);
  return DBG_OK;
}

// The payload order of node records: (e << 1 | role) of `edges` edges, the
// side bits on top or not, with or without reads of exactly k bases; or of
// read numbers below `reads`.
inline int bit_length(uint64_t x) {
  int b = 0;
  while (x >> b) b++;
  return b;
}
// x << shift, as a key
inline uint64_t key_from(uint64_t x, int shift, uint64_t) { return shift < 64 ? x << shift : 0; }
inline Key128 key_from(uint64_t x, int shift, Key128) {
  if (shift >= 64) return Key128{x << (shift - 64), 0};
  return Key128{shift ? x >> (64 - shift) : 0, x << shift};
}
inline ValOrder edge_end_order(uint64_t edges, bool sides, bool isolated) {
  ValOrder vo;
  vo.shift = sides ? 2 : 0;
  vo.pb = std::max(1, std::min(31, bit_length(edges)));
  vo.dups = isolated;
  return vo;
}
inline ValOrder read_order(uint64_t reads) {
  ValOrder vo;
  vo.pb = std::max(1, std::min(31, bit_length(reads / 2 + 1)));
  return vo;
}

// The plan of a record sort.  Least significant first, with records ranked
// within groups, the digits are aligned with the top of the key, so that the
// global passes resolve 8 bits each of it and leave short groups.
template <class K>
SortPlan<K> plan_records(const dbg_ctx *ctx, uint64_t R, int bits, bool align, double density = 1.0) {
  SortPlan<K> p = plan_sort<K>(ctx, R, bits, ctx->partition_first && ctx->seg_rank, density);
  if (!p.msd && ctx->hybrid_sort && ctx->seg_rank && align) {
    const int adj = (8 - bits % 8) % 8;
    const int q0 = hybrid_first_pass<K>(R, bits + adj);
    if (q0 > 0) {
      p.first_pass = q0;
      p.adj = adj;
    }
  }
  return p;
}

// K6 by reduce-then-scan over R sorted node records; returns the node count
// and the number of edge ends.  E_all > 0: the records hold both ends of
// all E_all edges, and src / dst are written through the partition of the
// edge ends by edge range (k_scatter_ends) instead of at random.  adj_side
// (E_all > 0 only): the payloads carry the side bits, stored per slot.
template <class K>
dbg_status assign_node_ids(dbg_ctx *ctx, const K *rk, const uint32_t *rv, uint64_t R, K *node_keys,
                           uint64_t *row_ptr, dbg_graph *g, uint32_t base_v, uint64_t base_slot, uint64_t *V,
                           uint64_t *ends, uint64_t E_all = 0, uint8_t *adj_side = nullptr) {
  cudaStream_t s = ctx->stream;
  const uint64_t tiles = (R + RS_TILE - 1) / RS_TILE;
  DevBuf hc, ec, ho, eo;
  DBG_TRY(alloc_tmp(ctx, hc, tiles * 4));
  DBG_TRY(alloc_tmp(ctx, ec, tiles * 4));
  DBG_TRY(alloc_tmp(ctx, ho, (tiles + 1) * 8));
  DBG_TRY(alloc_tmp(ctx, eo, (tiles + 1) * 8));
  DBG_LAUNCH(ctx, ST_NODE_IDS, (double)R * (sizeof(K) + 4),
             k_count_heads<K><<<(unsigned)tiles, SCAN_BLOCK, 0, s>>>(rk, rv, R, hc.as<uint32_t>(), ec.as<uint32_t>()));
  uint32_t nv = 0, ne = 0;
  DBG_TRY(scan_u32(ctx, hc.as<uint32_t>(), tiles, ho.as<uint64_t>(), &nv, ST_NODE_IDS));
  DBG_TRY(scan_u32(ctx, ec.as<uint32_t>(), tiles, eo.as<uint64_t>(), &ne, ST_NODE_IDS));
  if (E_all > 0) {
    int bshift = 10;
    while ((E_all + (1ull << bshift) - 1) >> bshift > 256) bshift++;
    DevBuf part, fill;
    DBG_TRY(alloc_tmp(ctx, part, 2 * E_all * 8));
    DBG_TRY(alloc_tmp(ctx, fill, 256 * 4));
    DBG_CUDA_TRY(cudaMemsetAsync(fill.p, 0, 256 * 4, s));
    const double wbytes = (double)R * (sizeof(K) + 4) + (double)nv * (sizeof(K) + 8) + (double)ne * (adj_side ? 14 : 13);
    if constexpr (sizeof(K) == 8) {
      // persistent CTAs, two per SM, with the next tile's records in flight
      constexpr size_t smem = sizeof(WriteNodesSmem<K>);
      set_smem_attrs(k_write_nodes_p<K, true>, smem);
      const unsigned grid = (unsigned)std::min<uint64_t>(tiles, 2ull * (uint64_t)ctx->num_sms);
      DBG_LAUNCH(ctx, ST_NODE_IDS, wbytes,
                 k_write_nodes_p<K, true><<<grid, SCAN_BLOCK, smem, s>>>(
                     rk, rv, R, ho.as<uint64_t>(), eo.as<uint64_t>(), node_keys, row_ptr, g->src.as<uint32_t>(),
                     g->dst.as<uint32_t>(), g->adj_edge.as<uint32_t>(), g->adj_role.as<uint8_t>(), base_v,
                     base_slot, part.as<uint64_t>(), fill.as<uint32_t>(), bshift, ctx->spin_limit, ctx->d_err,
                     adj_side));
    } else {
      DBG_LAUNCH(ctx, ST_NODE_IDS, wbytes,
                 k_write_nodes<K, true><<<(unsigned)tiles, SCAN_BLOCK, 0, s>>>(
                     rk, rv, R, ho.as<uint64_t>(), eo.as<uint64_t>(), node_keys, row_ptr, g->src.as<uint32_t>(),
                     g->dst.as<uint32_t>(), g->adj_edge.as<uint32_t>(), g->adj_role.as<uint8_t>(), base_v,
                     base_slot, part.as<uint64_t>(), fill.as<uint32_t>(), bshift, adj_side));
    }
    DBG_LAUNCH(ctx, ST_NODE_IDS, 2.0 * E_all * (8 + 4),
               k_scatter_ends<<<grid_for(2 * E_all, 256 * 16), 256, 0, s>>>(part.as<uint64_t>(), 2 * E_all,
                                                                          g->src.as<uint32_t>(),
                                                                          g->dst.as<uint32_t>()));
  } else {
    DBG_LAUNCH(ctx, ST_NODE_IDS, (double)R * (sizeof(K) + 4) + (double)nv * (sizeof(K) + 8) + (double)ne * 9,
               k_write_nodes<K, false><<<(unsigned)tiles, SCAN_BLOCK, 0, s>>>(
                   rk, rv, R, ho.as<uint64_t>(), eo.as<uint64_t>(), node_keys, row_ptr, g->src.as<uint32_t>(),
                   g->dst.as<uint32_t>(), g->adj_edge.as<uint32_t>(), g->adj_role.as<uint8_t>(), base_v, base_slot,
                   nullptr, nullptr, 0));
  }
  DBG_CUDA_TRY(cudaGetLastError());
  *V = nv;
  *ends = ne;
  return DBG_OK;
}

// The local pass over R node records in the groups gr, fused with the node-ID
// pass: the graph's node keys, row_ptr, adjacency and edge ends.  Returns
// |V| and the number of edge ends; *done = false, with the oversize tiles
// gathered, where the unfused passes are to do it.
template <class K>
dbg_status rank_and_assign(dbg_ctx *ctx, K *rk, uint32_t *rv, K *ukeys, uint32_t *vals, uint64_t R,
                           uint64_t E, uint64_t I, int key_bits, Groups &gr, ValOrder vo, TileSet &ts, dbg_graph *g,
                           bool sides, bool uneven, bool *done, uint64_t *V, uint64_t *ends) {
  cudaStream_t s = ctx->stream;
  const uint64_t tiles = ts.tiles;
  DevBuf heads, tcount, hoff, ecount, eoff, fb;
  DBG_TRY(alloc_tmp(ctx, heads, (R / 32 + tiles + 2) * 4));
  DBG_TRY(alloc_tmp(ctx, tcount, tiles * 4));
  DBG_TRY(alloc_tmp(ctx, hoff, (tiles + 1) * 8));
  DBG_TRY(alloc_tmp(ctx, fb, tiles * 4));
  if (I > 0) {
    DBG_TRY(alloc_tmp(ctx, ecount, tiles * 4));
    DBG_TRY(alloc_tmp(ctx, eoff, (tiles + 1) * 8));
  }
  uint32_t c[CT_LAST + 1], *nlisted = ctx->d_counters + CT_LISTED;
  // the tiles' node and edge-end counts, scanned
  auto scan_tiles = [&]() -> dbg_status {
    if (I > 0) {
      DBG_LAUNCH(ctx, ST_NODE_IDS, 4.0 * R,
                 k_tile_ends<<<(unsigned)std::min<uint64_t>(tiles, 152ull * 16), 256, 0, s>>>(
                     ts.bound.as<uint64_t>(), (uint32_t)tiles, vals, ecount.as<uint32_t>()));
      DBG_TRY(scan_u32_async(ctx, ecount.as<uint32_t>(), tiles, eoff.as<uint64_t>(), ST_NODE_IDS, CT_ENDS));
    }
    DBG_TRY(scan_u32_async(ctx, tcount.as<uint32_t>(), tiles, hoff.as<uint64_t>(), ST_NODE_IDS, CT_TOTAL));
    return read_counters(ctx, c);
  };
  static_assert(SegRankSmem<K>::CAP == SEG_BLOCK * SegShape<K>::ITEMS, "same tile capacity as the digit-pass kernel");
  auto rank = k_seg_rank<K, true>;
  set_smem_attrs(rank, sizeof(SegRankSmem<K>));
  auto split = [&](bool *did) -> dbg_status {
    DBG_TRY((msd_split<K, true>(ctx, rk, ukeys, rv, vals, R, gr, ST_SORT_NODES, did)));
    return *did ? seg_tiles<K>(ctx, rk, R, gr, ts, ST_LOCAL_SORT_NODES) : DBG_OK;
  };
  // (where the edge keys had long groups, the records have: split before the
  // first try)
  bool again = false;
  if (uneven) DBG_TRY(split(&again));
  for (again = true; again;) {
    DBG_LAUNCH(ctx, ST_LOCAL_SORT_NODES, 2.0 * (double)R * (sizeof(K) + 4),
               rank<<<(unsigned)tiles, RANK_BLOCK, sizeof(SegRankSmem<K>), s>>>(
                   rk, rv, ts.bound.as<uint64_t>(), ts.osize.as<uint32_t>(), nullptr, nullptr, nullptr, ukeys, vals,
                   gr.lb, vo, fb.as<uint32_t>(), nlisted, heads.as<uint32_t>(), tcount.as<uint32_t>()));
    DBG_CUDA_TRY(cudaGetLastError());
    DBG_TRY(scan_tiles());
    ts.gathered = c[CT_GATHERED];
    ts.oversize = c[CT_OVERSIZE];
    again = false;
    if (!uneven && worth_split(c, R)) DBG_TRY(split(&again));
  }
  // many records in oversize tiles, which one CTA each would go through (a
  // million records: about 0.3 ms): the unfused passes
  *done = ts.gathered <= 1u << 20;
  if (!*done) return seg_gather<K, true>(ctx, rk, rv, vo, key_bits, ts, ST_LOCAL_SORT_NODES);
  if (c[CT_LISTED] || ts.oversize) {
    const uint32_t listed = c[CT_LISTED], both = listed + ts.oversize;
    ctx->rank_fallback_tiles += listed;
    const unsigned grid = (unsigned)std::min<uint64_t>(both, 4ull * (uint64_t)std::max(1, ctx->num_sms));
    DBG_TRY((seg_gather<K, true>(ctx, rk, rv, vo, key_bits, ts, ST_LOCAL_SORT_NODES)));
    if (ts.oversize)
      DBG_LAUNCH(ctx, ST_LOCAL_SORT_NODES, 2.0 * ts.gathered * (sizeof(K) + 4),
                 k_seg_place<K><<<grid, 256, 0, s>>>(ts.bound.as<uint64_t>(), ts.osize.as<uint32_t>(),
                                                     ts.ooff.as<uint64_t>(), ts.olist.as<uint32_t>(), ts.oversize,
                                                     ts.gk.as<K>(), ts.gv.as<uint32_t>(), ukeys, vals));
    if (listed) {
      // (the gathered keys' sort may have used the counters)
      DBG_CUDA_TRY(cudaMemcpyAsync(nlisted, &listed, 4, cudaMemcpyHostToDevice, s));
      DBG_TRY(seg_sort_listed<K>(ctx, rk, rv, ukeys, vals, gr, vo, ts, fb.as<uint32_t>(), nlisted, listed));
    }
    DBG_LAUNCH(ctx, ST_LOCAL_SORT_NODES, 0.0,
               k_tile_heads<K><<<grid, RANK_BLOCK, 0, s>>>(ukeys, ts.bound.as<uint64_t>(), fb.as<uint32_t>(), listed,
                                                           ts.olist.as<uint32_t>(), ts.oversize,
                                                           heads.as<uint32_t>(), tcount.as<uint32_t>()));
    DBG_CUDA_TRY(cudaGetLastError());
    DBG_TRY(scan_tiles());
  }
  const uint32_t nv = c[CT_TOTAL], ne = I > 0 ? c[CT_ENDS] : (uint32_t)R;
  *V = nv;
  *ends = ne;
  if (ne != 2 * E) return DBG_OK;  // (the caller reports it)
  DBG_TRY(alloc_block(ctx, g->block[1],
                      {{&g->node_keys, nv * sizeof(K)},
                       {&g->row_ptr, ((uint64_t)nv + 1) * sizeof(uint64_t)},
                       {&g->src, E * sizeof(uint32_t)},
                       {&g->dst, E * sizeof(uint32_t)},
                       {&g->adj_edge, 2 * E * sizeof(uint32_t)},
                       {&g->adj_nbr, 2 * E * sizeof(uint32_t)},
                       {&g->adj_role, 2 * E},
                       {&g->adj_side, sides ? 2 * E : 0}}));
  if (!sides) g->adj_side.p = nullptr;
  int bshift = 10;
  while ((E + (1ull << bshift) - 1) >> bshift > 256) bshift++;
  DevBuf part, fill;
  DBG_TRY(alloc_tmp(ctx, part, 2 * E * 8));
  DBG_TRY(alloc_tmp(ctx, fill, 256 * 4));
  DBG_CUDA_TRY(cudaMemsetAsync(fill.p, 0, 256 * 4, s));
  auto kern = I > 0 ? k_node_tiles<K, true> : k_node_tiles<K, false>;
  DBG_LAUNCH(ctx, ST_NODE_IDS,
             4.0 * R + R / 8.0 + (double)nv * (2 * sizeof(K) + 8) + (double)ne * (g->adj_side.p ? 14 : 13),
             kern<<<(unsigned)tiles, RANK_BLOCK, 0, s>>>(
                 ts.bound.as<uint64_t>(), (uint32_t)tiles, ukeys, vals, heads.as<uint32_t>(), tcount.as<uint32_t>(),
                 hoff.as<uint64_t>(), eoff.as<uint64_t>(), g->node_keys.as<K>(), g->row_ptr.as<uint64_t>(),
                 g->adj_edge.as<uint32_t>(), g->adj_role.as<uint8_t>(), g->adj_side.as<uint8_t>(),
                 part.as<uint64_t>(), fill.as<uint32_t>(), bshift));
  DBG_LAUNCH(ctx, ST_NODE_IDS, 2.0 * E * (8 + 4),
             k_scatter_ends<<<grid_for(2 * E, 256 * 16), 256, 0, s>>>(part.as<uint64_t>(), 2 * E,
                                                                      g->src.as<uint32_t>(), g->dst.as<uint32_t>()));
  DBG_CUDA_TRY(cudaGetLastError());
  return DBG_OK;
}

// Node multiplicities: the k-mers of the reads (each read of length L >= k
// holds L - k + 1), emitted, sorted and counted like STEP-2's edge keys.  The
// distinct canonical k-mers of the reads of length >= k are exactly the
// nodes, in the same ascending order, so counts[i] belongs to node i; *Vk =
// their number, which the caller checks against |V|.
template <class K>
dbg_status count_node_kmers(dbg_ctx *ctx, const DevBuf &packed, const DevBuf &base_off, const uint32_t *d_lengths,
                            uint64_t n, uint64_t N, uint32_t k, unsigned long long *d_hist,
                            uint64_t *d_digit_base, DevBuf &counts, uint64_t *Vk) {
  cudaStream_t s = ctx->stream;
  *Vk = 0;
  if (n == 0) return DBG_OK;
  // the k-mers number at most N + n (N edge instances, one more k-mer per
  // read); the offsets' scan keeps 32-bit totals
  if (N + n > 0xffffffffull) {
    set_error("%llu edge instances and %llu reads: too many k-mers to count in one build",
              (unsigned long long)N, (unsigned long long)n);
    return DBG_EOVERFLOW;
  }
  DevBuf per, koff;
  DBG_TRY(alloc_tmp(ctx, per, n * sizeof(uint32_t)));
  DBG_TRY(alloc_tmp(ctx, koff, (n + 1) * sizeof(uint64_t)));
  DBG_LAUNCH(ctx, ST_NODE_MULT, 8.0 * n,
             k_kmer_counts<<<grid_for(n, 256), 256, 0, s>>>(d_lengths, n, k, per.as<uint32_t>()));
  uint32_t low32 = 0;
  DBG_TRY(scan_u32(ctx, per.as<uint32_t>(), n, koff.as<uint64_t>(), &low32, ST_NODE_MULT));
  uint64_t M = 0;
  DBG_TRY(read_small(ctx, koff.as<uint64_t>() + n, sizeof(uint64_t), &M));
  if (M == 0) return DBG_OK;
  const int kbits = 2 * (int)k;
  const SortPlan<K> plan = plan_sort<K>(ctx, M, kbits, ctx->partition_first);
  DevBuf ka, kb, headpos;
  DBG_TRY(alloc_tmp(ctx, ka, M * sizeof(K) + MSD_PAD));
  DBG_TRY(alloc_tmp(ctx, kb, M * sizeof(K) + MSD_PAD));
  DBG_CUDA_TRY(cudaMemsetAsync(d_hist, 0, MAX_PASSES * RADIX * sizeof(unsigned long long), s));
  const DigitSpec digits = plan.digits();
  // emitting with k - 1 gives windows of k bases at the k-mer offsets
  DBG_LAUNCH(ctx, ST_NODE_MULT, 8.0 * n + (double)M * sizeof(K),
             (digits.wide ? k_emit<K, true> : k_emit<K, false>)<<<(unsigned)std::min<uint64_t>(grid_for(n, EMIT_BLOCK / 32), 152ull * 64), EMIT_BLOCK, 0, s>>>(
                 packed.as<uint64_t>(), base_off.as<uint64_t>(), koff.as<uint64_t>(), n, k - 1, ka.as<K>(),
                 digits, d_hist, nullptr, nullptr));
  DBG_CUDA_TRY(cudaGetLastError());
  K *kp = ka.as<K>(), *alt = kb.as<K>();
  uint32_t *vn = nullptr, *van = nullptr;
  uint64_t D = 0;
  if (plan.local()) {
    DBG_TRY(sort_count_keys<K>(ctx, &kp, &alt, M, plan, d_hist, d_digit_base, &counts, nullptr, &D));
  } else {
    DBG_TRY(alloc_tmp(ctx, headpos, (M + 1) * sizeof(uint32_t)));
    DBG_TRY((radix_sort<K, false>(ctx, &kp, &alt, &vn, &van, M, kbits, d_hist, d_digit_base)));
    DBG_TRY(run_length_reduce<K>(ctx, kp, M, alt, headpos.as<uint32_t>(), &D));
    DBG_TRY(alloc_buf(ctx, counts, std::max<uint64_t>(1, D) * sizeof(uint32_t)));
    DBG_LAUNCH(ctx, ST_NODE_MULT, 8.0 * D,
               k_counts_from_heads<<<grid_for(D, 256), 256, 0, s>>>(headpos.as<uint32_t>(), D,
                                                                   counts.as<uint32_t>()));
  }
  DBG_CUDA_TRY(cudaGetLastError());
  DBG_TRY(check_device_error(ctx));
  *Vk = D;
  return DBG_OK;
}

// Distinct reads per node (the roadmap counts): every k-mer of the reads
// with its read index, stably sorted by key (the records of one key keep
// their read order, which is ascending), then per key the number of records
// that start its run or follow a record of another read.  As for the
// multiplicities, the distinct keys are exactly the nodes, in node order.
template <class K>
dbg_status count_node_reads(dbg_ctx *ctx, const DevBuf &packed, const DevBuf &base_off, const uint32_t *d_lengths,
                            uint64_t n, uint64_t N, uint32_t k, unsigned long long *d_hist,
                            uint64_t *d_digit_base, DevBuf &counts, uint64_t *Vk) {
  cudaStream_t s = ctx->stream;
  *Vk = 0;
  if (n == 0) return DBG_OK;
  if (N + n > 0xffffffffull) {
    set_error("%llu edge instances and %llu reads: too many k-mers to count in one build",
              (unsigned long long)N, (unsigned long long)n);
    return DBG_EOVERFLOW;
  }
  DevBuf per, koff;
  DBG_TRY(alloc_tmp(ctx, per, n * sizeof(uint32_t)));
  DBG_TRY(alloc_tmp(ctx, koff, (n + 1) * sizeof(uint64_t)));
  DBG_LAUNCH(ctx, ST_NODE_MULT, 8.0 * n,
             k_kmer_counts<<<grid_for(n, 256), 256, 0, s>>>(d_lengths, n, k, per.as<uint32_t>()));
  uint32_t low32 = 0;
  DBG_TRY(scan_u32(ctx, per.as<uint32_t>(), n, koff.as<uint64_t>(), &low32, ST_NODE_MULT));
  uint64_t M = 0;
  DBG_TRY(read_small(ctx, koff.as<uint64_t>() + n, sizeof(uint64_t), &M));
  if (M == 0) return DBG_OK;
  per.release();
  const int kbits = 2 * (int)k;
  const SortPlan<K> plan = plan_records<K>(ctx, M, kbits, false);
  DevBuf ka, kb, va, vb;
  DBG_TRY(alloc_tmp(ctx, ka, M * sizeof(K) + MSD_PAD));
  DBG_TRY(alloc_tmp(ctx, kb, M * sizeof(K) + MSD_PAD));
  DBG_TRY(alloc_tmp(ctx, va, M * sizeof(uint32_t) + MSD_PAD));
  DBG_TRY(alloc_tmp(ctx, vb, M * sizeof(uint32_t) + MSD_PAD));
  DBG_CUDA_TRY(cudaMemsetAsync(d_hist, 0, MAX_PASSES * RADIX * sizeof(unsigned long long), s));
  const DigitSpec digits = plan.digits();
  // windows of k bases at the k-mer offsets, each with its read index
  DBG_LAUNCH(ctx, ST_NODE_MULT, 8.0 * n + (double)M * (sizeof(K) + 4),
             (digits.wide ? k_emit<K, true> : k_emit<K, false>)<<<(unsigned)std::min<uint64_t>(grid_for(n, EMIT_BLOCK / 32), 152ull * 64), EMIT_BLOCK, 0, s>>>(
                 packed.as<uint64_t>(), base_off.as<uint64_t>(), koff.as<uint64_t>(), n, k - 1, ka.as<K>(),
                 digits, d_hist, nullptr, va.as<uint32_t>()));
  DBG_CUDA_TRY(cudaGetLastError());
  koff.release();
  K *kp = ka.as<K>(), *kalt = kb.as<K>();
  uint32_t *vp = va.as<uint32_t>(), *valt = vb.as<uint32_t>();
  DBG_TRY(sort_records<K>(ctx, &kp, &kalt, &vp, &valt, M, plan, read_order(n), d_hist, d_digit_base));
  // flags into the free payload buffer, their scan, the key runs
  DBG_LAUNCH(ctx, ST_NODE_MULT, (double)M * (2 * sizeof(K) + 12),
             k_read_change_flags<K><<<grid_for(M, 256 * 8), 256, 0, s>>>(kp, vp, M, valt));
  DevBuf F, headpos;
  DBG_TRY(alloc_tmp(ctx, F, (M + 1) * sizeof(uint64_t)));
  uint32_t low = 0;
  DBG_TRY(scan_u32(ctx, valt, M, F.as<uint64_t>(), &low, ST_NODE_MULT));
  DBG_TRY(alloc_tmp(ctx, headpos, (M + 1) * sizeof(uint32_t)));
  uint64_t D = 0;
  DBG_TRY(run_length_reduce<K>(ctx, kp, M, kalt, headpos.as<uint32_t>(), &D));
  DBG_TRY(alloc_buf(ctx, counts, std::max<uint64_t>(1, D) * sizeof(uint32_t)));
  DBG_LAUNCH(ctx, ST_NODE_MULT, 12.0 * D,
             k_counts_between<<<grid_for(D, 256), 256, 0, s>>>(headpos.as<uint32_t>(), F.as<uint64_t>(), D,
                                                               counts.as<uint32_t>()));
  DBG_CUDA_TRY(cudaGetLastError());
  DBG_TRY(check_device_error(ctx));
  *Vk = D;
  return DBG_OK;
}

template <class K>
dbg_status build_graph_impl(dbg_ctx *ctx, const BuildInput &in, dbg_graph *g) {
  cudaStream_t s = ctx->stream;
  const uint32_t k = in.k;
  const uint64_t n = in.n;
  g->k = k;
  g->key_words = sizeof(K) / 8;

  // ---- per-read offsets (exclusive scans of L and max(0, L - k)) ----
  DevBuf base_off, edge_off, tile_sums, small;
  const uint64_t off_tiles = (n + OFF_TILE - 1) / OFF_TILE;
  DBG_TRY(alloc_tmp(ctx, base_off, (n + 1) * sizeof(uint64_t)));
  DBG_TRY(alloc_tmp(ctx, edge_off, (n + 1) * sizeof(uint64_t)));
  DBG_TRY(alloc_tmp(ctx, tile_sums, std::max<uint64_t>(1, off_tiles) * sizeof(Sum3)));
  DBG_TRY(alloc_tmp(ctx, small, 64 * sizeof(uint64_t) + (MAX_PASSES * RADIX) * 16));
  uint64_t *d_totals = small.as<uint64_t>();
  unsigned long long *d_hist = reinterpret_cast<unsigned long long *>(d_totals + 64);
  uint64_t *d_digit_base = reinterpret_cast<uint64_t *>(d_hist + MAX_PASSES * RADIX);
  if (n > 0) {
    DBG_LAUNCH(ctx, ST_OFFSETS, 4.0 * n,
               k_read_tile_sums<<<(unsigned)off_tiles, OFF_BLOCK, 0, s>>>(in.d_lengths, n, k, tile_sums.as<Sum3>()));
  }
  {
    DBG_LAUNCH(ctx, ST_OFFSETS, 0.0,
               k_scan_tile_sums<<<1, 1024, 0, s>>>(tile_sums.as<Sum3>(), (uint32_t)off_tiles, d_totals,
                                      base_off.as<uint64_t>(), edge_off.as<uint64_t>(), n));
  }
  if (n > 0) {
    DBG_LAUNCH(ctx, ST_OFFSETS, 20.0 * n,
               k_read_offsets<<<(unsigned)off_tiles, OFF_BLOCK, 0, s>>>(in.d_lengths, n, k, tile_sums.as<Sum3>(),
                                                             base_off.as<uint64_t>(), edge_off.as<uint64_t>()));
  }
  DBG_CUDA_TRY(cudaGetLastError());
  uint64_t totals[3];
  DBG_TRY(read_small(ctx, d_totals, sizeof(totals), totals));
  const uint64_t total_bases = totals[0], N = totals[1], I = totals[2];
  tile_sums.release();
  g->num_instances = N;
  if (N > 0xffffffffull) {
    set_error("%llu edge instances exceed one in-memory build (2^32 - 1)", (unsigned long long)N);
    return DBG_EOVERFLOW;
  }

  // ---- K2 set-up: key buffers and histograms come first, so that host
  // reads can be emitted chunk by chunk as they are packed ----
  const int kbits = 2 * ((int)k + 1);
  DevBuf keys_a, keys_b, headpos, uniq;
  EdgeTiles edge_tiles;  // the distinct keys in uniq, unless its run heads are in headpos
  uint64_t E = 0;
  const SortPlan<K> plan = plan_sort<K>(ctx, N, kbits, ctx->partition_first);
  if (N > 0) {
    DBG_TRY(alloc_tmp(ctx, keys_a, N * sizeof(K) + MSD_PAD));
    DBG_TRY(alloc_tmp(ctx, keys_b, N * sizeof(K) + MSD_PAD));
    DBG_CUDA_TRY(cudaMemsetAsync(d_hist, 0, MAX_PASSES * RADIX * sizeof(unsigned long long), s));
  }
  DevBuf packed;
  const uint64_t nwords = (total_bases + 31) / 32;
  // K2 emit over the keys [krange[0], krange[1]) (all of them: nullptr)
  const DigitSpec digits = plan.digits();
  auto emit = [&](const uint64_t *krange, double bytes) -> dbg_status {
    DBG_LAUNCH(ctx, ST_EMIT, bytes,
               (digits.wide ? k_emit<K, true> : k_emit<K, false>)<<<(unsigned)std::min<uint64_t>(grid_for(n, EMIT_BLOCK / 32), 152ull * 64), EMIT_BLOCK, 0,
                           s>>>(packed.as<uint64_t>(), base_off.as<uint64_t>(), edge_off.as<uint64_t>(), n, k,
                                keys_a.as<K>(), digits, d_hist, krange, nullptr));
    DBG_CUDA_TRY(cudaGetLastError());
    return DBG_OK;
  };

  // ---- K1 pack (+ K2 emit) ----
  DBG_TRY(alloc_tmp(ctx, packed, (nwords + 3) * sizeof(uint64_t)));
  DBG_CUDA_TRY(cudaMemsetAsync(packed.as<uint64_t>() + nwords, 0, 3 * sizeof(uint64_t), s));
  bool emitted = false;
  if (nwords > 0 && !in.h_reads) {
    DBG_LAUNCH(ctx, ST_PACK, (double)total_bases + 8.0 * nwords,
               k_pack<<<grid_for(nwords, 256), 256, 0, s>>>(in.reads, total_bases, packed.as<uint64_t>(), nwords,
                                                 ctx->d_err));
  } else if (nwords > 0) {
    // host reads: chunks are copied on a stream of their own into two
    // staging buffers in turn while the build's stream packs the previous
    // chunk and emits the reads that end in the chunks packed so far
    const uint64_t chunk = 256ull << 20;  // bases per copy (a multiple of 32)
    const uint32_t chunks = (uint32_t)((total_bases + chunk - 1) / chunk);
    DBG_TRY(ensure_copy_stream(ctx));
    cudaStream_t cs = ctx->copy_stream;
    DevBuf stage[2], kbound;
    const uint64_t slen = std::min(chunk, total_bases);
    DBG_TRY(alloc_buf(ctx, stage[0], slen));
    if (chunks > 1) DBG_TRY(alloc_buf(ctx, stage[1], slen));
    DBG_TRY(alloc_tmp(ctx, kbound, (chunks + 1) * sizeof(uint64_t)));
    if (N > 0)
      DBG_LAUNCH(ctx, ST_EMIT, 0.0,
                 k_chunk_key_bounds<<<grid_for(chunks + 1, 64), 64, 0, s>>>(
                     base_off.as<uint64_t>(), edge_off.as<uint64_t>(), n, chunk, chunks, kbound.as<uint64_t>()));
    EventSet ev;
    DBG_TRY(ev.create(2 * chunks + 1));
    cudaEvent_t ready = ev.e[2 * chunks];  // the stage buffers exist on the build's stream
    DBG_CUDA_TRY(cudaEventRecord(ready, s));
    DBG_CUDA_TRY(cudaStreamWaitEvent(cs, ready, 0));
    for (uint32_t c = 0; c < chunks; c++) {
      const uint64_t off = (uint64_t)c * chunk, len = std::min(chunk, total_bases - off);
      DevBuf &st = stage[c & 1];
      if (c >= 2) DBG_CUDA_TRY(cudaStreamWaitEvent(cs, ev.e[2 * (c - 2) + 1], 0));  // packed c - 2
      DBG_CUDA_TRY(cudaMemcpyAsync(st.p, in.reads + off, len, cudaMemcpyHostToDevice, cs));
      DBG_CUDA_TRY(cudaEventRecord(ev.e[2 * c], cs));
      DBG_CUDA_TRY(cudaStreamWaitEvent(s, ev.e[2 * c], 0));
      DBG_LAUNCH(ctx, ST_PACK, (double)len * 1.25,
                 k_pack_at<<<grid_for((len + 31) / 32, 256), 256, 0, s>>>(st.as<uint8_t>(), len,
                                                                        packed.as<uint64_t>(), off / 32, ctx->d_err));
      DBG_CUDA_TRY(cudaEventRecord(ev.e[2 * c + 1], s));
      if (N > 0) DBG_TRY(emit(kbound.as<uint64_t>() + c, (double)len / 4.0 + (double)N * sizeof(K) / chunks));
    }
    emitted = true;
  }

  // ---- K2 emit + digit histograms, K3 sort, K4 run-length reduce ----
  if (N > 0) {
    if (!emitted) DBG_TRY(emit(nullptr, 8.0 * nwords + 16.0 * n + (double)N * sizeof(K)));
    DBG_CUDA_TRY(cudaGetLastError());
    K *kp = keys_a.as<K>(), *alt = keys_b.as<K>();
    uint32_t *vn = nullptr, *van = nullptr;
    if (plan.local()) {
      // high digits globally, then the local sort with the run-length
      // reduce: distinct keys into alt, by tiles
      // (its last read-back brought the error word)
      DBG_TRY(sort_count_keys<K>(ctx, &kp, &alt, N, plan, d_hist, d_digit_base, nullptr, &edge_tiles, &E));
    } else {
      // every digit globally, then the run-length reduce
      DBG_TRY(alloc_tmp(ctx, headpos, (N + 1) * sizeof(uint32_t)));
      DBG_TRY((radix_sort<K, false>(ctx, &kp, &alt, &vn, &van, N, kbits, d_hist, d_digit_base)));
      DBG_TRY(run_length_reduce<K>(ctx, kp, N, alt, headpos.as<uint32_t>(), &E));
      DBG_TRY(check_device_error(ctx));
    }
    // keep the buffer holding the unique keys (alt); the sorted keys are done
    if (alt == keys_b.as<K>()) { uniq = std::move(keys_b); keys_a.release(); }
    else { uniq = std::move(keys_a); keys_b.release(); }
  }
  if (E >= 0x80000000ull) {
    set_error("%llu unique edges exceed one in-memory build (2^31 - 1)", (unsigned long long)E);
    return DBG_EOVERFLOW;
  }
  g->num_edges = E;

  // ---- node multiplicities (optional), while the packed reads are here ----
  DevBuf node_counts, read_counts;
  uint64_t Vk = 0, Vr = 0;
  if ((ctx->node_mult || ctx->node_reads) && E > 0 && !headpos.p) {
    // the counts' sorts are the fullest point then: 4 bytes per edge beside
    // them instead of 4 per instance
    DevBuf dense;
    DBG_TRY(alloc_tmp(ctx, dense, E * sizeof(uint32_t)));
    DBG_LAUNCH(ctx, ST_NODE_MULT, 8.0 * E,
               k_mult_compact<<<(unsigned)std::min<uint64_t>(edge_tiles.tiles, 152ull * 16), 256, 0, s>>>(
                   edge_tiles.bound.as<uint64_t>(), edge_tiles.tcount.as<uint32_t>(), edge_tiles.toff.as<uint64_t>(),
                   edge_tiles.tiles, edge_tiles.mult.as<uint32_t>(), dense.as<uint32_t>()));
    DBG_CUDA_TRY(cudaGetLastError());
    edge_tiles.mult = std::move(dense);
    edge_tiles.dense = true;
  }
  if (ctx->node_mult)
    DBG_TRY(count_node_kmers<K>(ctx, packed, base_off, in.d_lengths, n, N, k, d_hist, d_digit_base, node_counts,
                                &Vk));
  if (ctx->node_reads)
    DBG_TRY(count_node_reads<K>(ctx, packed, base_off, in.d_lengths, n, N, k, d_hist, d_digit_base, read_counts,
                                &Vr));

  // ---- K5 edge ends + records of reads of length k ----
  const uint64_t R = 2 * E + I;
  const int nbits = 2 * (int)k;
  DBG_TRY(alloc_block(ctx, g->block[0],
                      {{&g->edge_keys, E * sizeof(K)}, {&g->mult, E * sizeof(uint32_t)}, {&g->orient, E}}));
  DevBuf rk_a, rk_b, rv_a, rv_b;
  DBG_TRY(alloc_tmp(ctx, rk_a, R * sizeof(K) + MSD_PAD));
  DBG_TRY(alloc_tmp(ctx, rv_a, R * sizeof(uint32_t) + MSD_PAD));
  DBG_CUDA_TRY(cudaMemsetAsync(d_hist, 0, MAX_PASSES * RADIX * sizeof(unsigned long long), s));
  const SortPlan<K> rplan = plan_records<K>(ctx, R, nbits, true);
  const DigitSpec nspec = rplan.digits();
  // below 2^29 edges the payloads carry both sides of each edge end, and
  // the node IDs pass stores them per adjacency slot (for the compaction)
  const bool sides = E > 0 && E < (1ull << 29);
  if (E > 0) {
    const EdgeOut<K> out{g->edge_keys.as<K>(), g->mult.as<uint32_t>(), g->orient.as<uint8_t>(),
                         rk_a.as<K>(),         rv_a.as<uint32_t>(),    sides};
    const double bytes = (double)E * (4 * sizeof(K) + 4 + 4 + 1 + 8);
    if (headpos.p)
      DBG_LAUNCH(ctx, ST_ENDPOINTS, bytes,
                 k_endpoints<K><<<grid_for(E, EMIT_TILE), EMIT_BLOCK, 0, s>>>(uniq.as<K>(), headpos.as<uint32_t>(), E,
                                                                             k, out, nspec, d_hist));
    else
    {
      const uint64_t per = std::min<uint64_t>(4, edge_tiles.tiles / (152 * 8) + 1);
      DBG_LAUNCH(ctx, ST_ENDPOINTS, bytes,
                 k_endpoints_tiles<K><<<(unsigned)((edge_tiles.tiles + per - 1) / per), EMIT_BLOCK, 0, s>>>(
                     edge_tiles.bound.as<uint64_t>(), edge_tiles.tcount.as<uint32_t>(),
                     edge_tiles.toff.as<uint64_t>(), (uint32_t)edge_tiles.tiles, (uint32_t)per, uniq.as<K>(),
                     edge_tiles.mult.as<uint32_t>(), edge_tiles.dense, k, out, nspec, d_hist));
    }
  }
  if (I > 0) {
    DBG_CUDA_TRY(cudaMemsetAsync(ctx->d_counters + 2, 0, sizeof(uint32_t), s));
    DBG_LAUNCH(ctx, ST_ENDPOINTS, (double)n * 4 + (double)I * (sizeof(K) + 4),
               k_isolated<K><<<grid_for(n, 256), 256, 0, s>>>(packed.as<uint64_t>(), base_off.as<uint64_t>(),
                                                   in.d_lengths, n, k, rk_a.as<K>() + 2 * E,
                                                   rv_a.as<uint32_t>() + 2 * E, ctx->d_counters + 2, nspec,
                                                   d_hist));
  }
  DBG_CUDA_TRY(cudaGetLastError());
  uniq.release();
  headpos.release();
  edge_tiles.release();
  packed.release();
  base_off.release();
  edge_off.release();
  DBG_TRY(alloc_tmp(ctx, rk_b, R * sizeof(K) + MSD_PAD));
  DBG_TRY(alloc_tmp(ctx, rv_b, R * sizeof(uint32_t) + MSD_PAD));

  // ---- STEP-3 sort of the node records (payload order kept), K6 node IDs +
  // adjacency rows, K7 neighbours ----
  K *rk = rk_a.as<K>(), *rk_alt = rk_b.as<K>();
  uint32_t *rv = rv_a.as<uint32_t>(), *rv_alt = rv_b.as<uint32_t>();
  const ValOrder vo = edge_end_order(E, sides, I > 0);
  DevBuf row_tmp;
  auto alloc_adjacency = [&]() -> dbg_status {
    DBG_TRY(alloc_buf(ctx, g->src, std::max<uint64_t>(1, E) * sizeof(uint32_t)));
    DBG_TRY(alloc_buf(ctx, g->dst, std::max<uint64_t>(1, E) * sizeof(uint32_t)));
    DBG_TRY(alloc_buf(ctx, g->adj_edge, std::max<uint64_t>(1, 2 * E) * sizeof(uint32_t)));
    DBG_TRY(alloc_buf(ctx, g->adj_role, std::max<uint64_t>(1, 2 * E)));
    DBG_TRY(alloc_buf(ctx, g->adj_nbr, std::max<uint64_t>(1, 2 * E) * sizeof(uint32_t)));
    if (sides) DBG_TRY(alloc_buf(ctx, g->adj_side, 2 * E));
    return DBG_OK;
  };
  uint64_t V = 0;
  // The local pass hands the node-ID pass the tiles' distinct keys and head
  // bits instead of sorted keys.
  bool fused = false;
  if (E > 0 && rplan.local() && ctx->seg_rank) {
    Groups gr;
    TileSet ts;
    ValOrder fvo = vo;
    uint64_t ends = 0;
    DBG_TRY(sort_records_global<K>(ctx, &rk, &rk_alt, &rv, &rv_alt, R, rplan, fvo, d_hist, d_digit_base, gr, ts));
    DBG_TRY(rank_and_assign<K>(ctx, rk, rv, rk_alt, rv_alt, R, E, I, nbits, gr, fvo, ts, g, sides,
                               edge_tiles.uneven, &fused, &V, &ends));
    if (!fused) {
      DBG_TRY(seg_sort_records<K>(ctx, rk, rv, rk_alt, rv_alt, R, gr, fvo, ts));
      std::swap(rk, rk_alt);
      std::swap(rv, rv_alt);
    } else if (ends != 2 * E) {
      set_error("adjacency holds %llu edge ends, expected %llu", (unsigned long long)ends,
                (unsigned long long)(2 * E));
      return DBG_EINTERNAL;
    }
  } else {
    DBG_TRY(sort_records<K>(ctx, &rk, &rk_alt, &rv, &rv_alt, R, rplan, vo, d_hist, d_digit_base));
  }
  if (!fused) {
    DBG_TRY(alloc_tmp(ctx, row_tmp, (R + 1) * sizeof(uint64_t)));
    DBG_TRY(alloc_adjacency());
  }
  if (R > 0 && !fused) {
    // node keys go to the free record buffer first (|V| is known only after)
    uint64_t ends = 0;
    DBG_TRY(assign_node_ids<K>(ctx, rk, rv, R, rk_alt, row_tmp.as<uint64_t>(), g, 0u, 0ull, &V, &ends, E,
                               sides ? g->adj_side.as<uint8_t>() : nullptr));
    DBG_TRY(check_device_error(ctx));
    if (ends != 2 * E) {
      set_error("adjacency holds %llu edge ends, expected %llu", (unsigned long long)ends,
                (unsigned long long)(2 * E));
      return DBG_EINTERNAL;
    }
  }
  g->num_nodes = V;
  if (ctx->node_mult) {
    if (Vk != V) {
      set_error("node multiplicities: %llu distinct k-mers for %llu nodes", (unsigned long long)Vk,
                (unsigned long long)V);
      return DBG_EINTERNAL;
    }
    if (V == 0) DBG_TRY(alloc_buf(ctx, node_counts, sizeof(uint32_t)));
    g->node_mult = std::move(node_counts);
  }
  if (ctx->node_reads) {
    if (Vr != V) {
      set_error("node read counts: %llu distinct k-mers for %llu nodes", (unsigned long long)Vr,
                (unsigned long long)V);
      return DBG_EINTERNAL;
    }
    if (V == 0) DBG_TRY(alloc_buf(ctx, read_counts, sizeof(uint32_t)));
    g->node_reads = std::move(read_counts);
  }
  if (!fused) {
    DBG_TRY(alloc_buf(ctx, g->node_keys, std::max<uint64_t>(1, V) * sizeof(K)));
    DBG_TRY(alloc_buf(ctx, g->row_ptr, (V + 1) * sizeof(uint64_t)));
  }
  if (fused) {
    // written in place
  } else if (V > 0) {
    Span sp(ctx, ST_COPIES, 2.0 * V * (sizeof(K) + 8), 0);
    DBG_CUDA_TRY(cudaMemcpyAsync(g->node_keys.p, rk_alt, V * sizeof(K), cudaMemcpyDeviceToDevice, s));
    DBG_CUDA_TRY(cudaMemcpyAsync(g->row_ptr.p, row_tmp.p, (V + 1) * sizeof(uint64_t), cudaMemcpyDeviceToDevice, s));
  } else {
    DBG_CUDA_TRY(cudaMemsetAsync(g->row_ptr.p, 0, sizeof(uint64_t), s));
  }
  if (E > 0) {
    DBG_LAUNCH(ctx, ST_ADJACENCY, 2.0 * E * (4 + 1 + 4 + 4),
               k_adj_nbr<<<grid_for(2 * E, 256 * 8), 256, 0, s>>>(g->adj_edge.as<uint32_t>(), g->adj_role.as<uint8_t>(),
                                                     g->src.as<uint32_t>(), g->dst.as<uint32_t>(), 2 * E,
                                                     g->adj_nbr.as<uint32_t>()));
    DBG_CUDA_TRY(cudaGetLastError());
  }
  return check_device_error(ctx);  // waits for the stream
}

}  // namespace dbg

namespace dbg {

// ---------------------------------------------------------------------------
// Autotuner: times one digit pass of every variant of a key kind on n
// synthetic keys (a counter-based hash of the index, so all digits vary) and
// keeps the fastest.  ms_out[v] receives each variant's pass time.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint64_t tune_hash(uint64_t x) {
  x += 0x9e3779b97f4a7c15ull;
  x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
  x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
  return x ^ (x >> 31);
}

template <class K>
__global__ void k_tune_fill(K *keys, uint32_t *vals, uint64_t n) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    K k;
    if constexpr (sizeof(K) == 8) {
      k = tune_hash(i);
    } else {
      k = Key128{tune_hash(2 * i), tune_hash(2 * i + 1)};
    }
    keys[i] = k;
    if (vals) vals[i] = (uint32_t)i;
  }
}

// digit histogram of one 8-bit digit position of arbitrary keys
template <class K>
__global__ void k_tune_hist(const K *keys, uint64_t n, int shift, unsigned long long *hist) {
  __shared__ uint32_t h[RADIX];
  for (int i = threadIdx.x; i < RADIX; i += blockDim.x) h[i] = 0;
  __syncthreads();
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
    atomicAdd(&h[KeyOps<K>::digit(keys[i], shift, RADIX_BITS)], 1u);
  __syncthreads();
  for (int i = threadIdx.x; i < RADIX; i += blockDim.x)
    if (h[i]) atomicAdd(hist + i, (unsigned long long)h[i]);
}

template <class K, bool V>
dbg_status autotune_kind(dbg_ctx *ctx, uint64_t n, double *ms_out) {
  cudaStream_t s = ctx->stream;
  int count = 0;
  const SortVariant *t = SortKind<K, V>::table(&count);
  DevBuf ka, kb, va, vb, small;
  DBG_TRY(alloc_tmp(ctx, ka, n * sizeof(K)));
  DBG_TRY(alloc_tmp(ctx, kb, n * sizeof(K)));
  if (V) {
    DBG_TRY(alloc_tmp(ctx, va, n * 4));
    DBG_TRY(alloc_tmp(ctx, vb, n * 4));
  }
  DBG_TRY(alloc_tmp(ctx, small, RADIX * 16));
  unsigned long long *hist = small.as<unsigned long long>();
  uint64_t *dbase = reinterpret_cast<uint64_t *>(hist + RADIX);
  k_tune_fill<K><<<1024, 256, 0, s>>>(ka.as<K>(), V ? va.as<uint32_t>() : nullptr, n);
  DBG_CUDA_TRY(cudaMemsetAsync(hist, 0, RADIX * 8, s));
  k_tune_hist<K><<<1024, 256, 0, s>>>(ka.as<K>(), n, 8, hist);
  k_digit_base<<<1, RADIX, 0, s>>>(hist, dbase);
  int min_tile = t[0].tile;
  for (int v = 0; v < count; v++) min_tile = std::min(min_tile, t[v].tile);
  DBG_TRY(ensure_status(ctx, ((n + min_tile - 1) / min_tile) * RADIX));
  cudaEvent_t e0, e1;
  DBG_CUDA_TRY(cudaEventCreate(&e0));
  DBG_CUDA_TRY(cudaEventCreate(&e1));
  int best = 0;
  double best_ms = 1e30;
  for (int v = 0; v < count; v++) {
    float total = 0.f;
    for (int rep = 0; rep < 4; rep++) {
      uint32_t epoch;
      DBG_TRY(next_epoch(ctx, &epoch));
      DBG_CUDA_TRY(cudaMemsetAsync(ctx->d_counters, 0, sizeof(uint32_t), s));
      cudaEventRecord(e0, s);
      t[v].launch(ctx, ka.p, kb.p, V ? va.as<uint32_t>() : nullptr, V ? vb.as<uint32_t>() : nullptr, n, 8, dbase,
                  epoch);
      cudaEventRecord(e1, s);
      DBG_CUDA_TRY(cudaEventSynchronize(e1));
      float ms = 0.f;
      cudaEventElapsedTime(&ms, e0, e1);
      if (rep > 0) total += ms;  // the first launch is a warm-up
    }
    const double ms = total / 3.0;
    if (ms_out) ms_out[v] = ms;
    if (ms < best_ms) {
      best_ms = ms;
      best = v;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  DBG_CUDA_TRY(cudaGetLastError());
  DBG_TRY(check_device_error(ctx));
  ctx->sort_variant[SortKind<K, V>::kind] = best;
  return DBG_OK;
}

template <class K, bool V>
const char *variant_name(uint32_t v, uint32_t *count) {
  int c = 0;
  const SortVariant *t = SortKind<K, V>::table(&c);
  *count = (uint32_t)c;
  return v < (uint32_t)c ? t[v].name : nullptr;
}

}  // namespace dbg

namespace dbg {

// ---------------------------------------------------------------------------
// The bucket path (dbg_build_bucketed): Section 5's out-of-core
// construction with key-range partitioning in place of the external merge.
// ---------------------------------------------------------------------------
// Cuts the prefix bins into consecutive ranges of at most `cap` items (a
// single bin above cap gets a range of its own).
inline std::vector<std::pair<uint32_t, uint32_t>> plan_ranges(const uint64_t *hist, uint64_t cap,
                                                              std::vector<uint64_t> *sizes) {
  std::vector<std::pair<uint32_t, uint32_t>> out;
  uint32_t lo = 0;
  uint64_t acc = 0;
  for (uint32_t b = 0; b < (uint32_t)PREFIX_BINS; b++) {
    if (acc > 0 && acc + hist[b] > cap) {
      out.emplace_back(lo, b);
      sizes->push_back(acc);
      lo = b;
      acc = 0;
    }
    acc += hist[b];
  }
  out.emplace_back(lo, (uint32_t)PREFIX_BINS);
  sizes->push_back(acc);
  return out;
}

// The keys of prefixes [lo, hi) among keys of key_bits bits: the first of
// them, the bits of their offsets from it, and how much denser those are than
// if they filled all values of as many bits.
template <class K>
struct KeyRange {
  K base;
  int bits;
  double density;
};
template <class K>
KeyRange<K> key_range(uint32_t lo, uint32_t hi, int key_bits) {
  hi = std::min(hi, 1u << std::min(PREFIX_BITS, key_bits));  // (short keys have fewer prefixes than there are bins)
  if (hi <= lo) hi = lo + 1;                                 // (of an empty range)
  const int low = std::max(0, key_bits - PREFIX_BITS), top = bit_length(hi - lo - 1);
  return KeyRange<K>{key_from(lo, low, K{}), std::max(1, low + top), std::ldexp(1.0, top) / (hi - lo)};
}

template <class K>
dbg_status concat_chunks(dbg_ctx *ctx, std::vector<DevBuf> &chunks, const std::vector<uint64_t> &counts,
                         size_t elem, void *dst) {
  uint64_t at = 0;
  for (size_t i = 0; i < chunks.size(); i++) {
    if (counts[i])
      DBG_CUDA_TRY(cudaMemcpyAsync(static_cast<char *>(dst) + at * elem, chunks[i].p, counts[i] * elem,
                                   cudaMemcpyDeviceToDevice, ctx->stream));
    at += counts[i];
    chunks[i].release();
  }
  return DBG_OK;
}

template <class K>
dbg_status build_bucketed_impl(dbg_ctx *ctx, const BucketInput &in, uint64_t budget, dbg_graph *g,
                               uint32_t *n_edge_buckets, uint32_t *n_node_buckets) {
  cudaStream_t s = ctx->stream;
  const uint32_t k = in.k;
  const uint64_t n = in.n;
  const int m = (int)k + 1;
  const uint64_t w = sizeof(K);
  g->k = k;
  g->key_words = sizeof(K) / 8;
  DBG_CUDA_TRY(cudaStreamSynchronize(s));  // the pinned mirror is free

  // ---- per-read offsets ----
  DevBuf base_off, edge_off, tile_sums, small;
  const uint64_t off_tiles = (n + OFF_TILE - 1) / OFF_TILE;
  DBG_TRY(alloc_tmp(ctx, base_off, (n + 1) * 8));
  DBG_TRY(alloc_tmp(ctx, edge_off, (n + 1) * 8));
  DBG_TRY(alloc_tmp(ctx, tile_sums, std::max<uint64_t>(1, off_tiles) * sizeof(Sum3)));
  DBG_TRY(alloc_tmp(ctx, small, 64 * 8 + MAX_PASSES * RADIX * 16 + PREFIX_BINS * 8));
  uint64_t *d_totals = small.as<uint64_t>();
  unsigned long long *d_hist = reinterpret_cast<unsigned long long *>(d_totals + 64);
  uint64_t *d_digit_base = reinterpret_cast<uint64_t *>(d_hist + MAX_PASSES * RADIX);
  unsigned long long *d_phist = reinterpret_cast<unsigned long long *>(d_digit_base + MAX_PASSES * RADIX);
  if (n > 0)
    DBG_LAUNCH(ctx, ST_OFFSETS, 4.0 * n,
               k_read_tile_sums<<<(unsigned)off_tiles, OFF_BLOCK, 0, s>>>(in.d_lengths, n, k, tile_sums.as<Sum3>()));
  DBG_LAUNCH(ctx, ST_OFFSETS, 0.0,
             k_scan_tile_sums<<<1, 1024, 0, s>>>(tile_sums.as<Sum3>(), (uint32_t)off_tiles, d_totals,
                                                 base_off.as<uint64_t>(), edge_off.as<uint64_t>(), n));
  if (n > 0)
    DBG_LAUNCH(ctx, ST_OFFSETS, 20.0 * n,
               k_read_offsets<<<(unsigned)off_tiles, OFF_BLOCK, 0, s>>>(in.d_lengths, n, k, tile_sums.as<Sum3>(),
                                                                        base_off.as<uint64_t>(),
                                                                        edge_off.as<uint64_t>()));
  DBG_CUDA_TRY(cudaGetLastError());
  uint64_t totals[3];
  DBG_TRY(read_small(ctx, d_totals, sizeof(totals), totals));
  const uint64_t total_bases = totals[0], N = totals[1], I = totals[2];
  tile_sums.release();
  g->num_instances = N;

  // ---- pack the reads once; host reads stream through a staging buffer ----
  DevBuf packed;
  const uint64_t nwords = (total_bases + 31) / 32;
  DBG_TRY(alloc_tmp(ctx, packed, (nwords + 3) * 8));
  DBG_CUDA_TRY(cudaMemsetAsync(packed.as<uint64_t>() + nwords, 0, 3 * 8, s));
  if (nwords > 0) {
    if (in.reads_on_device) {
      DBG_LAUNCH(ctx, ST_PACK, (double)total_bases * 1.25,
                 k_pack<<<grid_for(nwords, 256), 256, 0, s>>>(reinterpret_cast<const uint8_t *>(in.reads),
                                                              total_bases, packed.as<uint64_t>(), nwords, ctx->d_err));
    } else {
      const uint64_t chunk = 256ull << 20;  // bases per staged copy (a multiple of 32)
      DevBuf stage;
      DBG_TRY(alloc_buf(ctx, stage, std::min(chunk, total_bases)));
      for (uint64_t off = 0; off < total_bases; off += chunk) {
        const uint64_t len = std::min(chunk, total_bases - off);
        DBG_CUDA_TRY(cudaMemcpyAsync(stage.p, in.reads + off, len, cudaMemcpyHostToDevice, s));
        DBG_LAUNCH(ctx, ST_PACK, (double)len * 1.25,
                   k_pack_at<<<grid_for((len + 31) / 32, 256), 256, 0, s>>>(stage.as<uint8_t>(), len,
                                                                          packed.as<uint64_t>(), off / 32,
                                                                          ctx->d_err));
      }
      DBG_CUDA_TRY(cudaStreamSynchronize(s));  // the staging buffer is released next
    }
  }
  DBG_CUDA_TRY(cudaGetLastError());
  DBG_TRY(check_device_error(ctx));

  // ---- edge-key ranges ----
  const unsigned emit_grid = (unsigned)std::min<uint64_t>(grid_for(n, EMIT_BLOCK / 32), 152ull * 64);
  std::vector<uint64_t> hist(PREFIX_BINS, 0);
  if (N > 0) {
    DBG_CUDA_TRY(cudaMemsetAsync(d_phist, 0, PREFIX_BINS * 8, s));
    DBG_LAUNCH(ctx, ST_EMIT, 8.0 * nwords + 16.0 * n,
               k_emit_prefix_hist<K><<<emit_grid, EMIT_BLOCK, 0, s>>>(packed.as<uint64_t>(), base_off.as<uint64_t>(),
                                                                      edge_off.as<uint64_t>(), n, k, d_phist));
    DBG_CUDA_TRY(cudaMemcpyAsync(hist.data(), d_phist, PREFIX_BINS * 8, cudaMemcpyDeviceToHost, s));
    DBG_CUDA_TRY(cudaStreamSynchronize(s));
  }
  const uint64_t persistent = (nwords + 3) * 8 + (n + 1) * 16;
  const uint64_t room = budget > persistent ? budget - persistent : 0;
  const uint64_t key_cap = std::max<uint64_t>(1ull << 16, room / (2 * w + 4 + 4));
  std::vector<uint64_t> sizes;
  auto ranges = plan_ranges(hist.data(), key_cap, &sizes);
  *n_edge_buckets = (uint32_t)ranges.size();

  const int kbits = 2 * m;
  std::vector<DevBuf> ck, cm, co;
  std::vector<uint64_t> ce;
  uint64_t E = 0;
  for (size_t b = 0; b < ranges.size(); b++) {
    const uint64_t cnt = sizes[b];
    if (cnt == 0) continue;
    DevBuf ka, kb, headpos;
    DBG_TRY(alloc_tmp(ctx, ka, cnt * w + MSD_PAD));
    DBG_TRY(alloc_tmp(ctx, kb, cnt * w + MSD_PAD));
    DBG_TRY(alloc_tmp(ctx, headpos, (cnt + 1) * 4));
    DBG_CUDA_TRY(cudaMemsetAsync(d_hist, 0, MAX_PASSES * RADIX * 8, s));
    DBG_CUDA_TRY(cudaMemsetAsync(ctx->d_counters + 8, 0, 4, s));
    const KeyRange<K> kr = key_range<K>(ranges[b].first, ranges[b].second, kbits);
    const SortPlan<K> plan = plan_sort<K>(ctx, cnt, kr.bits, ctx->partition_first, kr.density);
    DBG_LAUNCH(ctx, ST_EMIT, 8.0 * nwords + 16.0 * n + (double)cnt * w,
               k_emit_range<K><<<emit_grid, EMIT_BLOCK, EMIT_BLOCK / 32 * EMIT_BUF<K> * sizeof(K), s>>>(packed.as<uint64_t>(), base_off.as<uint64_t>(),
                                                                edge_off.as<uint64_t>(), n, k, ranges[b].first,
                                                                ranges[b].second, kr.base, ka.as<K>(), ctx->d_counters + 8,
                                                                plan.digits(), d_hist));
    DBG_CUDA_TRY(cudaGetLastError());
    K *kp = ka.as<K>(), *alt = kb.as<K>();
    uint32_t *vn = nullptr, *van = nullptr;
    uint64_t eb64 = 0;
    if (plan.local()) {
      // multiplicities go where the run heads would (headpos is cnt + 1 long)
      DevBuf mdense;
      DBG_TRY(sort_count_keys<K>(ctx, &kp, &alt, cnt, plan, d_hist, d_digit_base, &mdense, nullptr, &eb64));
      if (eb64) DBG_CUDA_TRY(cudaMemcpyAsync(headpos.p, mdense.p, eb64 * 4, cudaMemcpyDeviceToDevice, s));
    } else {
      DBG_TRY((radix_sort<K, false>(ctx, &kp, &alt, &vn, &van, cnt, kr.bits, d_hist, d_digit_base)));
      DBG_TRY(run_length_reduce<K>(ctx, kp, cnt, alt, headpos.as<uint32_t>(), &eb64));
    }
    DBG_TRY(check_device_error(ctx));
    const uint32_t eb = (uint32_t)eb64;
    DevBuf k1, m1, o1;
    DBG_TRY(alloc_tmp(ctx, k1, std::max<uint64_t>(1, eb) * w));
    DBG_TRY(alloc_tmp(ctx, m1, std::max<uint64_t>(1, eb) * 4));
    DBG_TRY(alloc_tmp(ctx, o1, std::max<uint64_t>(1, eb)));
    if (eb)
      DBG_LAUNCH(ctx, ST_ENDPOINTS, (double)eb * (2 * w + 9),
                 k_edge_finish<K><<<grid_for(eb, 256), 256, 0, s>>>(alt, kr.base, plan.local() ? nullptr : headpos.as<uint32_t>(),
                                                                   headpos.as<uint32_t>(), eb, k, k1.as<K>(),
                                                                   m1.as<uint32_t>(), o1.as<uint8_t>()));
    ck.push_back(std::move(k1));
    cm.push_back(std::move(m1));
    co.push_back(std::move(o1));
    ce.push_back(eb);
    E += eb;
  }
  if (E >= 0x80000000ull) {
    set_error("%llu unique edges exceed one build (2^31 - 1)", (unsigned long long)E);
    return DBG_EOVERFLOW;
  }
  g->num_edges = E;
  const uint64_t E1 = std::max<uint64_t>(1, E);
  DBG_TRY(alloc_buf(ctx, g->edge_keys, E1 * w));
  DBG_TRY(alloc_buf(ctx, g->mult, E1 * 4));
  DBG_TRY(alloc_buf(ctx, g->orient, E1));
  DBG_TRY(concat_chunks<K>(ctx, ck, ce, w, g->edge_keys.p));
  DBG_TRY(concat_chunks<K>(ctx, cm, ce, 4, g->mult.p));
  DBG_TRY(concat_chunks<K>(ctx, co, ce, 1, g->orient.p));

  // ---- node-key ranges ----
  DBG_TRY(alloc_buf(ctx, g->src, E1 * 4));
  DBG_TRY(alloc_buf(ctx, g->dst, E1 * 4));
  DBG_TRY(alloc_buf(ctx, g->adj_edge, 2 * E1 * 4));
  DBG_TRY(alloc_buf(ctx, g->adj_role, 2 * E1));
  DBG_TRY(alloc_buf(ctx, g->adj_nbr, 2 * E1 * 4));
  std::fill(hist.begin(), hist.end(), 0);
  if (E > 0) {
    DBG_CUDA_TRY(cudaMemsetAsync(d_phist, 0, PREFIX_BINS * 8, s));
    DBG_LAUNCH(ctx, ST_ENDPOINTS, (double)E * w,
               k_node_prefix_hist<K><<<grid_for(E, 256 * 8), 256, 0, s>>>(g->edge_keys.as<K>(), E, k, d_phist));
    DBG_CUDA_TRY(cudaMemcpyAsync(hist.data(), d_phist, PREFIX_BINS * 8, cudaMemcpyDeviceToHost, s));
    DBG_CUDA_TRY(cudaStreamSynchronize(s));
  }
  const uint64_t held = persistent + E1 * (w + 4 + 1 + 4 + 4 + 2 * 9);
  const uint64_t room2 = budget > held ? budget - held : 0;
  const uint64_t rec_cap = std::max<uint64_t>(1ull << 16, room2 / (2 * (w + 4) + 16));
  sizes.clear();
  auto nranges = plan_ranges(hist.data(), rec_cap, &sizes);
  *n_node_buckets = (uint32_t)nranges.size();
  const uint64_t etiles = (E + ENDS_TILE - 1) / ENDS_TILE;
  DevBuf tcount, toff, flags;
  if (E > 0) {
    DBG_TRY(alloc_tmp(ctx, flags, (E + 31) / 32 * 8));
    DBG_TRY(alloc_tmp(ctx, tcount, etiles * 4));
    DBG_TRY(alloc_tmp(ctx, toff, (etiles + 1) * 8));
  }
  const int nbits = 2 * (int)k;
  std::vector<DevBuf> cnk, crp;
  std::vector<uint64_t> cv;
  uint64_t base_v = 0, base_slot = 0;
  for (size_t c = 0; c < nranges.size(); c++) {
    const uint32_t lo = nranges[c].first, hi = nranges[c].second;
    uint32_t Rc = 0;
    if (E > 0) {
      DBG_LAUNCH(ctx, ST_ENDPOINTS, (double)E * w,
                 k_count_ends<K><<<(unsigned)etiles, ENDS_BLOCK, 0, s>>>(
                     g->edge_keys.as<K>(), E, k, lo, hi, flags.as<uint2>(), tcount.as<uint32_t>()));
      DBG_TRY(scan_u32(ctx, tcount.as<uint32_t>(), etiles, toff.as<uint64_t>(), &Rc, ST_ENDPOINTS));
    }
    const uint64_t cap = (uint64_t)Rc + I;
    if (cap == 0) continue;
    DevBuf ra, rb, va, vb, row_tmp;
    DBG_TRY(alloc_tmp(ctx, ra, cap * w + MSD_PAD));
    DBG_TRY(alloc_tmp(ctx, rb, cap * w + MSD_PAD));
    DBG_TRY(alloc_tmp(ctx, va, cap * 4 + MSD_PAD));
    DBG_TRY(alloc_tmp(ctx, vb, cap * 4 + MSD_PAD));
    // (planned for every record that the range may hold: isolated reads are
    // counted by the range only)
    const KeyRange<K> kr = key_range<K>(lo, hi, nbits);
    const SortPlan<K> rplan = plan_records<K>(ctx, cap, kr.bits, false, kr.density);
    DBG_CUDA_TRY(cudaMemsetAsync(d_hist, 0, MAX_PASSES * RADIX * 8, s));
    if (Rc > 0)
      DBG_LAUNCH(ctx, ST_ENDPOINTS, (double)E * w + (double)Rc * (w + 4),
                 k_gather_ends<K><<<(unsigned)std::min<uint64_t>(etiles, 152ull * 8), ENDS_BLOCK, 0, s>>>(
                     g->edge_keys.as<K>(), E, k, flags.as<uint2>(), toff.as<uint64_t>(), etiles, kr.base, ra.as<K>(), va.as<uint32_t>(),
                     rplan.digits(), d_hist));
    uint64_t R = Rc;
    if (I > 0) {
      DBG_CUDA_TRY(cudaMemsetAsync(ctx->d_counters + 9, 0, 4, s));
      DBG_LAUNCH(ctx, ST_ENDPOINTS, (double)n * 4,
                 k_isolated_range<K><<<grid_for(n, 256), 256, 0, s>>>(packed.as<uint64_t>(), base_off.as<uint64_t>(),
                                                                     in.d_lengths, n, k, lo, hi, kr.base, ra.as<K>() + Rc,
                                                                     va.as<uint32_t>() + Rc, ctx->d_counters + 9,
                                                                     rplan.digits(), d_hist));
      uint32_t iso = 0;
      DBG_TRY(read_small(ctx, ctx->d_counters + 9, 4, &iso));
      R += iso;
    }
    if (R == 0) continue;
    K *rk = ra.as<K>(), *rk_alt = rb.as<K>();
    uint32_t *rv = va.as<uint32_t>(), *rv_alt = vb.as<uint32_t>();
    DBG_TRY(sort_records<K>(ctx, &rk, &rk_alt, &rv, &rv_alt, R, rplan, edge_end_order(E, false, I > 0), d_hist,
                            d_digit_base));
    DBG_TRY(alloc_tmp(ctx, row_tmp, (R + 1) * 8));
    uint64_t tot[2] = {0, 0};
    DBG_TRY(assign_node_ids<K>(ctx, rk, rv, R, rk_alt, row_tmp.as<uint64_t>(), g, (uint32_t)base_v, base_slot,
                               &tot[0], &tot[1]));
    DBG_TRY(check_device_error(ctx));
    const uint64_t Vc = tot[0];
    DevBuf nk, rp;
    DBG_TRY(alloc_tmp(ctx, nk, std::max<uint64_t>(1, Vc) * w));
    DBG_TRY(alloc_tmp(ctx, rp, std::max<uint64_t>(1, Vc) * 8));
    if (Vc) {
      DBG_LAUNCH(ctx, ST_COPIES, 2.0 * Vc * w,
                 k_add_base<K><<<grid_for(Vc, 256 * 8), 256, 0, s>>>(rk_alt, Vc, kr.base, nk.as<K>()));
      DBG_CUDA_TRY(cudaMemcpyAsync(rp.p, row_tmp.p, Vc * 8, cudaMemcpyDeviceToDevice, s));
    }
    cnk.push_back(std::move(nk));
    crp.push_back(std::move(rp));
    cv.push_back(Vc);
    base_v += Vc;
    base_slot += tot[1];
  }
  if (base_slot != 2 * E) {
    set_error("adjacency holds %llu edge ends, expected %llu", (unsigned long long)base_slot,
              (unsigned long long)(2 * E));
    return DBG_EINTERNAL;
  }
  const uint64_t V = base_v;
  g->num_nodes = V;
  DBG_TRY(alloc_buf(ctx, g->node_keys, std::max<uint64_t>(1, V) * w));
  DBG_TRY(alloc_buf(ctx, g->row_ptr, (V + 1) * 8));
  DBG_TRY(concat_chunks<K>(ctx, cnk, cv, w, g->node_keys.p));
  DBG_TRY(concat_chunks<K>(ctx, crp, cv, 8, g->row_ptr.p));
  uint64_t *last = reinterpret_cast<uint64_t *>(ctx->h_pinned + 64);  // pinned: safe for an async copy
  *last = 2 * E;
  DBG_CUDA_TRY(cudaMemcpyAsync(g->row_ptr.as<uint64_t>() + V, last, 8, cudaMemcpyHostToDevice, s));
  if (E > 0)
    DBG_LAUNCH(ctx, ST_ADJACENCY, 2.0 * E * 13,
               k_adj_nbr<<<grid_for(2 * E, 256 * 8), 256, 0, s>>>(g->adj_edge.as<uint32_t>(), g->adj_role.as<uint8_t>(),
                                                                 g->src.as<uint32_t>(), g->dst.as<uint32_t>(), 2 * E,
                                                                 g->adj_nbr.as<uint32_t>()));
  DBG_CUDA_TRY(cudaGetLastError());
  return check_device_error(ctx);  // waits for the stream
}

}  // namespace dbg
