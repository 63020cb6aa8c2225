// msm.cu -- multi-scalar multiplication on BN254 G1 and BLS12-381 G1 by the
// paper's Layout-Stationary Pippenger (MORPH, Algorithm 2), GB300 form.
//
//   MSM = sum_{n<N} S_n P_n, S_n < r (254 or 255 bits), P_n affine points.
//
// Every kernel that touches points is a template over the curve (its base
// field's traits and its scalar field); the sort and scan kernels are shared.
// Each scalar is cut into K = ceil((S^BL + 1) / c) signed c-bit digits
// d_k in [-(2^(c-1) - 1), 2^(c-1)] (sum_k d_k 2^(k c) = S_n); window k keeps
// 2^(c-1) buckets, bucket j collecting the points whose digit has magnitude
// j + 1 (negated when the digit is negative).  The four phases of
// Algorithm 2 map to kernels:
//
//   Bucketize    msm_count_kernel      bucket sizes (one counter per bucket,
//                                      atomics in L2; zero digits skipped)
//                scan_*_kernel         exclusive scan -> bucket offsets
//                msm_scatter_kernel    point index (and digit sign) into the
//                                      next slot of its bucket: the argsort of
//                                      the digits as a counting sort
//   BA           msm_accumulate_kernel the bucket-sorted entries cut into
//                                      segments of exactly S; one thread adds
//                                      its S points (XYZZ += affine), writing a
//                                      bucket that lies inside its segment
//                                      straight to the bucket array and the
//                                      pieces of the (at most two) buckets
//                                      that cross its ends to piece slots;
//                msm_combine_kernel    the pieces of each crossing bucket added
//                                      up, one thread or four lanes per bucket
//                msm_combine_long_kernel  buckets over many segments: a radix-4
//                                      tree over their pieces (a skewed or
//                                      constant scalar set stays parallel and
//                                      balanced)
//   BR           msm_reduce_level_kernel  the tree of Algorithm 2, one launch
//                                      per level, all windows at once:
//                                      W_b = W_2b + W_2b+1 + B_2b+1,
//                                      B_b = 2 (B_2b + B_2b+1); the leaves
//                                      start at W_j = B_j, so the root holds
//                                      sum_j (j + 1) B_j
//                msm_reduce_chunk_kernel  its lowest levels at once where there
//                                      are many buckets
//                msm_reduce_level_quad_kernel  levels of few nodes: four lanes
//                                      for a W, four for a B
//   WM           msm_merge_kernel      Horner over the windows, top one first
//                                      (MSM = 2^c MSM + W_k), four lanes per
//                                      point, then the affine standard-form
//                                      result.
//
// The paper streams the sorted points straight into bucket accumulation on
// the TPU; here the sort moves 4-byte point indices and the accumulation
// gathers the 64- or 96-byte points by index (a point is read once per
// window from HBM; the accumulation is bound by the integer multiply pipe,
// not by these reads).  Points are converted to Montgomery form once per
// call (msm_prepare_kernel), which also checks that every point lies on the
// curve.
//
// Two variants reuse the same kernels: a window range [kb, ke) (the count
// and scatter kernels skip the other windows' digits, the tree and merge run
// over the range only) gives one rank's part of a window-sharded MSM; and
// precomputed bases (msm_bases_kernel stores every point's window copies
// 2^(k c) P once) put all windows' digits into one bucket set ("flat" count
// and scatter), so one tree replaces K and the window merge disappears.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <cstring>
#include <map>
#include <mutex>
#include <new>

#include "../../include/msm_gb300.h"
#include "ec_xyzz.cuh"
#include "nvtx_range.h"

namespace gb300ntt {
namespace {

constexpr int kScanThreads = 256;
constexpr int kScanPer = 8;
constexpr int kScanTile = kScanThreads * kScanPer;
constexpr int kEcThreads = 128;
constexpr uint32_t kSignBit = 0x80000000u;
// A bucket that crosses few segment ends is added up by one thread (or four
// lanes); longer ones by a tree of radix 4 over their pieces (three additions a
// level; radix 8 took 154 us instead of the tree's 100 for 1300 pieces of
// BLS12-381, radix 2 needs twice the launches).  Where the average bucket is
// shorter than a segment the longer ones are few, the tree runs for the longest
// anyway, and the limit is the additions of one level (50,000 witness scalars of
// BLS12-381: 1531 us a call with 3, 1604 with 8).  Where the average bucket
// crosses several ends nearly all of them do, and one thread for each fills the
// GPU (BLS12-381 commitment, 2^20 points: 6655 us with 8, 6713 with 3).
constexpr uint32_t kShortSpan = 3, kShortSpanLongBuckets = 8;
// Entries that one sweep of the scatter is meant to write, 4 bytes each at random
// places of its windows' part of the sorted array: 64 MiB stay in the L2 (129 MB)
// until their sectors are complete, while the scalars are read again for each
// sweep.  (The sweeps of a block follow one another, those of different blocks need
// not.)  2^22 points of BN254: 1134 us in one sweep of 15 windows, 804 in five (the
// whole call 12.65 ms, 12.39 with 2^23 entries, 12.29 with 2^24, 12.34 with 2^25).
// Above 2^24 points a sweep is one window, larger than that, and still the best:
// whole calls of BN254, one window a sweep, two, all: 2^25 84.6, 87.4 and 91.3 ms,
// 2^26 170, 176 and 183 ms; BLS12-381 2^25 172.5, 175.3 and 179.2 ms.
constexpr uint64_t kSweepEntries = 1ull << 24;
constexpr uint32_t kSegMask = (1u << 28) - 1u;   // a segment index (span - 1 above it in a crossing item)
constexpr int kLongLevels = 14;    // 4^14 pieces
// Tree levels of at most this many nodes per SM take eight lanes per node.
constexpr uint32_t kQuadNodesPerSm = 128;

// Curves: base-field traits, the scalar modulus r (for the input check),
// the curve constant b, and the CTAs of 128 threads per SM that the register
// budget of the point kernels allows.  The scalar bit length and the
// generator are host-side (curve_scalar_bits, curve_generator).
struct CurveBn254 {
  using T = FqBn254;
  static constexpr int kMinBlocks = 4;
  static constexpr int kTreeMinBlocks = 4;  // reduction-tree and combine kernels
  static constexpr uint32_t kB = 3;
  __device__ static bool scalar_ok(const uint32_t s[8]) {
    const uint32_t r[8] = {0xf0000001u, 0x43e1f593u, 0x79b97091u, 0x2833e848u,
                           0x8181585du, 0xb85045b6u, 0xe131a029u, 0x30644e72u};
#pragma unroll
    for (int j = 7; j >= 0; --j)
      if (s[j] != r[j]) return s[j] < r[j];
    return false;
  }
};

struct CurveBls381 {
  using T = FqBls381;
  static constexpr int kMinBlocks = 3;
  static constexpr int kTreeMinBlocks = 2;  // two XYZZ points live: 255 registers, no spill
  static constexpr uint32_t kB = 4;
  __device__ static bool scalar_ok(const uint32_t s[8]) {
    const uint32_t r[8] = {0x00000001u, 0xffffffffu, 0xfffe5bfeu, 0x53bda402u,
                           0x09a1d805u, 0x3339d808u, 0x299d7d48u, 0x73eda753u};
#pragma unroll
    for (int j = 7; j >= 0; --j)
      if (s[j] != r[j]) return s[j] < r[j];
    return false;
  }
};

template <class T>
struct EcConst {
  uint32_t one[T::L];  // 2^(32 L) mod q (Montgomery 1)
  uint32_t r2[T::L];   // 2^(64 L) mod q (to Montgomery form)
  uint32_t b3[T::L];   // b 2^(32 L) mod q (curve constant, Montgomery)
  uint32_t gx[T::L];   // generator, standard form
  uint32_t gy[T::L];
};

struct MsmTotals {
  uint32_t entries;                // points placed in buckets (digit != 0)
  uint32_t seg_len;                // S, entries per segment (from the entries there are)
  uint32_t crossing;               // buckets over few segments (short_span)
  uint32_t items[kLongLevels];     // work items of the levels of the long buckets' trees
  uint32_t err;                    // MSM_ERR_* bits
};

// Work lists of the combine kernels, filled by the accumulation: `crossing` the
// segment in which each short crossing bucket starts; `items` + item_base[l]
// the segments whose piece is a node of level l of a long bucket's tree (bit
// 31: the head piece, in the segment where the bucket starts).
struct CombineLists {
  uint32_t *crossing;
  uint32_t *items;
  uint32_t item_base[kLongLevels];
};

// ----------------------------------------------------------- small helpers

template <class T>
__device__ __forceinline__ void load_point_xyzz(Xyzz<T> &p, const uint4 *base, uint64_t i) {
  T::load(p.X, base, 4 * i + 0);
  T::load(p.Y, base, 4 * i + 1);
  T::load(p.ZZ, base, 4 * i + 2);
  T::load(p.ZZZ, base, 4 * i + 3);
}

template <class T>
__device__ __forceinline__ void store_point_xyzz(uint4 *base, uint64_t i, const Xyzz<T> &p) {
  T::store(base, 4 * i + 0, p.X);
  T::store(base, 4 * i + 1, p.Y);
  T::store(base, 4 * i + 2, p.ZZ);
  T::store(base, 4 * i + 3, p.ZZZ);
}

// Raw c-bit digit of window k of the scalar s (8 little-endian words); c <= 22.
__device__ __forceinline__ uint32_t raw_digit(const uint32_t s[8], uint32_t k, uint32_t c) {
  const uint32_t bit = k * c, w = bit >> 5, sh = bit & 31u;
  if (w >= 8) return 0u;
  uint64_t v = s[w];
  if (w + 1 < 8) v |= (uint64_t)s[w + 1] << 32;
  return (uint32_t)(v >> sh) & ((1u << c) - 1u);
}

// Next signed digit: v = raw + carry in [0, 2^c]; v > 2^(c-1) becomes
// v - 2^c (negative) with a carry into the next window.  Returns the
// magnitude (0 for a zero digit); neg is the sign.
__device__ __forceinline__ uint32_t signed_digit(const uint32_t s[8], uint32_t k, uint32_t c, uint32_t &carry,
                                                 bool &neg) {
  const uint32_t v = raw_digit(s, k, c) + carry;
  neg = v > (1u << (c - 1));
  carry = neg ? 1u : 0u;
  return neg ? (1u << c) - v : v;
}

// ---------------------------------------------------------------- kernels

// Points to Montgomery form (x R, y R); (0, 0) stays the point at infinity.
// Flags points that are not canonical or not on y^2 = x^3 + b (and treats
// them as O so that the arithmetic below never sees a value >= q).
template <class C>
__global__ void __launch_bounds__(kEcThreads) msm_prepare_kernel(const uint4 *pts, uint64_t n,
                                                                 EcConst<typename C::T> k, uint4 *pts_m,
                                                                 MsmTotals *tot) {
  using T = typename C::T;
  constexpr int L = T::L;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t x[L], y[L];
    T::load(x, pts, 2 * i);
    T::load(y, pts, 2 * i + 1);
    if (fv_is_zero<L>(x) && fv_is_zero<L>(y)) {
      T::store(pts_m, 2 * i, x);
      T::store(pts_m, 2 * i + 1, y);
      continue;
    }
    bool ok = T::canonical(x) && T::canonical(y);
    if (ok) {
      T::mul(x, x, k.r2);
      T::mul(y, y, k.r2);
      uint32_t l[L], r[L];
      f_sqr<T, false>(l, y);
      f_sqr<T, false>(r, x);
      T::mul(r, r, x);
      T::add(r, r, k.b3);
      ok = fv_equal<L>(l, r);
    }
    if (!ok) {
      atomicOr(&tot->err, (uint32_t)MSM_ERR_POINT);
      fv_zero<L>(x);
      fv_zero<L>(y);
    }
    T::store(pts_m, 2 * i, x);
    T::store(pts_m, 2 * i + 1, y);
  }
}

// Bucketize, pass 1: one counter per (window, digit magnitude), windows
// [kb, ke) (the digits below kb are still recoded for their carries).
// With precomputed bases (flat = true) every window uses the same 2^(c-1)
// buckets: the point of digit k of scalar i is the copy 2^(k c) P_i.
template <class C>
__global__ void __launch_bounds__(256) msm_count_kernel(const uint4 *__restrict__ scalars, uint64_t n, uint32_t c,
                                                        uint32_t kb, uint32_t ke, bool flat,
                                                        uint32_t *__restrict__ counts, MsmTotals *tot) {
  const uint32_t lb = flat ? 0u : c - 1;  // window stride of the bucket index (log2)
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t s[8];
    fe_load_global(s, scalars, i);
    if (!C::scalar_ok(s)) atomicOr(&tot->err, (uint32_t)MSM_ERR_SCALAR);
    uint32_t carry = 0;
    for (uint32_t k = 0; k < ke; ++k) {
      bool neg;
      const uint32_t m = signed_digit(s, k, c, carry, neg);
      if (m && k >= kb) atomicAdd(&counts[(flat ? 0ull : ((uint64_t)k << lb)) + m - 1], 1u);
    }
  }
}

// Inclusive scan across a warp.
__device__ __forceinline__ uint32_t warp_scan(uint32_t v) {
  const uint32_t lane = threadIdx.x & 31u;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t a = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= (uint32_t)o) v += a;
  }
  return v;
}

// Exclusive scan of v over the CTA (blockDim.x = kScanThreads); *total gets
// the CTA's sum.
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t *total) {
  __shared__ uint32_t warp_sums[kScanThreads / 32];
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const uint32_t inc = warp_scan(v);
  if (lane == 31) warp_sums[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    const uint32_t w = lane < kScanThreads / 32 ? warp_sums[lane] : 0u;
    const uint32_t wi = warp_scan(w);
    if (lane < kScanThreads / 32) warp_sums[lane] = wi - w;
    if (lane == kScanThreads / 32 - 1) *total = wi;
  }
  __syncthreads();
  const uint32_t base = warp_sums[warp];
  __syncthreads();
  return base + inc - v;
}

// Scan pass 1: per-tile sums of the bucket sizes.
__global__ void __launch_bounds__(kScanThreads) scan_reduce_kernel(const uint32_t *counts, uint64_t nb,
                                                                   uint32_t *tile_sums) {
  const uint64_t base = (uint64_t)blockIdx.x * kScanTile + (uint64_t)threadIdx.x * kScanPer;
  uint32_t v = 0;
#pragma unroll
  for (int j = 0; j < kScanPer; ++j)
    if (base + j < nb) v += counts[base + j];
  __shared__ uint32_t total;
  block_excl_scan(v, &total);
  if (threadIdx.x == 0) tile_sums[blockIdx.x] = total;
}

// Scan pass 2 (one CTA): exclusive scan of the tile sums in place; the total
// goes to tot->entries and offsets[nb], and fixes the segment length.
__global__ void __launch_bounds__(kScanThreads) scan_tiles_kernel(uint32_t *tile_sums, uint32_t num_tiles,
                                                                  uint64_t nb, uint32_t *offsets, uint32_t max_segments,
                                                                  MsmTotals *tot) {
  __shared__ uint32_t chunk_total;
  uint32_t carry = 0;
  for (uint32_t b0 = 0; b0 < num_tiles; b0 += kScanThreads) {
    const uint32_t i = b0 + threadIdx.x;
    const uint32_t v = i < num_tiles ? tile_sums[i] : 0u;
    const uint32_t ex = block_excl_scan(v, &chunk_total);
    if (i < num_tiles) tile_sums[i] = carry + ex;
    __syncthreads();
    carry += chunk_total;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    tot->entries = carry;
    // as many segments as the plan has room for (a whole number of waves),
    // with at least 8 entries each: sparse scalars make fewer entries
    tot->seg_len = max(8u, (uint32_t)(((uint64_t)carry + max_segments - 1) / max_segments));
    offsets[nb] = carry;
  }
}

// Scan pass 3: bucket offsets, also copied to the scatter cursors.
__global__ void __launch_bounds__(kScanThreads) scan_apply_kernel(const uint32_t *counts, uint64_t nb,
                                                                  const uint32_t *tile_sums, uint32_t *offsets,
                                                                  uint32_t *cursor) {
  const uint64_t base = (uint64_t)blockIdx.x * kScanTile + (uint64_t)threadIdx.x * kScanPer;
  uint32_t cnt[kScanPer];
  uint32_t v = 0;
#pragma unroll
  for (int j = 0; j < kScanPer; ++j) {
    cnt[j] = base + j < nb ? counts[base + j] : 0u;
    v += cnt[j];
  }
  __shared__ uint32_t total;
  uint32_t run = block_excl_scan(v, &total) + tile_sums[blockIdx.x];
#pragma unroll
  for (int j = 0; j < kScanPer; ++j) {
    if (base + j < nb) {
      offsets[base + j] = run;
      cursor[base + j] = run;
    }
    run += cnt[j];
  }
}

// Bucketize, pass 2: each point index (sign in bit 31) into the next free
// slot of its bucket, windows [kb, ke), `sweep` windows at a time; the atomics of
// up to eight windows are in flight at once.
__global__ void __launch_bounds__(256) msm_scatter_kernel(const uint4 *__restrict__ scalars, uint64_t n, uint32_t c,
                                                          uint32_t kb, uint32_t ke, uint32_t sweep,
                                                          uint32_t flat_stride, uint32_t *__restrict__ cursor,
                                                          uint32_t *__restrict__ sorted) {
  // flat_stride > 0: precomputed bases, one bucket set, point copy k at k * flat_stride
  const uint32_t lb = c - 1;
  for (uint32_t g0 = kb; g0 < ke; g0 += sweep) {
    const uint32_t g1 = min(g0 + sweep, ke);
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
      uint32_t s[8];
      fe_load_global(s, scalars, i);
      uint32_t carry = 0;
      for (uint32_t k = 0; k < g0; ++k) {
        bool neg;
        signed_digit(s, k, c, carry, neg);
      }
      for (uint32_t k0 = g0; k0 < g1; k0 += 8) {
        uint32_t pos[8], val[8];
#pragma unroll
        for (uint32_t j = 0; j < 8; ++j) {
          const uint32_t k = k0 + j;
          bool neg = false;
          const uint32_t m = k < g1 ? signed_digit(s, k, c, carry, neg) : 0u;
          const uint64_t bucket = (flat_stride ? 0ull : ((uint64_t)k << lb)) + m - 1;
          pos[j] = m ? atomicAdd(&cursor[bucket], 1u) : 0xffffffffu;
          val[j] = ((uint32_t)i + k * flat_stride) | (neg ? kSignBit : 0u);
        }
#pragma unroll
        for (uint32_t j = 0; j < 8; ++j)
          if (pos[j] != 0xffffffffu) sorted[pos[j]] = val[j];
      }
    }
  }
}

// Largest b with offsets[b] <= e (offsets non-decreasing, offsets[0] = 0,
// e < offsets[nb]): the bucket holding sorted entry e.
__device__ __forceinline__ uint32_t bucket_of_entry(const uint32_t *offsets, uint64_t nb, uint32_t e) {
  uint64_t lo = 0, hi = nb;  // offsets[lo] <= e < offsets[hi]
  while (hi - lo > 1) {
    const uint64_t mid = (lo + hi) >> 1;
    if (__ldg(offsets + mid) <= e) lo = mid;
    else hi = mid;
  }
  return (uint32_t)lo;
}

// Where the partial sum of bucket b over segment t goes: a bucket inside the
// segment is complete (bucket array); a bucket that started in an earlier
// segment leaves its piece in slot 2t; one that starts here and continues
// leaves its head piece in slot 2t + 1.
template <class T>
__device__ __forceinline__ void emit_piece(const Xyzz<T> &acc, uint32_t b, uint32_t t, bool started_before,
                                           bool continues, uint4 *bucket_sum, uint4 *pieces) {
  if (!started_before && !continues) store_point_xyzz(bucket_sum, b, acc);
  else if (started_before) store_point_xyzz(pieces, 2 * (uint64_t)t, acc);
  else store_point_xyzz(pieces, 2 * (uint64_t)t + 1, acc);
}

// `used`: the buckets of the windows that the call runs over.
__device__ __forceinline__ uint32_t short_span(const MsmTotals *tot, uint64_t used) {
  return tot->entries >= used * tot->seg_len ? kShortSpanLongBuckets : kShortSpan;
}

// Piece i of a bucket over `span` + 1 segments, in segment t: a node of every
// level l of its tree for which i is a multiple of 4^(l + 1) and i + 4^l <=
// span.  One atomic per item: the lanes of a warp that are here together may be
// at different levels, so that one atomic for all of them would take a slot of
// one level's list for an item of another's.
__device__ __forceinline__ void push_items(MsmTotals *tot, const CombineLists &lists, uint32_t t, uint32_t i,
                                           uint32_t span, uint32_t limit) {
  if (span <= limit) return;
  uint32_t step = 1;
  for (int l = 0; l < kLongLevels && (i & (4 * step - 1)) == 0 && i + step <= span; ++l, step *= 4)
    lists.items[lists.item_base[l] + atomicAdd(&tot->items[l], 1u)] = t | (i == 0 ? kSignBit : 0u);
}

// BA: segment t adds the points of sorted entries [t S, t S + S).
template <class C>
__global__ void __launch_bounds__(kEcThreads, C::kMinBlocks)
    msm_accumulate_kernel(const uint4 *__restrict__ pts_m, const uint32_t *__restrict__ sorted,
                          const uint32_t *__restrict__ offsets, uint64_t nb, uint64_t used, EcConst<typename C::T> k,
                          MsmTotals *tot, CombineLists lists, uint4 *bucket_sum, uint4 *pieces) {
  using T = typename C::T;
  constexpr int L = T::L;
  const uint32_t n_entries = tot->entries, S = tot->seg_len;
  const uint32_t num_segs = (n_entries + S - 1) / S, limit = short_span(tot, used);
  for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < num_segs; t += gridDim.x * blockDim.x) {
    const uint32_t e0 = t * S, e1 = min(e0 + S, n_entries);
    uint32_t b = bucket_of_entry(offsets, nb, e0);
    uint32_t end_b = __ldg(offsets + b + 1);
    bool started_before = __ldg(offsets + b) < e0;
    if (started_before) {
      const uint32_t t0 = __ldg(offsets + b) / S;
      push_items(tot, lists, t, t - t0, (end_b - 1) / S - t0, limit);
    }
    Xyzz<T> acc;
    xyzz_set_inf(acc);
    for (uint32_t e = e0; e < e1; ++e) {
      if (e == end_b) {  // bucket b ends inside the segment
        emit_piece(acc, b, t, started_before, false, bucket_sum, pieces);
        xyzz_set_inf(acc);
        do {
          ++b;
          end_b = __ldg(offsets + b + 1);
        } while (end_b == e);  // skip empty buckets
        started_before = false;
      }
      const uint32_t v = __ldg(sorted + e);
      const uint64_t idx = v & ~kSignBit;
      uint32_t x[L], y[L];
      T::load(x, pts_m, 2 * idx);
      T::load(y, pts_m, 2 * idx + 1);
      if (fv_is_zero<L>(x) && fv_is_zero<L>(y)) continue;  // point at infinity
      if (v & kSignBit) {
        uint32_t zero[L];
        fv_zero<L>(zero);
        T::sub(y, zero, y);
      }
      xyzz_madd<T>(acc, x, y, k.one);
    }
    const bool continues = end_b > e1;
    emit_piece(acc, b, t, started_before, continues, bucket_sum, pieces);
    if (continues && !started_before) {
      const uint32_t span = (end_b - 1) / S - t;  // segments after t that hold bucket b
      if (span <= limit) lists.crossing[atomicAdd(&tot->crossing, 1u)] = t | (uint32_t)(span - 1) << 28;
      else push_items(tot, lists, t, 0, span, limit);
    }
  }
}

// The pieces of a bucket that crosses the ends of segments t0 < t0 + 1 < ... <
// t0 + span form V[0] = head slot 2 t0 + 1, V[i] = slot 2 (t0 + i); their sum
// goes to V[0].  One thread per bucket, or, when there are too few buckets to
// fill the grid, four lanes (an addition is then 4 products deep, not 14).
template <class C>
__global__ void __launch_bounds__(kEcThreads, C::kTreeMinBlocks)
    msm_combine_kernel(const MsmTotals *tot, const uint32_t *__restrict__ crossing, uint4 *pieces) {
  using T = typename C::T;
  constexpr int L = T::L;
  const uint32_t count = tot->crossing, threads = gridDim.x * blockDim.x;
  const uint32_t id = blockIdx.x * blockDim.x + threadIdx.x;
  if (count <= threads / 4) {
    for (uint32_t i0 = (id & ~31u) / 4; i0 < count; i0 += threads / 4) {   // uniform in a warp
      const uint32_t i = i0 + (id & 31u) / 4;
      const bool live = i < count;
      const uint32_t item = crossing[live ? i : i0];
      const uint32_t t = item & kSegMask, span = live ? (item >> 28) + 1 : 0u;
      const uint32_t most = __reduce_max_sync(0xffffffffu, span);
      uint32_t v[L], w[L];
      quad_load<T>(v, pieces, 2 * (uint64_t)t + 1);
#pragma unroll 1
      for (uint32_t j = 1; j <= most; ++j) {
        if (j <= span) quad_load<T>(w, pieces, 2 * (uint64_t)(t + j));
        else fv_zero<L>(w);   // O
        quad_add<T>(v, w);
      }
      if (live) quad_store<T>(pieces, 2 * (uint64_t)t + 1, v);
    }
    return;
  }
  for (uint32_t i = id; i < count; i += threads) {
    const uint32_t item = crossing[i], t = item & kSegMask, span = (item >> 28) + 1;
    Xyzz<T> a;
    load_point_xyzz(a, pieces, 2 * (uint64_t)t + 1);
#pragma unroll 1
    for (uint32_t j = 1; j <= span; ++j) {
      Xyzz<T> q;
      load_point_xyzz(q, pieces, 2 * (uint64_t)(t + j));
      xyzz_add<T, true>(a, q);
    }
    store_point_xyzz(pieces, 2 * (uint64_t)t + 1, a);
  }
}

// Level l of the long buckets' trees: V[i] += V[i + m 4^l], m = 1..3, for the
// listed i (multiples of 4^(l + 1)); four lanes per item.
template <class C>
__global__ void __launch_bounds__(kEcThreads)
    msm_combine_long_kernel(const uint32_t *__restrict__ offsets, uint64_t nb, const MsmTotals *tot,
                            CombineLists lists, int level, uint4 *pieces) {
  using T = typename C::T;
  constexpr int L = T::L;
  const uint32_t count = tot->items[level], threads = gridDim.x * blockDim.x, S = tot->seg_len;
  const uint32_t id = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t *items = lists.items + lists.item_base[level];
  const uint32_t step = 1u << (2 * level);
  for (uint32_t i0 = (id & ~31u) / 4; i0 < count; i0 += threads / 4) {   // uniform in a warp
    const uint32_t i = i0 + (id & 31u) / 4;
    const bool live = i < count;
    const uint32_t item = items[live ? i : i0];
    const uint32_t t = item & ~kSignBit;
    const uint64_t slot = 2 * (uint64_t)t + (item & kSignBit ? 1u : 0u);
    // segments of this bucket after t: up to the segment of its last entry
    const uint32_t e = item & kSignBit ? min((t + 1) * S, tot->entries) - 1 : t * S;
    const uint32_t b = bucket_of_entry(offsets, nb, e);
    const uint32_t after = live ? (__ldg(offsets + b + 1) - 1) / S - t : 0u;
    uint32_t v[L], w[L];
    quad_load<T>(v, pieces, slot);
#pragma unroll 1
    for (uint32_t m = 1; m < 4; ++m) {
      const bool add = after >= m * step;
      if (!__any_sync(0xffffffffu, add)) break;
      if (add) quad_load<T>(w, pieces, 2 * (uint64_t)(t + m * step));
      else fv_zero<L>(w);
      quad_add<T>(v, w);
    }
    if (live) quad_store<T>(pieces, slot, v);
  }
}

// Bucket b's sum after accumulation: O, the complete sum, or the head piece.
template <class T>
__device__ __forceinline__ void load_bucket(Xyzz<T> &p, const uint4 *bucket_sum, const uint4 *pieces,
                                            const uint32_t *offsets, uint32_t S, uint64_t b) {
  const uint32_t ob = offsets[b], ob1 = offsets[b + 1];
  if (ob1 == ob) xyzz_set_inf(p);
  else if (ob / S == (ob1 - 1) / S) load_point_xyzz(p, bucket_sum, b);
  else load_point_xyzz(p, pieces, 2 * (uint64_t)(ob / S) + 1);
}

// BR, level s of the tree (all windows): node (k, b), b < 2^s, from its two
// children.  Window k has 2^(c-1) leaves (the buckets); level s of its tree
// is stored at heap index 2^s + b.  At the level above the leaves the
// children's W are the leaves themselves (W_j = B_j).
template <class C>
__global__ void __launch_bounds__(kEcThreads, C::kTreeMinBlocks)
    msm_reduce_level_kernel(uint32_t s, uint32_t lb, uint32_t kb, uint32_t nk, const uint4 *bucket_sum,
                            const uint4 *pieces, const uint32_t *offsets, const MsmTotals *tot, uint4 *heap_w,
                            uint4 *heap_b) {
  using T = typename C::T;
  const uint32_t S = tot->seg_len;
  const uint64_t per = 1ull << s, total = per * nk;  // windows kb .. kb + nk - 1
  for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < total;
       t += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t k = kb + (t >> s), b = t & (per - 1);
    const uint64_t heap0 = k << lb;  // window k's heap
    const uint64_t node = heap0 + per + b;
    Xyzz<T> a, br;
    if (s + 1 == lb) {
      const uint64_t leaf = heap0 + 2 * b;
      load_bucket(a, bucket_sum, pieces, offsets, S, leaf);
      load_bucket(br, bucket_sum, pieces, offsets, S, leaf + 1);
      xyzz_add<T, true>(a, br);                     // B_L + B_R
      Xyzz<T> w = a;
      xyzz_add<T, true>(w, br);                     // W = W_L + W_R + B_R with W_j = B_j
      store_point_xyzz(heap_w, node, w);
      if (s == 0) continue;                // the root's B is not needed
    } else {
      const uint64_t child = heap0 + 2 * per + 2 * b;
      load_point_xyzz(a, heap_w, child);
      load_point_xyzz(br, heap_w, child + 1);
      xyzz_add<T, true>(a, br);
      load_point_xyzz(br, heap_b, child + 1);
      xyzz_add<T, true>(a, br);
      store_point_xyzz(heap_w, node, a);   // W = W_L + W_R + B_R
      if (s == 0) continue;
      load_point_xyzz(a, heap_b, child);
      xyzz_add<T, true>(a, br);                     // B_L + B_R
    }
    xyzz_dbl<T, true>(a, a);
    store_point_xyzz(heap_b, node, a);     // B = 2 (B_L + B_R)
  }
}

// BR, the lowest levels at once where there are many buckets: one thread takes
// 2^j adjacent leaves of a window by running sums (W = sum (i + 1) B_i, B = 2^j
// sum B_i), 2 additions a bucket (28 products) where the tree's levels take 51
// products per node.
template <class C>
__global__ void __launch_bounds__(kEcThreads, C::kTreeMinBlocks)
    msm_reduce_chunk_kernel(uint32_t j, uint32_t lb, uint32_t kb, uint32_t nk, const uint4 *bucket_sum,
                            const uint4 *pieces, const uint32_t *offsets, const MsmTotals *tot, uint4 *heap_w,
                            uint4 *heap_b) {
  using T = typename C::T;
  const uint32_t S = tot->seg_len, s = lb - j;
  const uint64_t per = 1ull << s, total = per * nk;
  for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < total;
       t += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t heap0 = (kb + (t >> s)) << lb, b = t & (per - 1);
    Xyzz<T> w, run, q;
    xyzz_set_inf(w);
    xyzz_set_inf(run);
#pragma unroll 1
    for (int i = (1 << j) - 1; i >= 0; --i) {
      load_bucket(q, bucket_sum, pieces, offsets, S, heap0 + (b << j) + i);
      xyzz_add<T, true>(run, q);
      xyzz_add<T, true>(w, run);
    }
    const uint64_t node = heap0 + per + b;
    store_point_xyzz(heap_w, node, w);
#pragma unroll 1
    for (uint32_t i = 0; i < j; ++i) xyzz_dbl<T, true>(run, run);
    store_point_xyzz(heap_b, node, run);
  }
}

// Coordinate `lane` of bucket b's sum (load_bucket, four lanes per point).
template <class T>
__device__ __forceinline__ void quad_load_bucket(uint32_t v[T::L], const uint4 *bucket_sum, const uint4 *pieces,
                                                 const uint32_t *offsets, uint32_t S, uint64_t b) {
  const uint32_t ob = offsets[b], ob1 = offsets[b + 1];
  if (ob1 == ob) fv_zero<T::L>(v);
  else if (ob / S == (ob1 - 1) / S) quad_load<T>(v, bucket_sum, b);
  else quad_load<T>(v, pieces, 2 * (uint64_t)(ob / S) + 1);
}

// The same level with four lanes for a node's W and four, of another warp, for
// its B: a level with few nodes takes the time of its dependent products, 8 or 7
// deep this way instead of 51 (BLS12-381: 65 us a level by one thread per node).
template <class C>
__global__ void __launch_bounds__(kEcThreads)
    msm_reduce_level_quad_kernel(uint32_t s, uint32_t lb, uint32_t kb, uint32_t nk, const uint4 *bucket_sum,
                                 const uint4 *pieces, const uint32_t *offsets, const MsmTotals *tot, uint4 *heap_w,
                                 uint4 *heap_b) {
  using T = typename C::T;
  constexpr int L = T::L;
  const uint32_t S = tot->seg_len;
  const uint64_t per = 1ull << s, total = per * nk;
  // warp pairs: eight nodes' W and B
  const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) / 32, warps = gridDim.x * (blockDim.x / 32);
  const bool is_b = warp & 1u, leaves = s + 1 == lb;
  if (is_b && s == 0) return;   // the root's B is not needed
  // every lane of the warp takes part in each step; a node past the end is a
  // copy of the last one that is not stored
  for (uint64_t t0 = 8ull * (warp / 2); t0 < total; t0 += 8ull * (warps / 2)) {
    const uint64_t t = t0 + (threadIdx.x % 32) / 4;
    const bool live = t < total;
    const uint64_t tc = live ? t : total - 1;
    const uint64_t k = kb + (tc >> s), b = tc & (per - 1);
    const uint64_t heap0 = k << lb, node = heap0 + per + b, child = heap0 + 2 * per + 2 * b;
    uint32_t v[L], w[L];
    if (leaves) {
      quad_load_bucket<T>(v, bucket_sum, pieces, offsets, S, heap0 + 2 * b);
      quad_load_bucket<T>(w, bucket_sum, pieces, offsets, S, heap0 + 2 * b + 1);
    } else {
      quad_load<T>(v, is_b ? heap_b : heap_w, child);
      quad_load<T>(w, is_b ? heap_b : heap_w, child + 1);
    }
    quad_add<T, true>(v, w);
    if (is_b) {
      if (!quad_all_inf<T>(v)) quad_dbl<T>(v);      // B = 2 (B_L + B_R)
    } else {
      if (!leaves) quad_load<T>(w, heap_b, child + 1);
      quad_add<T, true>(v, w);                            // W = W_L + W_R + B_R (leaves: W_j = B_j)
    }
    if (live) quad_store<T>(is_b ? heap_b : heap_w, node, v);
  }
}

// WM: sum_{kb <= k < ke} 2^(k c) W_k by Horner (then kb c doublings), in
// affine standard form; the whole MSM for [0, K).  With one bucket per
// window (c = 1) W_k is that bucket.  A chain of about 255 doublings: one warp
// with four lanes per point (every group of four does the same).
template <class C>
__global__ void msm_merge_kernel(uint32_t c, uint32_t kb, uint32_t ke, const uint4 *heap_w, const uint4 *bucket_sum,
                                 const uint4 *pieces, const uint32_t *offsets, const MsmTotals *tot,
                                 EcConst<typename C::T> kc, uint4 *result) {
  using T = typename C::T;
  constexpr int L = T::L;
  if (blockIdx.x != 0 || threadIdx.x >= 32) return;
  const uint32_t lb = c - 1, S = tot->seg_len;
  uint32_t v[L];
  fv_zero<L>(v);
  uint32_t doublings = 0;
  for (int k = (int)ke - 1; k >= (int)kb; --k) {
    uint32_t w[L];
    if (lb == 0) quad_load_bucket<T>(w, bucket_sum, pieces, offsets, S, (uint64_t)k);
    else quad_load<T>(w, heap_w, ((uint64_t)k << lb) + 1);
    // (empty windows above the first point: nothing to double)
    if (quad_all_inf<T>(v)) doublings = 0;
#pragma unroll 1
    for (uint32_t j = 0; j < doublings; ++j) quad_dbl<T, false>(v);
    quad_add<T, true>(v, w);
    doublings = c;
  }
  if (!quad_all_inf<T>(v)) {
#pragma unroll 1
    for (uint32_t j = 0; j < c * kb; ++j) quad_dbl<T, false>(v);
  }
  // affine: x = X ZZZ / (ZZ ZZZ), y = Y ZZ / (ZZ ZZZ)
  uint32_t z[L], t[L];
  quad_get<L>(z, v, 2);
  quad_get<L>(t, v, 3);
  const bool inf = fv_is_zero<L>(z);
  uint32_t inv[L], p[L];
  f_mul<T, true>(p, z, t);
  f_inverse<T>(inv, p, kc.r2);           // 0 for O
  quad_pick<L>(z, (threadIdx.x & 3) == 0, t, z);
  f_mul<T, true>(z, inv, z);
  f_mul<T, true>(z, z, v);
  T::redc(z, z);
  if (inf) fv_zero<L>(z);
  if (threadIdx.x < 2) T::store(result, threadIdx.x, z);
}

// Precomputed bases (fixed points reused across calls): for every point P_i
// the window copies 2^(k c) P_i, k < K, in affine Montgomery form at index
// k * stride + i; then all windows share one bucket set, and the
// per-window reduction trees and the window merge collapse into one window.
// The copies are normalised with one inversion per point (Montgomery's
// simultaneous inversion over its K copies).  Neither group has a point of
// order two, so no copy of a point other than O is O.  Invalid points are
// flagged and become O, as in msm_prepare_kernel.
constexpr uint32_t kMaxBaseWindows = 32;

template <class C>
__global__ void __launch_bounds__(kEcThreads) msm_bases_kernel(const uint4 *pts, uint64_t n, uint32_t c, uint32_t K,
                                                               uint64_t stride, EcConst<typename C::T> kc,
                                                               uint4 *bases, MsmTotals *tot) {
  using T = typename C::T;
  constexpr int L = T::L;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t x[L], y[L];
    T::load(x, pts, 2 * i);
    T::load(y, pts, 2 * i + 1);
    bool inf = fv_is_zero<L>(x) && fv_is_zero<L>(y);
    if (!inf) {
      bool ok = T::canonical(x) && T::canonical(y);
      if (ok) {
        T::mul(x, x, kc.r2);
        T::mul(y, y, kc.r2);
        uint32_t l[L], r[L];
        T::mul(l, y, y);
        T::mul(r, x, x);
        T::mul(r, r, x);
        T::add(r, r, kc.b3);
        ok = fv_equal<L>(l, r);
      }
      if (!ok) {
        atomicOr(&tot->err, (uint32_t)MSM_ERR_POINT);
        inf = true;
      }
    }
    if (inf) {
      fv_zero<L>(x);
      for (uint32_t k = 0; k < K; ++k) {
        T::store(bases, 2 * (k * stride + i), x);
        T::store(bases, 2 * (k * stride + i) + 1, x);
      }
      continue;
    }
    Xyzz<T> q[kMaxBaseWindows];
    uint32_t pre[kMaxBaseWindows][L];
    fv_copy<L>(q[0].X, x);
    fv_copy<L>(q[0].Y, y);
    fv_copy<L>(q[0].ZZ, kc.one);
    fv_copy<L>(q[0].ZZZ, kc.one);
    fv_copy<L>(pre[0], kc.one);  // ZZ ZZZ of the affine copy
    for (uint32_t k = 1; k < K; ++k) {
      q[k] = q[k - 1];
      for (uint32_t j = 0; j < c; ++j) xyzz_dbl<T>(q[k], q[k]);
      uint32_t z[L];
      T::mul(z, q[k].ZZ, q[k].ZZZ);
      T::mul(pre[k], pre[k - 1], z);  // prefix products of z_k = ZZ_k ZZZ_k
    }
    uint32_t inv[L];
    f_inverse<T>(inv, pre[K - 1], kc.r2);  // (z_0 ... z_{K-1})^-1
    for (int k = (int)K - 1; k >= 0; --k) {
      uint32_t ik[L], z[L], zi[L], ax[L], ay[L];
      if (k > 0) {
        T::mul(ik, inv, pre[k - 1]);        // z_k^-1
        T::mul(z, q[k].ZZ, q[k].ZZZ);
        T::mul(inv, inv, z);                // (z_0 ... z_{k-1})^-1
      } else {
        fv_copy<L>(ik, inv);
      }
      T::mul(zi, ik, q[k].ZZZ);             // ZZ^-1
      T::mul(ax, q[k].X, zi);
      T::mul(zi, ik, q[k].ZZ);              // ZZZ^-1
      T::mul(ay, q[k].Y, zi);
      T::store(bases, 2 * (k * stride + i), ax);
      T::store(bases, 2 * (k * stride + i) + 1, ay);
    }
  }
}

// ------------------------------------------------- fixed-base generation

// Comb table T[w][d] = d 2^(8 w) G (w < 32, d < 256), XYZZ, one thread per w.
template <class C>
__global__ void fixed_base_table_kernel(EcConst<typename C::T> kc, uint4 *table_xyzz) {
  using T = typename C::T;
  constexpr int L = T::L;
  const uint32_t w = threadIdx.x;
  if (blockIdx.x != 0 || w >= 32) return;
  Xyzz<T> base;
  T::mul(base.X, kc.gx, kc.r2);  // G in Montgomery form
  T::mul(base.Y, kc.gy, kc.r2);
  fv_copy<L>(base.ZZ, kc.one);
  fv_copy<L>(base.ZZZ, kc.one);
  for (uint32_t j = 0; j < 8 * w; ++j) xyzz_dbl<T>(base, base);
  Xyzz<T> acc;
  xyzz_set_inf(acc);
  store_point_xyzz(table_xyzz, 256 * w, acc);
  for (uint32_t d = 1; d < 256; ++d) {
    xyzz_add<T>(acc, base);
    store_point_xyzz(table_xyzz, 256 * w + d, acc);
  }
}

// Table entries to affine Montgomery form ((0, 0) for O).
template <class C>
__global__ void __launch_bounds__(kEcThreads) fixed_base_affine_kernel(EcConst<typename C::T> kc,
                                                                       const uint4 *table_xyzz, uint4 *table_aff) {
  using T = typename C::T;
  constexpr int L = T::L;
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 32 * 256) return;
  Xyzz<T> p;
  load_point_xyzz(p, table_xyzz, i);
  uint32_t x[L], y[L];
  if (xyzz_is_inf(p)) {
    fv_zero<L>(x);
    fv_zero<L>(y);
  } else {
    uint32_t t[L], inv[L], zi[L];
    T::mul(t, p.ZZ, p.ZZZ);
    f_inverse<T>(inv, t, kc.r2);
    T::mul(zi, inv, p.ZZZ);
    T::mul(x, p.X, zi);
    T::mul(zi, inv, p.ZZ);
    T::mul(y, p.Y, zi);
  }
  T::store(table_aff, 2 * i, x);
  T::store(table_aff, 2 * i + 1, y);
}

// P_n = t_n G = sum_w T[w][byte w of t_n], affine standard form.
template <class C>
__global__ void __launch_bounds__(kEcThreads) fixed_base_points_kernel(EcConst<typename C::T> kc,
                                                                       const uint4 *table_aff, const uint4 *ts,
                                                                       uint64_t n, uint4 *out) {
  using T = typename C::T;
  constexpr int L = T::L;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t t[8];
    fe_load_global(t, ts, i);
    Xyzz<T> acc;
    xyzz_set_inf(acc);
    for (uint32_t w = 0; w < 32; ++w) {
      const uint32_t d = (t[w >> 2] >> (8 * (w & 3))) & 0xffu;
      if (!d) continue;
      uint32_t x[L], y[L];
      T::load(x, table_aff, 2 * (256 * w + d));
      T::load(y, table_aff, 2 * (256 * w + d) + 1);
      xyzz_madd<T>(acc, x, y, kc.one);
    }
    uint32_t x[L], y[L];
    xyzz_to_affine_std<T>(x, y, acc, kc.r2);
    T::store(out, 2 * i, x);
    T::store(out, 2 * i + 1, y);
  }
}

// ------------------------------------------------------------------ host

// x = 2 x mod q on L-limb numbers (x < q < 2^(32 L - 1)).
void host_double_mod(uint32_t *x, const uint32_t *q, int L) {
  uint32_t carry = 0;
  for (int j = 0; j < L; ++j) {
    const uint32_t nc = x[j] >> 31;
    x[j] = (x[j] << 1) | carry;
    carry = nc;
  }
  bool ge = true;
  for (int j = L - 1; j >= 0; --j)
    if (x[j] != q[j]) {
      ge = x[j] > q[j];
      break;
    }
  if (ge) {
    int64_t br = 0;
    for (int j = 0; j < L; ++j) {
      const int64_t v = (int64_t)x[j] - q[j] + br;
      x[j] = (uint32_t)v;
      br = v < 0 ? -1 : 0;
    }
  }
}

// x = x + y mod q (x, y < q)
void host_add_mod(uint32_t *x, const uint32_t *y, const uint32_t *q, int L) {
  uint64_t c = 0;
  for (int j = 0; j < L; ++j) {
    c += (uint64_t)x[j] + y[j];
    x[j] = (uint32_t)c;
    c >>= 32;
  }
  bool ge = true;
  for (int j = L - 1; j >= 0; --j)
    if (x[j] != q[j]) {
      ge = x[j] > q[j];
      break;
    }
  if (ge) {
    int64_t br = 0;
    for (int j = 0; j < L; ++j) {
      const int64_t v = (int64_t)x[j] - q[j] + br;
      x[j] = (uint32_t)v;
      br = v < 0 ? -1 : 0;
    }
  }
}

template <class C>
void curve_modulus(uint32_t *q);
template <>
void curve_modulus<CurveBn254>(uint32_t *q) {
  using F = FieldBn254Fq;
  const uint32_t v[8] = {F::P0, F::P1, F::P2, F::P3, F::P4, F::P5, F::P6, F::P7};
  std::memcpy(q, v, sizeof(v));
}
template <>
void curve_modulus<CurveBls381>(uint32_t *q) {
  using F = FieldBls12381Fq;
  const uint32_t v[12] = {F::P0, F::P1, F::P2, F::P3, F::P4, F::P5, F::P6, F::P7, F::P8, F::P9, F::P10, F::P11};
  std::memcpy(q, v, sizeof(v));
}

// Generators (public curve parameters), standard form.
template <class C>
void curve_generator(uint32_t *gx, uint32_t *gy);
template <>
void curve_generator<CurveBn254>(uint32_t *gx, uint32_t *gy) {
  for (int j = 0; j < 8; ++j) gx[j] = gy[j] = 0;
  gx[0] = 1;
  gy[0] = 2;
}
template <>
void curve_generator<CurveBls381>(uint32_t *gx, uint32_t *gy) {
  const uint32_t x[12] = {0xdb22c6bbu, 0xfb3af00au, 0xf97a1aefu, 0x6c55e83fu, 0x171bac58u, 0xa14e3a3fu,
                          0x9774b905u, 0xc3688c4fu, 0x4fa9ac0fu, 0x2695638cu, 0x3197d794u, 0x17f1d3a7u};
  const uint32_t y[12] = {0x46c5e7e1u, 0x0caa2329u, 0xa2888ae4u, 0xd03cc744u, 0x2c04b3edu, 0x00db18cbu,
                          0xd5d00af6u, 0xfcf5e095u, 0x741d8ae4u, 0xa09e30edu, 0xe3aaa0f1u, 0x08b3f481u};
  std::memcpy(gx, x, sizeof(x));
  std::memcpy(gy, y, sizeof(y));
}

// Montgomery constants from the modulus alone: R = 2^(32 L) mod q by
// doubling 1, R^2 by doubling R, b R by adding R.
template <class C>
EcConst<typename C::T> make_const() {
  constexpr int L = C::T::L;
  uint32_t q[L];
  curve_modulus<C>(q);
  EcConst<typename C::T> k;
  for (int j = 0; j < L; ++j) k.one[j] = 0;
  k.one[0] = 1;
  for (int i = 0; i < 32 * L; ++i) host_double_mod(k.one, q, L);
  std::memcpy(k.r2, k.one, sizeof(k.one));
  for (int i = 0; i < 32 * L; ++i) host_double_mod(k.r2, q, L);
  for (int j = 0; j < L; ++j) k.b3[j] = 0;
  for (uint32_t i = 0; i < C::kB; ++i) host_add_mod(k.b3, k.one, q, L);
  curve_generator<C>(k.gx, k.gy);
  return k;
}

ntt_status cuda_st(cudaError_t e) {
  if (e == cudaSuccess) return NTT_OK;
  cudaGetLastError();
  return e == cudaErrorMemoryAllocation ? NTT_ERR_OOM : NTT_ERR_CUDA;
}

#define MSM_TRY(expr)               \
  do {                              \
    const ntt_status _s = (expr);   \
    if (_s != NTT_OK) return _s;    \
  } while (0)

ntt_status check_device(int *dev_out, int *sms) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return NTT_ERR_NO_DEVICE;
  }
  cudaDeviceProp prop;
  if (cudaGetDeviceProperties(&prop, dev) != cudaSuccess) {
    cudaGetLastError();
    return NTT_ERR_NO_DEVICE;
  }
  if (prop.major != 10 || prop.minor != 3) return NTT_ERR_NO_DEVICE;
  *dev_out = dev;
  *sms = prop.multiProcessorCount;
  return NTT_OK;
}

// K c >= S^BL + 1 (signed digits)
uint32_t num_windows(uint32_t c, uint32_t scalar_bits) { return (scalar_bits + 1 + c - 1) / c; }

// Window size minimising a modelled multiply count K (10 n + 26 2^(c-1)): one
// 10-product mixed addition per point and window and 26 products per bucket.  The
// 26 was fitted to an earlier reduction tree (a bucket now takes 28 products by
// running sums, a tree node 51 or a few four-lane steps), so small and middle sizes
// get windows up to 3 bits from their best; larger ones are at it.  GB300, uniform
// scalars, us with the default window and with the best one: BN254 10^4 766 (10)
// and 681 (11), 5 10^4 980 (13) and 858 (11), 2^20 3914 (16), 2^22 12312 (17), 2^24
// 44005 (20); BLS12-381 5 10^4 1853 (13) and 1559 (11), 2.5 10^5 3864 (14) and 2942
// (15), 2^20 7834 (16), 2^22 28724 (18) and 25074 (17).  Windows that leave the top
// one nearly full bits (11, 15, 17, 20) are the good ones.
uint32_t default_window(uint64_t n, uint32_t scalar_bits) {
  uint32_t best = 4;
  double best_cost = 1e300;
  for (uint32_t c = 4; c <= 21; ++c) {
    const double cost =
        (double)num_windows(c, scalar_bits) * (10.0 * (double)n + 26.0 * (double)(1u << (c - 1)));
    if (cost < best_cost) {
      best_cost = cost;
      best = c;
    }
  }
  return best;
}

// Entries per accumulation segment: the segments of a full call fill the GPU a
// whole number of times (1 to 8 times the threads that are resident, so that the
// last wave is not nearly empty), with 64 additions or more each where there
// are enough entries: longer segments cut the buckets that cross a segment end,
// hence the combine work.  At most 128 entries: calls with more than 8 waves of
// those (80 M entries for BN254) take as many waves as it needs, 22 at 2^24 points.
uint32_t segment_length(uint64_t max_n, uint32_t K, int sms, int blocks_per_sm) {
  const uint64_t entries = max_n * K, resident = (uint64_t)sms * blocks_per_sm * kEcThreads;
  const uint64_t waves = std::max<uint64_t>(1, std::min<uint64_t>(8, entries / (resident * 64)));
  return (uint32_t)std::max<uint64_t>(8, std::min<uint64_t>(128, (entries + waves * resident - 1) / (waves * resident)));
}

// Item list bases: level l of the long trees has at most segments / 4^(l + 1)
// + one head per bucket; a bucket with a node there crosses more than kShortSpan
// segment ends, and 4^l at least.
uint64_t item_bases(uint64_t segments, uint32_t base[kLongLevels]) {
  uint64_t total = 0, per = 4;
  for (int l = 0; l < kLongLevels; ++l) {
    base[l] = (uint32_t)total;
    total += segments / per + segments / std::max<uint64_t>(kShortSpan, per / 4) + 1;
    per *= 4;
  }
  return total;
}

uint32_t curve_scalar_bits(int curve) { return curve == MSM_CURVE_BLS12_381_G1 ? 255u : 254u; }
uint32_t curve_elem_bytes(int curve) { return curve == MSM_CURVE_BLS12_381_G1 ? 48u : 32u; }

}  // namespace
}  // namespace gb300ntt

using namespace gb300ntt;

struct msm_plan_s {
  int device = 0;
  int sms = 0;
  int curve = 0;
  uint32_t elem_bytes = 32;   // one coordinate
  uint64_t max_n = 0;
  uint32_t c = 0, K = 0, S = 0;
  uint64_t nb = 0;            // K 2^(c-1) buckets
  uint64_t max_segments = 0;
  uint32_t num_tiles = 0;
  EcConst<FqBn254> k254;
  EcConst<FqBls381> k381;
  uint4 *pts_m = nullptr;     // max_n points, Montgomery form
  uint32_t *counts = nullptr, *offsets = nullptr, *cursor = nullptr, *tile_sums = nullptr;
  MsmTotals *tot = nullptr;
  uint32_t *sorted = nullptr;
  CombineLists lists{};       // work lists of the combine kernels
  uint4 *bucket_sum = nullptr, *pieces = nullptr;   // nb and 2 max_segments XYZZ points
  uint4 *heap_w = nullptr, *heap_b = nullptr;       // nb XYZZ points each
  uint4 *bases = nullptr;     // precomputed window copies: K x max_n points (msm_plan_set_bases)
  uint64_t bases_n = 0;       // points set (0: none)
  uint64_t device_bytes = 0;
};

namespace {

void free_plan(msm_plan p) {
  void *bufs[] = {p->pts_m, p->counts, p->offsets, p->cursor, p->tile_sums, p->tot, p->sorted,
                  p->lists.crossing, p->lists.items, p->bucket_sum, p->pieces, p->heap_w, p->heap_b, p->bases};
  for (void *b : bufs)
    if (b) cudaFree(b);
  delete p;
}

template <class T>
ntt_status alloc(T **ptr, uint64_t bytes, uint64_t *total) {
  *total += bytes;
  return cuda_st(cudaMalloc((void **)ptr, bytes ? bytes : 16));
}

int grid_for(uint64_t work, int threads, int sms, int per_sm) {
  const uint64_t blocks = (work + threads - 1) / threads;
  return (int)std::max<uint64_t>(1, std::min<uint64_t>(blocks, (uint64_t)sms * per_sm));
}

template <class C>
const EcConst<typename C::T> &plan_const(const msm_plan p);
template <>
const EcConst<FqBn254> &plan_const<CurveBn254>(const msm_plan p) { return p->k254; }
template <>
const EcConst<FqBls381> &plan_const<CurveBls381>(const msm_plan p) { return p->k381; }

// The launch sequence of one MSM (all on stream st).
// flat: the plan's precomputed bases (pt unused): one bucket set for all
// windows, the points gathered from the window copies, one reduction tree
// and no window merge.
template <class C>
ntt_status enqueue_msm(msm_plan p, const uint4 *sc, const uint4 *pt, uint64_t n, uint32_t kb, uint32_t ke,
                       uint4 *result, cudaStream_t st, bool flat = false) {
  const auto &k = plan_const<C>(p);
  const int sms = p->sms;
  const uint32_t lb = p->c - 1;
  const uint64_t nb = flat ? (1ull << lb) : p->nb;           // buckets in use
  const uint32_t num_tiles = (uint32_t)((nb + kScanTile - 1) / kScanTile);
  const uint4 *pts = flat ? p->bases : p->pts_m;
  const uint32_t tree_kb = flat ? 0 : kb, tree_ke = flat ? 1 : ke;
  MSM_TRY(cuda_st(cudaMemsetAsync(p->counts, 0, nb * 4, st)));
  // keep the error bits (read by msm_poll_error), reset the rest
  MSM_TRY(cuda_st(cudaMemsetAsync(p->tot, 0, offsetof(MsmTotals, err), st)));
  if (n > 0) {
    if (!flat)
      msm_prepare_kernel<C><<<grid_for(n, kEcThreads, sms, 16), kEcThreads, 0, st>>>(pt, n, k, p->pts_m, p->tot);
    msm_count_kernel<C><<<grid_for(n, 256, sms, 8), 256, 0, st>>>(sc, n, p->c, kb, ke, flat, p->counts, p->tot);
  }
  scan_reduce_kernel<<<num_tiles, kScanThreads, 0, st>>>(p->counts, nb, p->tile_sums);
  scan_tiles_kernel<<<1, kScanThreads, 0, st>>>(p->tile_sums, num_tiles, nb, p->offsets,
                                                (uint32_t)std::max<uint64_t>(1, p->max_segments - 1), p->tot);
  scan_apply_kernel<<<num_tiles, kScanThreads, 0, st>>>(p->counts, nb, p->tile_sums, p->offsets, p->cursor);
  if (n > 0) {
    const uint32_t sweep = flat ? p->K : (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(p->K, kSweepEntries / n));
    msm_scatter_kernel<<<grid_for(n, 256, sms, 5), 256, 0, st>>>(sc, n, p->c, kb, ke, sweep,
                                                                 flat ? (uint32_t)p->max_n : 0u, p->cursor,
                                                                 p->sorted);
    const uint64_t segs = std::min<uint64_t>((n * p->K + 7) / 8, p->max_segments);
    const int g = grid_for(segs, kEcThreads, sms, C::kMinBlocks);
    const uint64_t used = (uint64_t)(tree_ke - tree_kb) << lb;
    msm_accumulate_kernel<C><<<g, kEcThreads, 0, st>>>(pts, p->sorted, p->offsets, nb, used, k, p->tot, p->lists,
                                                       p->bucket_sum, p->pieces);
    const int gt = grid_for(segs, kEcThreads, sms, C::kTreeMinBlocks);
    msm_combine_kernel<C><<<gt, kEcThreads, 0, st>>>(p->tot, p->lists.crossing, p->pieces);
    // a bucket holds at most n entries of one window (flat: of all of them), so
    // it crosses at most this many segment ends; empty levels exit at once
    // (segments of 8 entries at least, at most max_segments of them; the grid is
    // for K windows in a range of fewer too: each bucket adds an item to its
    // segments', and going round the loop again for those doubles a level's time)
    const uint64_t most = flat ? n * p->K : n;
    const uint64_t max_span = std::min<uint64_t>((most + 7) / 8, p->max_segments);
    uint64_t step = 1;
    for (int l = 0; l < kLongLevels && max_span > kShortSpan && step <= max_span; ++l, step *= 4)
      msm_combine_long_kernel<C><<<grid_for(4 * (max_span / (4 * step) + 1) * p->K, kEcThreads, sms, 4), kEcThreads, 0,
                                   st>>>(p->offsets, nb, p->tot, p->lists, l, p->pieces);
  }
  // leaves of the tree that one thread takes at once: while that still fills
  // the GPU about once
  int s = (int)lb - 1;
  if (tree_ke > tree_kb) {
    const uint64_t leaves = ((uint64_t)(tree_ke - tree_kb)) << lb;
    uint32_t j = 0;
    while (j + 1 < lb && (leaves >> (j + 1)) * 4 >= (uint64_t)sms * C::kTreeMinBlocks * kEcThreads * 3) ++j;
    if (j >= 2) {
      msm_reduce_chunk_kernel<C><<<grid_for(leaves >> j, kEcThreads, sms, C::kTreeMinBlocks), kEcThreads, 0, st>>>(
          j, lb, tree_kb, tree_ke - tree_kb, p->bucket_sum, p->pieces, p->offsets, p->tot, p->heap_w, p->heap_b);
      s = (int)(lb - j) - 1;
    }
  }
  for (; s >= 0 && tree_ke > tree_kb; --s) {
    const uint64_t work = ((uint64_t)(tree_ke - tree_kb)) << s;
    if (work <= (uint64_t)sms * kQuadNodesPerSm) {
      msm_reduce_level_quad_kernel<C><<<grid_for(8 * work, kEcThreads, sms, 8), kEcThreads, 0, st>>>(
          (uint32_t)s, lb, tree_kb, tree_ke - tree_kb, p->bucket_sum, p->pieces, p->offsets, p->tot, p->heap_w,
          p->heap_b);
      continue;
    }
    msm_reduce_level_kernel<C><<<grid_for(work, kEcThreads, sms, C::kTreeMinBlocks), kEcThreads, 0, st>>>(
        (uint32_t)s, lb, tree_kb, tree_ke - tree_kb, p->bucket_sum, p->pieces, p->offsets, p->tot, p->heap_w,
        p->heap_b);
  }
  msm_merge_kernel<C><<<1, 32, 0, st>>>(p->c, tree_kb, tree_ke, p->heap_w, p->bucket_sum, p->pieces, p->offsets,
                                        p->tot, k, result);
  return cuda_st(cudaGetLastError());
}

std::mutex g_fb_mutex;
std::map<std::pair<int, int>, uint4 *> g_fb_tables;  // (device, curve) -> affine comb table (8192 points)

template <class C>
ntt_status fixed_base_table(int dev, int curve, const EcConst<typename C::T> &kc, cudaStream_t st, uint4 **out) {
  std::lock_guard<std::mutex> lock(g_fb_mutex);
  auto it = g_fb_tables.find({dev, curve});
  if (it != g_fb_tables.end()) {
    *out = it->second;
    return NTT_OK;
  }
  const uint64_t eb = 4ull * C::T::L;  // bytes per coordinate
  uint4 *xyzz = nullptr, *aff = nullptr;
  MSM_TRY(cuda_st(cudaMalloc((void **)&xyzz, 8192ull * 4 * eb)));
  ntt_status s = cuda_st(cudaMalloc((void **)&aff, 8192ull * 2 * eb));
  if (s == NTT_OK) {
    fixed_base_table_kernel<C><<<1, 32, 0, st>>>(kc, xyzz);
    fixed_base_affine_kernel<C><<<8192 / kEcThreads, kEcThreads, 0, st>>>(kc, xyzz, aff);
    s = cuda_st(cudaGetLastError());
    if (s == NTT_OK) s = cuda_st(cudaStreamSynchronize(st));
  }
  cudaFree(xyzz);
  if (s != NTT_OK) {
    if (aff) cudaFree(aff);
    return s;
  }
  g_fb_tables[{dev, curve}] = aff;
  *out = aff;
  return NTT_OK;
}

template <class C>
ntt_status fixed_base(int dev, int sms, int curve, const uint4 *ts, uint64_t n, uint4 *out, cudaStream_t st) {
  const EcConst<typename C::T> kc = make_const<C>();
  uint4 *table = nullptr;
  MSM_TRY(fixed_base_table<C>(dev, curve, kc, st, &table));
  fixed_base_points_kernel<C><<<grid_for(n, kEcThreads, sms, 16), kEcThreads, 0, st>>>(kc, table, ts, n, out);
  return cuda_st(cudaGetLastError());
}

bool curve_valid(int curve) { return curve == MSM_CURVE_BN254_G1 || curve == MSM_CURVE_BLS12_381_G1; }

}  // namespace

extern "C" {

ntt_status msm_point_bytes(msm_curve curve, uint32_t *bytes) {
  if (!bytes || !curve_valid((int)curve)) return NTT_ERR_INVALID_ARG;
  *bytes = 2 * curve_elem_bytes((int)curve);
  return NTT_OK;
}

ntt_status msm_plan_create(msm_plan *out, msm_curve curve, uint64_t max_n, uint32_t window_bits) {
  if (!out) return NTT_ERR_INVALID_ARG;
  *out = nullptr;
  if (!curve_valid((int)curve)) return NTT_ERR_INVALID_ARG;
  if (max_n > MSM_MAX_POINTS) return NTT_ERR_UNSUPPORTED;
  if (window_bits > 22) return NTT_ERR_UNSUPPORTED;
  const uint32_t sbits = curve_scalar_bits((int)curve);
  const uint32_t c = window_bits ? window_bits : default_window(std::max<uint64_t>(max_n, 1), sbits);
  // sorted entries are counted in 32 bits (with room for one segment past
  // the end); point indices stay below 2^31, bit 31 carries the digit sign
  if (max_n * num_windows(c, sbits) >= (1ull << 32) - 256) return NTT_ERR_UNSUPPORTED;
  int dev = 0, sms = 0;
  MSM_TRY(check_device(&dev, &sms));
  msm_plan p = new (std::nothrow) msm_plan_s();
  if (!p) return NTT_ERR_OOM;
  p->device = dev;
  p->sms = sms;
  p->curve = (int)curve;
  p->elem_bytes = curve_elem_bytes((int)curve);
  p->max_n = max_n;
  p->c = c;
  p->K = num_windows(c, sbits);
  p->S = segment_length(max_n, p->K, sms,
                        p->curve == MSM_CURVE_BLS12_381_G1 ? CurveBls381::kMinBlocks : CurveBn254::kMinBlocks);
  p->nb = (uint64_t)p->K << (c - 1);
  const uint64_t entries = max_n * p->K;
  p->max_segments = (entries + p->S - 1) / p->S + 1;
  p->num_tiles = (uint32_t)((p->nb + kScanTile - 1) / kScanTile);
  if (p->curve == MSM_CURVE_BLS12_381_G1) p->k381 = make_const<CurveBls381>();
  else p->k254 = make_const<CurveBn254>();
  const uint64_t pb = 2ull * p->elem_bytes, xb = 4ull * p->elem_bytes;  // affine and XYZZ point bytes
  uint64_t &tb = p->device_bytes;
  ntt_status s = NTT_OK;
  if (s == NTT_OK) s = alloc(&p->pts_m, max_n * pb, &tb);
  if (s == NTT_OK) s = alloc(&p->counts, p->nb * 4, &tb);
  if (s == NTT_OK) s = alloc(&p->offsets, (p->nb + 1) * 4, &tb);
  if (s == NTT_OK) s = alloc(&p->cursor, p->nb * 4, &tb);
  if (s == NTT_OK) s = alloc(&p->tile_sums, (uint64_t)p->num_tiles * 4, &tb);
  if (s == NTT_OK) s = alloc(&p->tot, sizeof(MsmTotals), &tb);
  if (s == NTT_OK) s = alloc(&p->sorted, entries * 4, &tb);
  if (s == NTT_OK) s = alloc(&p->lists.crossing, p->max_segments * 4, &tb);
  if (s == NTT_OK) s = alloc(&p->lists.items, item_bases(p->max_segments, p->lists.item_base) * 4, &tb);
  if (s == NTT_OK) s = alloc(&p->bucket_sum, p->nb * xb, &tb);
  if (s == NTT_OK) s = alloc(&p->pieces, 2 * p->max_segments * xb, &tb);
  if (s == NTT_OK) s = alloc(&p->heap_w, p->nb * xb, &tb);
  if (s == NTT_OK) s = alloc(&p->heap_b, p->nb * xb, &tb);
  if (s == NTT_OK) s = cuda_st(cudaMemset(p->tot, 0, sizeof(MsmTotals)));
  if (s != NTT_OK) {
    free_plan(p);
    return s;
  }
  *out = p;
  return NTT_OK;
}

ntt_status msm_plan_info(msm_plan plan, msm_plan_desc *out) {
  if (!plan || !out) return NTT_ERR_INVALID_ARG;
  out->max_n = plan->max_n;
  out->window_bits = plan->c;
  out->num_windows = plan->K;
  out->segment_length = plan->S;
  out->reserved = 0;
  out->device_bytes = plan->device_bytes;
  return NTT_OK;
}

ntt_status msm_plan_destroy(msm_plan plan) {
  if (!plan) return NTT_ERR_INVALID_ARG;
  cudaDeviceSynchronize();
  free_plan(plan);
  return NTT_OK;
}

ntt_status msm_execute(msm_plan p, const void *d_scalars, const void *d_points, uint64_t n, void *d_result,
                       ntt_stream stream) {
  gb300ntt::NvtxRange range("msm_execute");
  if (!p || !d_result || ((uintptr_t)d_result % 16)) return NTT_ERR_INVALID_ARG;
  if (n > p->max_n) return NTT_ERR_INVALID_ARG;
  const uintptr_t pa = p->curve == MSM_CURVE_BLS12_381_G1 ? 16 : 32;  // one 128- or 256-bit access
  if ((uintptr_t)d_result % pa) return NTT_ERR_INVALID_ARG;
  if (n > 0 && (!d_scalars || !d_points || ((uintptr_t)d_scalars % 32) || ((uintptr_t)d_points % pa)))
    return NTT_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const uint4 *sc = (const uint4 *)d_scalars;
  const uint4 *pt = (const uint4 *)d_points;
  if (p->curve == MSM_CURVE_BLS12_381_G1)
    return enqueue_msm<CurveBls381>(p, sc, pt, n, 0, p->K, (uint4 *)d_result, st);
  return enqueue_msm<CurveBn254>(p, sc, pt, n, 0, p->K, (uint4 *)d_result, st);
}

ntt_status msm_execute_windows(msm_plan p, const void *d_scalars, const void *d_points, uint64_t n,
                               uint32_t window_begin, uint32_t window_end, void *d_result, ntt_stream stream) {
  if (!p || window_begin > window_end || window_end > p->K) return NTT_ERR_INVALID_ARG;
  if (window_begin == 0 && window_end == p->K) return msm_execute(p, d_scalars, d_points, n, d_result, stream);
  // the same argument checks as msm_execute
  if (!d_result || n > p->max_n) return NTT_ERR_INVALID_ARG;
  const uintptr_t pa = p->curve == MSM_CURVE_BLS12_381_G1 ? 16 : 32;
  if ((uintptr_t)d_result % pa) return NTT_ERR_INVALID_ARG;
  if (n > 0 && (!d_scalars || !d_points || ((uintptr_t)d_scalars % 32) || ((uintptr_t)d_points % pa)))
    return NTT_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const uint4 *sc = (const uint4 *)d_scalars;
  const uint4 *pt = (const uint4 *)d_points;
  if (p->curve == MSM_CURVE_BLS12_381_G1)
    return enqueue_msm<CurveBls381>(p, sc, pt, n, window_begin, window_end, (uint4 *)d_result, st);
  return enqueue_msm<CurveBn254>(p, sc, pt, n, window_begin, window_end, (uint4 *)d_result, st);
}

ntt_status msm_plan_set_bases(msm_plan p, const void *d_points, uint64_t n, ntt_stream stream) {
  if (!p || n > p->max_n) return NTT_ERR_INVALID_ARG;
  const uintptr_t pa = p->curve == MSM_CURVE_BLS12_381_G1 ? 16 : 32;
  if (n > 0 && (!d_points || ((uintptr_t)d_points % pa))) return NTT_ERR_INVALID_ARG;
  if (p->K > kMaxBaseWindows || (uint64_t)p->K * p->max_n >= (1ull << 31)) return NTT_ERR_UNSUPPORTED;
  if (!p->bases) {
    const uint64_t bytes = (uint64_t)p->K * std::max<uint64_t>(p->max_n, 1) * 2 * p->elem_bytes;
    MSM_TRY(cuda_st(cudaMalloc((void **)&p->bases, bytes)));
    p->device_bytes += bytes;
  }
  cudaStream_t st = (cudaStream_t)stream;
  p->bases_n = 0;
  if (n > 0) {
    const uint4 *pt = (const uint4 *)d_points;
    if (p->curve == MSM_CURVE_BLS12_381_G1)
      msm_bases_kernel<CurveBls381><<<grid_for(n, kEcThreads, p->sms, 8), kEcThreads, 0, st>>>(
          pt, n, p->c, p->K, p->max_n, p->k381, p->bases, p->tot);
    else
      msm_bases_kernel<CurveBn254><<<grid_for(n, kEcThreads, p->sms, 8), kEcThreads, 0, st>>>(
          pt, n, p->c, p->K, p->max_n, p->k254, p->bases, p->tot);
    MSM_TRY(cuda_st(cudaGetLastError()));
  }
  p->bases_n = n;
  return NTT_OK;
}

ntt_status msm_execute_bases(msm_plan p, const void *d_scalars, uint64_t n, void *d_result, ntt_stream stream) {
  if (!p || !d_result || n > p->bases_n || (n == 0 && !p->bases)) return NTT_ERR_INVALID_ARG;
  const uintptr_t pa = p->curve == MSM_CURVE_BLS12_381_G1 ? 16 : 32;
  if (((uintptr_t)d_result % pa) || (n > 0 && (!d_scalars || ((uintptr_t)d_scalars % 32))))
    return NTT_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const uint4 *sc = (const uint4 *)d_scalars;
  if (p->curve == MSM_CURVE_BLS12_381_G1)
    return enqueue_msm<CurveBls381>(p, sc, nullptr, n, 0, p->K, (uint4 *)d_result, st, true);
  return enqueue_msm<CurveBn254>(p, sc, nullptr, n, 0, p->K, (uint4 *)d_result, st, true);
}

ntt_status msm_poll_error(msm_plan p, uint32_t *flags) {
  if (!p || !flags) return NTT_ERR_INVALID_ARG;
  // the calls may run on non-blocking streams: wait for all of them
  MSM_TRY(cuda_st(cudaDeviceSynchronize()));
  MsmTotals t;
  MSM_TRY(cuda_st(cudaMemcpy(&t, p->tot, sizeof(t), cudaMemcpyDeviceToHost)));
  *flags = t.err;
  const uint32_t zero = 0;
  MSM_TRY(cuda_st(cudaMemcpy(&p->tot->err, &zero, sizeof(zero), cudaMemcpyHostToDevice)));
  return NTT_OK;
}

ntt_status msm_fixed_base(msm_curve curve, const void *d_scalars, uint64_t n, void *d_points, ntt_stream stream) {
  if (!curve_valid((int)curve)) return NTT_ERR_INVALID_ARG;
  if (n == 0) return NTT_OK;
  const uintptr_t pa = curve == MSM_CURVE_BLS12_381_G1 ? 16 : 32;
  if (!d_scalars || !d_points || ((uintptr_t)d_scalars % 32) || ((uintptr_t)d_points % pa))
    return NTT_ERR_INVALID_ARG;
  int dev = 0, sms = 0;
  MSM_TRY(check_device(&dev, &sms));
  cudaStream_t st = (cudaStream_t)stream;
  const uint4 *ts = (const uint4 *)d_scalars;
  if (curve == MSM_CURVE_BLS12_381_G1)
    return fixed_base<CurveBls381>(dev, sms, (int)curve, ts, n, (uint4 *)d_points, st);
  return fixed_base<CurveBn254>(dev, sms, (int)curve, ts, n, (uint4 *)d_points, st);
}

}  // extern "C"
