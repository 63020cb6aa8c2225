// ntt_wide.cuh -- NTT over the 377- and 753-bit fields (12 and 24 words).
//
// The paper evaluates its NTT at 256, 377 and 753 bits (Sec. 4.3.1,
// Tab. 3).  These fields run the tile routine of ntt_pass.cuh (four-/six-step
// passes, digit-reversed first pass, in-place inner passes with the inter-pass
// twiddle on load, bit-reversed store) over elements of their own
// (fp_wide.cuh): 12 or 24 consecutive 32-bit words in memory (48 or 96 bytes),
// standard form, canonical; constants are in Montgomery form, so mul(x, c R) =
// x c.
//
// Tile: 2^10 (377) or 2^9 (753) elements, 48 KiB, up to 8 elements per thread,
// 4 CTAs of 128 (377) or 64 threads (753: 200 registers each) per SM.  The
// 16-byte chunks of an element lie one tile length apart; within a chunk row the
// elements are XOR-swizzled by the same columns as the 256-bit tile, so eight
// consecutive lanes never meet in a bank.
//
// Multipliers: the first pass's table (mode kModeFirstPre) is indexed by
// the input position (the coset factors s^i, or N^-1 for a one-pass
// inverse), the inner passes' by (n, q) as in ntt_pass.cuh, and the
// optional output table `post` by the output position (s^-i in the last
// pass of a coset inverse).
#pragma once

#include <cstdint>

#include "fp_wide.cuh"
#include "ntt_pass.cuh"

namespace gb300ntt {

template <class F>
struct WideShape {
  static constexpr int kLog = F::L == 12 ? 10 : 9;   // largest tile: 2^kLog elements
  static constexpr int kThreads = 128;               // largest CTA
  static constexpr int kMinBlocks = F::L == 12 ? 4 : 2;   // of such CTAs (106 and 201 registers per thread)
  static constexpr int kBytes = (1 << kLog) * F::L * 4;
};

// Constants the host computes from the modulus (kernel argument).
template <class F>
struct WideConst {
  uint32_t one[F::L];   // R mod p, R = 2^(32 L)
  uint32_t r2[F::L];    // R^2 mod p
};

template <class F>
struct ElemWide {
  static constexpr int W = F::L;
  static constexpr uint32_t kTileRow = 16;
  static constexpr bool kPreByPosition = true;

  __device__ static __forceinline__ uint32_t tile_offset(uint32_t e) {
    return ((e & ~7u) | (((e << 1) & 6u) ^ swz(e))) << 4;
  }
  __device__ static __forceinline__ void tile_store(uint32_t tile, uint32_t off, uint32_t tl, const uint32_t *a) {
#pragma unroll
    for (int k = 0; k < W / 4; ++k)
      asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(tile + off + ((uint32_t)k << (tl + 4))),
                   "r"(a[4 * k]), "r"(a[4 * k + 1]), "r"(a[4 * k + 2]), "r"(a[4 * k + 3])
                   : "memory");
  }
  __device__ static __forceinline__ void tile_load(uint32_t *r, uint32_t tile, uint32_t off, uint32_t tl) {
#pragma unroll
    for (int k = 0; k < W / 4; ++k)
      asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                   : "=r"(r[4 * k]), "=r"(r[4 * k + 1]), "=r"(r[4 * k + 2]), "=r"(r[4 * k + 3])
                   : "r"(tile + off + ((uint32_t)k << (tl + 4)))
                   : "memory");
  }
  __device__ static __forceinline__ void copy_async(uint32_t tile, uint32_t off, uint32_t tl, const uint4 *base,
                                                    uint64_t elem) {
#pragma unroll
    for (int k = 0; k < W / 4; ++k)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tile + off + ((uint32_t)k << (tl + 4))),
                   "l"(base + elem * (W / 4) + k)
                   : "memory");
  }
  __device__ static __forceinline__ void load(uint32_t *r, const uint4 *base, uint64_t e) {
#pragma unroll
    for (int k = 0; k < W / 4; ++k) {
      const uint4 v = __ldg(base + e * (W / 4) + k);
      r[4 * k] = v.x; r[4 * k + 1] = v.y; r[4 * k + 2] = v.z; r[4 * k + 3] = v.w;
    }
  }
  __device__ static __forceinline__ void store(uint4 *base, uint64_t e, const uint32_t *a) {
#pragma unroll
    for (int k = 0; k < W / 4; ++k)
      base[e * (W / 4) + k] = make_uint4(a[4 * k], a[4 * k + 1], a[4 * k + 2], a[4 * k + 3]);
  }
  __device__ static __forceinline__ void load_twiddle(uint32_t *A, uint32_t *B, const uint4 *dft_tw, uint32_t w) {
    load(A, dft_tw, 2 * (uint64_t)w);
    load(B, dft_tw, 2 * (uint64_t)w + 1);
  }
  __device__ static __forceinline__ void add(uint32_t *r, const uint32_t *a, const uint32_t *b) {
    wide_add_lazy<F>(r, a, b);
  }
  __device__ static __forceinline__ void sub(uint32_t *r, const uint32_t *a, const uint32_t *b) {
    wide_sub_lazy<F>(r, a, b);
  }
  __device__ static __forceinline__ void mul_twiddle(uint32_t *r, const uint32_t *x, const uint32_t *A,
                                                     const uint32_t *B) {
    wide_mul_split<F>(r, x, A, B);
  }
  __device__ static __forceinline__ void mul_in(uint32_t *x, const uint32_t *w) { wide_mul<F>(x, w, x); }
  __device__ static __forceinline__ void mul_out(uint32_t *x, const uint32_t *w) { wide_mul<F>(x, w, x); }
  __device__ static __forceinline__ void finish(uint32_t *x) { wide_reduce_once<F, 0>(x); }
};

template <class F, int MODE>
__global__ void __launch_bounds__(WideShape<F>::kThreads, WideShape<F>::kMinBlocks)
    wide_pass_kernel(const __grid_constant__ PassArgs a, const TileShape s) {
  extern __shared__ uint4 wide_smem[];
  pdl_wait();
  pass_tile<ElemWide<F>, MODE, false>(a, s, blockIdx.x, (uint32_t)__cvta_generic_to_shared(wide_smem), threadIdx.x, 0);
}

// ---------------------------------------------------------------- tables

// out = base^e (Montgomery form in and out; e as 32-bit words), one thread.
template <class F>
__device__ void wide_pow(uint32_t out[F::L], const uint32_t base[F::L], const uint32_t *e, int words,
                         const WideConst<F> &C) {
  constexpr int L = F::L;
  uint32_t acc[L], b[L];
  for (int j = 0; j < L; ++j) {
    acc[j] = C.one[j];
    b[j] = base[j];
  }
  for (int w = 0; w < words; ++w)
    for (int bit = 0; bit < 32; ++bit) {
      if ((e[w] >> bit) & 1) wide_mul<F>(acc, acc, b);
      wide_mul<F>(b, b, b);
    }
  for (int j = 0; j < L; ++j) out[j] = acc[j];
}

// Per transform size 2^log_m: writes to `k` (Montgomery form, L limbs each)
//   k[0..31]   omega_M^(2^b)      k[32..63]  omega_M^-(2^b)
//   k[64]      M^-1               k[65]      R mod p (one)
// One thread.
template <class F>
__global__ void wide_constants_kernel(uint32_t *k, uint32_t log_m, const WideConst<F> C) {
  constexpr int L = F::L;
  uint32_t g[L], root[L], w[L];
  for (int j = 0; j < L; ++j) g[j] = j == 0 ? (uint32_t)F::kGenerator : 0u;
  wide_mul<F>(g, g, C.r2);                  // generator in Montgomery form
  uint32_t exp_c[L];   // (p - 1) / 2^32
  for (int j = 0; j < L; ++j) exp_c[j] = j + 1 < L ? F::p(j + 1) : 0u;
  wide_pow<F>(root, g, exp_c, L, C);           // primitive 2^32-th root
  for (uint32_t i = log_m; i < 32; ++i) wide_mul<F>(root, root, root);   // omega_M
  for (int j = 0; j < L; ++j) w[j] = root[j];
  for (int b = 0; b < 32; ++b) {
    for (int j = 0; j < L; ++j) k[b * L + j] = w[j];
    wide_mul<F>(w, w, w);
  }
  // omega^-1 = omega^(M - 1)
  const uint32_t e[1] = {(uint32_t)((1ull << log_m) - 1)};
  uint32_t inv[L];
  wide_pow<F>(inv, root, e, 1, C);
  for (int b = 0; b < 32; ++b) {
    for (int j = 0; j < L; ++j) k[(32 + b) * L + j] = inv[j];
    wide_mul<F>(inv, inv, inv);
  }
  // M^-1 = p - (p - 1) / M, then Montgomery form
  uint32_t mw[L];
  {
    uint32_t pm1[L];
    for (int j = 0; j < L; ++j) pm1[j] = F::p(j);
    pm1[0] -= 1;   // p is odd: no borrow
    for (int j = 0; j < L; ++j) {
      const uint64_t lo = pm1[j], hi = j + 1 < L ? pm1[j + 1] : 0u;
      mw[j] = (uint32_t)(((hi << 32) | lo) >> log_m);
    }
    int64_t br = 0;
    for (int j = 0; j < L; ++j) {
      const int64_t v = (int64_t)F::p(j) - mw[j] + br;
      mw[j] = (uint32_t)v;
      br = v >> 32;
    }
  }
  uint32_t mi[L];
  wide_mul<F>(mi, mw, C.r2);
  for (int j = 0; j < L; ++j) k[64 * L + j] = mi[j];
  for (int j = 0; j < L; ++j) k[65 * L + j] = C.one[j];
}

// The coset shift s for wide_table_kernel.  Reads s from k[64] (L words,
// standard form, 0 < s < p: the host checks) and writes
//   k[0..31]  s^(2^b)     k[32..63]  s^-(2^b)     k[65]  R mod p (one)
// (Montgomery form; s^-1 = s^(p-2) by Fermat's little theorem).  One thread.
template <class F>
__global__ void wide_coset_constants_kernel(uint32_t *k, const WideConst<F> C) {
  constexpr int L = F::L;
  uint32_t s[L], w[L];
  for (int j = 0; j < L; ++j) s[j] = k[64 * L + j];
  wide_mul<F>(s, s, C.r2);
  uint32_t em2[L];   // p - 2
  int64_t br = -2;
  for (int j = 0; j < L; ++j) {
    const int64_t v = (int64_t)F::p(j) + br;
    em2[j] = (uint32_t)v;
    br = v >> 32;
  }
  uint32_t inv[L];
  wide_pow<F>(inv, s, em2, L, C);
  for (int j = 0; j < L; ++j) w[j] = s[j];
  for (int b = 0; b < 32; ++b) {
    for (int j = 0; j < L; ++j) k[b * L + j] = w[j];
    wide_mul<F>(w, w, w);
  }
  for (int b = 0; b < 32; ++b) {
    for (int j = 0; j < L; ++j) k[(32 + b) * L + j] = inv[j];
    wide_mul<F>(inv, inv, inv);
  }
  for (int j = 0; j < L; ++j) k[65 * L + j] = C.one[j];
}

// out[n * Mp + q] = init * base^(n q)  (two_d: the inter-pass table), or
// out[i] = init * base^i; ladder[b] = base^(2^b); a null ladder gives the
// constant table out[i] = init.  With `split` an entry is the pair of residues
// of wide_mul_split (base^i 2^(16 L) and base^i 2^(32 L) mod p).
template <class F>
__global__ void wide_table_kernel(uint4 *out, uint32_t log_mp, const uint32_t *ladder, const uint32_t *init,
                                  uint64_t count, int two_d, int split) {
  constexpr int L = F::L;
  for (uint64_t idx = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; idx < count;
       idx += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t e = !ladder ? 0 : two_d ? (idx >> log_mp) * (idx & ((1ull << log_mp) - 1)) : idx;
    uint32_t acc[L];
#pragma unroll
    for (int j = 0; j < L; ++j) acc[j] = init[j];
    for (int b = 0; b < 32 && (e >> b) != 0; ++b) {
      if ((e >> b) & 1) {
        uint32_t w[L];
#pragma unroll
        for (int j = 0; j < L; ++j) w[j] = ladder[b * L + j];
        wide_mul<F>(acc, acc, w);
      }
    }
    if (split) {
      uint32_t half[L], low[L];
#pragma unroll
      for (int j = 0; j < L; ++j) half[j] = j == L / 2 ? 1u : 0u;
      wide_mul<F>(low, acc, half);
      ElemWide<F>::store(out, 2 * idx, low);
      ElemWide<F>::store(out, 2 * idx + 1, acc);
    } else {
      ElemWide<F>::store(out, idx, acc);
    }
  }
}

}  // namespace gb300ntt
