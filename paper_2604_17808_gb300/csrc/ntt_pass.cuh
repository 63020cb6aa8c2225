// ntt_pass.cuh -- one pass of the multi-pass (four-/six-step) NTT on sm_103a.
//
// Decomposition (the paper's 3-step / 5-step NTT, Sec. 3.3.2, Fig. 5b-c and
// Eq. 1, in the standard Cooley-Tukey index map): N = S_0 * S_1 * ... *
// S_{P-1}.  Write the input index as n = sum_j n_j * N / (S_0 ... S_j), so
// digit n_0 has the largest stride.  Then
//
//   pass 0:      for every value of the other digits, a size-S_0 DFT over
//                n_0 (input stride N/S_0); the result for output digit k_0
//                is stored at k_0 + S_0 * rev(n_1..n_{P-1}), i.e. the
//                untransformed digits are written in reversed significance
//                (this is the transpose of the four-step method);
//   pass j >= 1: in place, buffer position q + Mp*n_j + M*o with
//                Mp = S_0...S_{j-1}, M = Mp*S_j: each input is multiplied by
//                the inter-pass twiddle omega_M^(n_j*q) (the element-wise
//                "TF" product between the matrix steps of Eq. 1), then a
//                size-S_j DFT over n_j.  q is the already transformed low
//                part of the output index, o the untransformed rest.
//
// After the last pass the buffer holds X in natural order.  Coset and
// inverse scale factors are folded into the same per-element multipliers.
//
// Work split on the GPU: a group of threads owns a tile of 2^tl elements in
// shared memory = 2^(tl - logs) sub-transforms with consecutive sub-transform
// index, and each thread 2^pl of its elements at a time.  The DIF (Gentleman-Sande)
// radix-2 network over every sub-transform of the tile runs in rounds of up to
// pl stages: in a round a thread owns the 2^pl elements that differ in the
// round's index bits, so its stages need no barrier between them; barriers
// stand between rounds only.
//   first round: the thread copies its own elements from global memory
//                (cp.async, no registers) and multiplies them by the input
//                multiplier (pass >= 1: omega_M^(n q)), with no barrier before
//                its first butterfly: a warp starts as soon as its own copies
//                have landed;
//   last round:  stages pl-1..0; the last two in registers (their twiddles are
//                1 and omega_4: one multiply per 4 elements), written straight
//                to global memory at the bit-reversed output index (this undoes
//                the DIF output order).
// All index arithmetic takes logs, tl and pl at run time, so that the hot code
// is one butterfly body (about 230 instructions) whatever the pass.  What
// bounds a pass is the IMAD pipe: a butterfly is one mul_split (fp256.cuh; 90
// or 100 IMAD-pipe instructions of four cycles) beside which additions, shared
// memory (8 128-bit accesses) and twiddle loads (64 bytes) are issued.
// Values stay in [0, 2p) or [0, 3p) (fp256.cuh) from the first butterfly to the
// last store.
//
// The tile is XOR-swizzled on 16-byte chunks: chunk 2e + h of element e is
// stored at (2e + h) ^ swz(e), linear over GF(2) in the bits of e.  For every
// round above (any set of adjacent index bits, either thread order) eight
// consecutive lanes differ in three index bits whose columns are independent,
// so no access has a bank conflict.
#pragma once

#include <cstdint>

#include "fp256.cuh"

namespace gb300ntt {

// Tile of one pass launch: 2^tl elements, 2^pl per thread (2^(tl - pl) threads
// per CTA), sub-transforms of 2^logs points, logs <= tl, 1 <= pl <= 3.
struct TileShape {
  uint32_t logs, tl, pl;
};

// A CTA runs one tile, or several independent ones side by side: `groups` of
// 2^(tl - pl) threads, each with a tile of its own and a named barrier.  Three
// kernel instances:
//   up to 128 threads  one tile per CTA, 6 CTAs per SM for 1024-element tiles
//                      (32 KiB and another KiB that each CTA reserves);
//   896 threads        seven 1024-element tiles with 8 elements per thread,
//                      one CTA per SM, for passes that are one wave this way:
//                      the 1024 tiles of a 2^20-point pass took two waves of
//                      six (99 and 80 us a pass against 90 and 75; on 152 SMs
//                      this is the one power of two with such passes).  With many
//                      waves the CTAs that come and go on their own are faster
//                      (2^24: 2.9 against 3.1 ms);
//   256 threads        one 2048-element tile, 3 CTAs per SM.
constexpr uint32_t kGroups = 7;
constexpr uint32_t kGroupThreads = 128;
constexpr uint32_t kGroupBytes = 32u << 10;   // a 1024-element tile

template <int MAXT>
struct TileBounds {
  static constexpr int kMinBlocks = MAXT == 896 ? 1 : MAXT == 256 ? 3 : 6;
};

// Barrier of one group of `threads` threads; of the CTA where it has one group
// only (a barrier number in a register would claim all sixteen for the CTA).
template <bool GROUPED>
__device__ __forceinline__ void group_sync(uint32_t group, uint32_t threads) {
  if constexpr (GROUPED) asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "r"(threads) : "memory");
  else __syncthreads();
}

constexpr int kMaxPassLog = 11;                    // sub-transforms up to 2048 points

enum PassMode : int {
  kModeInner = 0,     // pass j >= 1: in place, 2-D input multiplier table [S][Mp]
  kModeFirst = 1,     // pass 0 without input multiplier
  kModeFirstPre = 2,  // pass 0 with a per-n_0 input multiplier table [S]
};

// At most this many passes per transform (NTT_MAX_PASSES of the C ABI: the
// matrix path splits 2^28 into ten passes of at most 2^3 points).
constexpr int kMaxPasses = 12;

struct PassArgs {
  const uint4 *src;      // input elements (2 x uint4 each)
  uint4 *dst;            // output elements
  const uint4 *mul;      // input multipliers (Montgomery form) or nullptr
  const uint4 *dft_tw;   // omega_S^i, i < S/2, 64 bytes each: the residues A, B of mul_split
  const uint4 *post;     // output multipliers indexed by output position, or nullptr
                         // (last pass of a coset inverse: s^-n)
  uint64_t num_sub;      // number of sub-transforms in the pass, N / S
  uint32_t log_mp;       // inner: log2 Mp; first: log2(N / S)
  uint32_t num_digits;   // first: P - 1 untransformed digits to reverse
  uint8_t digit_log[kMaxPasses];    // first: log2 S_j of digit j (j = 1..P-1) at index j-1
  uint8_t digit_shift[kMaxPasses];  // first: log2(S_1 ... S_{j-1}) at index j-1
  uint64_t n_vec;        // elements of src, dst and post (debug bounds checks)
  uint64_t n_mul;        // entries of mul (debug bounds checks)
  uint32_t *dbg_err;     // device error word the debug checks report to
};

// Debug builds (NTT_DEBUG): an index is checked against the extent recorded
// for its buffer; out of range, NTT_ERR_BOUNDS goes to the plan's error word
// and the access is skipped (no trap: the context stays usable).  Release
// builds compile the checks away.
#ifdef NTT_DEBUG
__device__ __forceinline__ bool dbg_in(const PassArgs &a, uint64_t idx, uint64_t n) {
  if (idx < n) return true;
  if (a.dbg_err) atomicCAS(a.dbg_err, 0u, 8u /* NTT_ERR_BOUNDS */);
  return false;
}
#else
__device__ __forceinline__ constexpr bool dbg_in(const PassArgs &, uint64_t, uint64_t) { return true; }
#endif

// Output row of pass 0 for untransformed digits d (their significance reversed).
__device__ __forceinline__ uint64_t reverse_digits(const PassArgs &a, uint64_t d) {
  uint64_t rest = d, rev = 0;
#pragma unroll 1
  for (int j = (int)a.num_digits - 1; j >= 0; --j) {
    const uint64_t nj = rest & ((1ull << a.digit_log[j]) - 1);
    rest >>= a.digit_log[j];
    rev |= nj << a.digit_shift[j];
  }
  return rev;
}

// ------------------------------------------------------------- swizzle
// Chunk c = 2e + h (16-byte half h of tile element e) is stored at
// c ^ swz(e), swz(e) = XOR of f_b over the set bits b >= 2 of e, with
// f_2..f_10 = 1,7,3,5,7,1,3,5,1 (3-bit columns).  Packed as three 8-entry
// lookup tables (3 bits per entry) for e bits 2-4, 5-7 and 8-10.
constexpr uint32_t swz_lut(uint32_t fa, uint32_t fb, uint32_t fc) {
  uint32_t lut = 0;
  for (uint32_t x = 0; x < 8; ++x) {
    const uint32_t v = ((x & 1) ? fa : 0) ^ ((x & 2) ? fb : 0) ^ ((x & 4) ? fc : 0);
    lut |= v << (3 * x);
  }
  return lut;
}
constexpr uint32_t kSwzLut0 = swz_lut(1, 7, 3);
constexpr uint32_t kSwzLut1 = swz_lut(5, 7, 1);
constexpr uint32_t kSwzLut2 = swz_lut(3, 5, 1);

__device__ __forceinline__ uint32_t swz(uint32_t e) {
  const uint32_t x0 = (e >> 2) & 7, x1 = (e >> 5) & 7, x2 = (e >> 8) & 7;
  return ((kSwzLut0 >> (3 * x0)) ^ (kSwzLut1 >> (3 * x1)) ^ (kSwzLut2 >> (3 * x2))) & 7u;
}

// What the tile routine asks of a field's elements (this one: 256-bit fields,
// eight words): their place in the tile, moves, and arithmetic on lazy values.
// `tile` is the tile's shared-memory address, `off` a byte offset that is linear
// over GF(2) in the bits of the element index; the accesses keep their program
// order (a thread reads back what it wrote).
template <class F>
struct Elem256 {
  static constexpr int W = 8;
  static constexpr uint32_t kTileRow = 32;        // tile offsets of 2^tl elements are below kTileRow 2^tl
  static constexpr bool kPreByPosition = false;   // pass-0 multipliers are indexed by n_0

  // low half of element e; the high half is at the offset ^ 16
  __device__ static __forceinline__ uint32_t tile_offset(uint32_t e) { return ((e << 1) ^ swz(e)) << 4; }

  __device__ static __forceinline__ void tile_store(uint32_t tile, uint32_t off, uint32_t, const uint32_t a[8]) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(tile + off), "r"(a[0]), "r"(a[1]), "r"(a[2]),
                 "r"(a[3])
                 : "memory");
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(tile + (off ^ 16u)), "r"(a[4]), "r"(a[5]),
                 "r"(a[6]), "r"(a[7])
                 : "memory");
  }

  __device__ static __forceinline__ void tile_load(uint32_t r[8], uint32_t tile, uint32_t off, uint32_t) {
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(tile + off)
                 : "memory");
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(tile + (off ^ 16u))
                 : "memory");
  }

  // Global -> shared copy of one element without registers, through L2 (data
  // that another CTA wrote earlier in the same launch is read coherently).
  __device__ static __forceinline__ void copy_async(uint32_t tile, uint32_t off, uint32_t, const uint4 *base,
                                                    uint64_t elem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tile + off), "l"(base + 2 * elem) : "memory");
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tile + (off ^ 16u)), "l"(base + 2 * elem + 1)
                 : "memory");
  }

  // entry w of the DFT table: the residues of mul_split
  __device__ static __forceinline__ void load_twiddle(uint32_t A[8], uint32_t B[8], const uint4 *dft_tw, uint32_t w) {
    const char *p = reinterpret_cast<const char *>(dft_tw) + (w << 6);
    asm("ld.global.nc.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=r"(A[0]), "=r"(A[1]), "=r"(A[2]), "=r"(A[3]), "=r"(A[4]), "=r"(A[5]), "=r"(A[6]), "=r"(A[7])
        : "l"(p));
    asm("ld.global.nc.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8+32];"
        : "=r"(B[0]), "=r"(B[1]), "=r"(B[2]), "=r"(B[3]), "=r"(B[4]), "=r"(B[5]), "=r"(B[6]), "=r"(B[7])
        : "l"(p));
  }
  __device__ static __forceinline__ void load(uint32_t r[8], const uint4 *base, uint64_t e) {
    fe_load_global(r, base, e);
  }
  __device__ static __forceinline__ void store(uint4 *base, uint64_t e, const uint32_t a[8]) {
    fe_store_global(base, e, a);
  }

  __device__ static __forceinline__ void add(uint32_t r[8], const uint32_t a[8], const uint32_t b[8]) {
    add_lazy<F>(r, a, b);
  }
  __device__ static __forceinline__ void sub(uint32_t r[8], const uint32_t a[8], const uint32_t b[8]) {
    sub_lazy<F>(r, a, b);
  }
  __device__ static __forceinline__ void mul_twiddle(uint32_t r[8], const uint32_t x[8], const uint32_t A[8],
                                                     const uint32_t B[8]) {
    mul_split<F>(r, x, A, B);
  }
  // w: a table entry in Montgomery form; below 2p
  __device__ static __forceinline__ void mul_in(uint32_t x[8], const uint32_t w[8]) { mont_mul_lazy<F>(x, w, x); }
  // canonical results
  __device__ static __forceinline__ void mul_out(uint32_t x[8], const uint32_t w[8]) { mont_mul<F>(x, w, x); }
  __device__ static __forceinline__ void finish(uint32_t x[8]) { reduce_lazy<F>(x, x); }
};

__device__ __forceinline__ void tile_copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// ------------------------------------------------- checked tile accesses
// Tile offsets and twiddle indices are computed at run time from the tile shape:
// debug builds check them against the tile and the table of 2^logs points, as they
// do the vectors (out of range: NTT_ERR_BOUNDS, the access skipped, zero loaded).
template <int W>
__device__ __forceinline__ void words_zero(uint32_t *x) {
#pragma unroll
  for (int k = 0; k < W; ++k) x[k] = 0;
}

template <class El>
__device__ __forceinline__ void tile_get(const PassArgs &a, const TileShape &s, uint32_t *x, uint32_t tile,
                                         uint32_t off) {
  if (dbg_in(a, off, El::kTileRow << s.tl)) El::tile_load(x, tile, off, s.tl);
  else words_zero<El::W>(x);
}

template <class El>
__device__ __forceinline__ void tile_put(const PassArgs &a, const TileShape &s, uint32_t tile, uint32_t off,
                                         const uint32_t *x) {
  if (dbg_in(a, off, El::kTileRow << s.tl)) El::tile_store(tile, off, s.tl, x);
}

template <class El>
__device__ __forceinline__ void twiddle_get(const PassArgs &a, const TileShape &s, uint32_t *A, uint32_t *B,
                                            const uint4 *dft_tw, uint32_t w) {
  if (dbg_in(a, w, s.logs > 1 ? 1u << (s.logs - 1) : 1u)) {
    El::load_twiddle(A, B, dft_tw, w);
  } else {
    words_zero<El::W>(A);
    words_zero<El::W>(B);
  }
}

// ----------------------------------------------------------- butterflies

// A thread's 2^pl elements of one round: tile offset of the first, and the
// offset differences of the private index bits (element j: base ^ the set bits'
// differences).
struct Private {
  uint32_t base, d0, d1, d2;
};

__device__ __forceinline__ uint32_t private_offset(const Private &v, uint32_t j) {
  return v.base ^ ((j & 1u) ? v.d0 : 0u) ^ ((j & 2u) ? v.d1 : 0u) ^ ((j & 4u) ? v.d2 : 0u);
}

// Private bits: the r round bits T .. T + r - 1 and, when r < pl, the top pl -
// r bits of the tile index.
template <class El>
__device__ __forceinline__ Private private_set(const TileShape &s, uint32_t e, uint32_t T, uint32_t r) {
  const uint32_t top = s.tl - s.pl;   // private bit k >= r is index bit top + k
  Private v;
  v.base = El::tile_offset(e);
  v.d0 = El::tile_offset(1u << (r > 0 ? T : top));
  v.d1 = El::tile_offset(1u << (r > 1 ? T + 1 : top + 1));
  v.d2 = El::tile_offset(1u << (r > 2 ? T + 2 : top + 2));
  return v;
}

// Private stages T + hi - 1 down to T + lo: pairs that differ in private bit
// b, twiddle omega_S^((p mod h) S / 2h) with h = 2^(T + b), p the position in
// the sub-transform; low = its bits below T.  (dft_tw is a.dft_tw in a register: the
// batched kernel's `a` is in global memory, and a load of the pointer before every
// twiddle made lists of 8 small jobs 2% to 8% slower.)
template <class El>
__device__ __forceinline__ void private_stages(const PassArgs &a, uint32_t tile, const uint4 *dft_tw,
                                               const TileShape &s, const Private &v, uint32_t T, int hi, int lo,
                                               uint32_t low) {
#pragma unroll 1
  for (int b = hi - 1; b >= lo; --b) {
    const uint32_t mask = (1u << b) - 1u, sh = s.logs - 1u - (T + (uint32_t)b);
    const uint32_t db = b == 0 ? v.d0 : b == 1 ? v.d1 : v.d2;
#pragma unroll 1
    for (uint32_t i = 0; i < (1u << (s.pl - 1)); ++i) {
      const uint32_t j = (i & mask) | ((i & ~mask) << 1);
      const uint32_t c = private_offset(v, j);
      const uint32_t w = (low | ((j & mask) << T)) << sh;
      uint32_t x[El::W], y[El::W], d[El::W];
      if (T == 0 && (j & mask) == 0) {   // twiddle 1, for every thread
        tile_get<El>(a, s, x, tile, c);
        tile_get<El>(a, s, y, tile, c ^ db);
        El::sub(d, x, y);
        El::add(x, x, y);
        tile_put<El>(a, s, tile, c, x);
        tile_put<El>(a, s, tile, c ^ db, d);
        continue;
      }
      uint32_t A[El::W], B[El::W];
      twiddle_get<El>(a, s, A, B, dft_tw, w);
      tile_get<El>(a, s, x, tile, c);
      tile_get<El>(a, s, y, tile, c ^ db);
      El::sub(d, x, y);
      El::add(x, x, y);
      tile_put<El>(a, s, tile, c, x);
      El::mul_twiddle(d, d, A, B);
      tile_put<El>(a, s, tile, c ^ db, d);
    }
  }
}

// One output element: canonical, times the output multiplier where there is
// one.
template <class El>
__device__ __forceinline__ void store_output(const PassArgs &a, uint64_t pos, uint32_t x[El::W]) {
  if (!dbg_in(a, pos, a.n_vec)) return;
  if (a.post) {   // uniform across the grid
    uint32_t w[El::W];
    El::load(w, a.post, pos);
    El::mul_out(x, w);
  } else {
    El::finish(x);
  }
  El::store(a.dst, pos, x);
}

// Global position of element n of sub-transform d (pass input; the in-place
// inner passes write output k of d to the same formula).
template <int MODE>
__device__ __forceinline__ uint64_t elem_pos(const PassArgs &a, uint32_t logs, uint64_t d, uint32_t n) {
  if constexpr (MODE == kModeInner) {
    const uint64_t q = d & ((1ull << a.log_mp) - 1), o = d >> a.log_mp;
    return q + ((uint64_t)n << a.log_mp) + (o << (a.log_mp + logs));
  } else {
    return d + ((uint64_t)n << a.log_mp);
  }
}

// Process tile `tile` of one pass.  All threads of the group call this (t: index
// in the group); the caller separates two tiles on the same shared memory with a
// barrier.
template <class El, int MODE, bool GROUPED>
__device__ __forceinline__ void pass_tile(const PassArgs &a, const TileShape s, uint64_t tile, uint32_t smem,
                                          uint32_t t, uint32_t group) {
  const uint32_t logs = s.logs, pl = s.pl, threads = 1u << (s.tl - pl);
  const uint32_t logg = s.tl - logs;                 // log2 of the tile's sub-transforms
  const uint64_t d0 = tile << logg;
  const uint32_t last = min(pl, logs);               // stages of the last round
  uint32_t T = logs;                                 // stages left

  // ---- first round: sub-transforms fastest across the threads (a warp reads
  // runs of consecutive elements)
  {
    const uint32_t r = logs > last ? min(pl, logs - last) : last;
    T -= r;
    const uint32_t gbits = logg - (pl - r);
    const uint32_t dl = t & ((1u << gbits) - 1u), low = t >> gbits;
    const Private v = private_set<El>(s, (dl << logs) | low, T, r);
    const uint32_t count = 1u << pl, rmask = (1u << r) - 1u;
    // element j is input low + ((j mod 2^r) << T) of sub-transform d; with r =
    // pl (sub-transforms of 2^pl points, and of 2^(2 pl) or more) its position is
    // linear in j
    const uint64_t dfirst = d0 + dl, step = 1ull << (a.log_mp + T);
    const bool linear = r == pl;
    auto sub_of = [&](uint32_t j) { return dfirst + ((uint64_t)(j >> r) << gbits); };
    uint64_t pos = elem_pos<MODE>(a, logs, dfirst, low);
#pragma unroll 1
    for (uint32_t j = 0; j < count; ++j, pos += step) {
      const uint64_t d = linear ? dfirst : sub_of(j);
      if (!linear) pos = elem_pos<MODE>(a, logs, d, low | ((j & rmask) << T));
      if (d >= a.num_sub) continue;
      const uint32_t c = private_offset(v, j);
      if (dbg_in(a, pos, a.n_vec) && dbg_in(a, c, El::kTileRow << s.tl)) {
        El::copy_async(smem, c, s.tl, a.src, pos);
      } else {
        uint32_t z[El::W] = {};
        tile_put<El>(a, s, smem, c, z);
      }
    }
    if constexpr (MODE != kModeFirst) {
      // the multiplier of the next element is on its way during a product
      const uint64_t q_mask = (1ull << a.log_mp) - 1;
      auto mul_of = [&](uint64_t d, uint32_t n) {
        if constexpr (MODE == kModeInner) return ((uint64_t)n << a.log_mp) + (d & q_mask);
        else return El::kPreByPosition ? elem_pos<MODE>(a, logs, d, n) : (uint64_t)n;
      };
      const uint64_t wstep = MODE == kModeInner || El::kPreByPosition ? step : 1ull << T;
      uint64_t wi = mul_of(dfirst, low);
      uint32_t w[El::W], next[El::W];
      auto load_mul = [&](uint32_t *x, uint32_t j) {
        const uint64_t d = linear ? dfirst : sub_of(j);
        if (!linear) wi = mul_of(d, low | ((j & rmask) << T));
        if (d < a.num_sub && dbg_in(a, wi, a.n_mul)) {
          El::load(x, a.mul, wi);
        } else {
#pragma unroll
          for (int k = 0; k < El::W; ++k) x[k] = 0;
        }
        wi += wstep;
      };
      load_mul(next, 0);
      tile_copy_wait();
#pragma unroll 1
      for (uint32_t j = 0; j < count; ++j) {
        const uint32_t c = private_offset(v, j);
#pragma unroll
        for (int k = 0; k < El::W; ++k) w[k] = next[k];
        if (j + 1 < count) load_mul(next, j + 1);
        uint32_t x[El::W];
        tile_get<El>(a, s, x, smem, c);
        El::mul_in(x, w);
        tile_put<El>(a, s, smem, c, x);
      }
    } else {
      tile_copy_wait();
    }
    if (T > 0) private_stages<El>(a, smem, a.dft_tw, s, v, T, (int)r, 0, low);
  }

  // ---- middle rounds
#pragma unroll 1
  while (T > last) {
    const uint32_t r = min(pl, T - last);
    T -= r;
    group_sync<GROUPED>(group, threads);
    const uint32_t low = t & ((1u << T) - 1u);
    const Private v = private_set<El>(s, low | ((t >> T) << (T + r)), T, r);
    private_stages<El>(a, smem, a.dft_tw, s, v, T, (int)r, 0, low);
  }

  // ---- last round: stages last - 1 .. 0; inner passes vary sub-transforms
  // fastest across threads (consecutive q), pass 0 the output index: either
  // way a warp writes runs of consecutive elements
  if (T > 0) group_sync<GROUPED>(group, threads);
  const uint32_t tbits = logs - last, gbits = logg - (pl - last);
  const uint32_t dl = MODE == kModeInner ? t & ((1u << gbits) - 1u) : t >> tbits;
  const uint32_t tt = MODE == kModeInner ? t >> gbits : t & ((1u << tbits) - 1u);
  const uint32_t p0 = tbits ? (__brev(tt) >> (32 - tbits)) << last : 0u;
  const Private v = private_set<El>(s, (dl << logs) | p0, 0, last);
  const uint32_t lmask = (1u << last) - 1u, half = 1u << (logs - 1);
  private_stages<El>(a, smem, a.dft_tw, s, v, 0, (int)last, last >= 2 ? 2 : 1, 0);
  const uint32_t unit = last >= 2 ? 4u : 2u;
#pragma unroll 1
  for (uint32_t j = 0; j < (1u << pl); j += unit) {
    const uint64_t d = d0 + dl + ((uint64_t)(j >> last) << gbits);
    const uint32_t c = private_offset(v, j);
    const uint32_t k = __brev(p0 | (j & lmask)) >> (32 - logs);   // output of the group's first position
    uint64_t out = 0;
    uint32_t sh = 0;
    if constexpr (MODE == kModeInner) {
      out = elem_pos<MODE>(a, logs, d, 0);
      sh = a.log_mp;
    } else if (d < a.num_sub) {
      out = reverse_digits(a, d) << logs;
    }
    uint32_t x0[El::W], x1[El::W], y[El::W];
    if (last >= 2) {
      uint32_t x2[El::W], x3[El::W];
      {
        uint32_t A[El::W], B[El::W];   // omega_4 = omega_S^(S/4)
        twiddle_get<El>(a, s, A, B, a.dft_tw, half >> 1);
        tile_get<El>(a, s, x1, smem, c ^ v.d0);
        tile_get<El>(a, s, x3, smem, c ^ v.d0 ^ v.d1);
        El::sub(y, x1, x3);
        El::add(x1, x1, x3);
        El::mul_twiddle(x3, y, A, B);
      }
      tile_get<El>(a, s, x0, smem, c);
      tile_get<El>(a, s, x2, smem, c ^ v.d1);
      El::sub(y, x0, x2);
      El::add(x0, x0, x2);
      El::add(x2, y, x3);
      El::sub(x3, y, x3);
      if (d < a.num_sub) {
        store_output<El>(a, out + ((uint64_t)(k + (half >> 1)) << sh), x2);
        store_output<El>(a, out + ((uint64_t)(k + (half >> 1) + half) << sh), x3);
      }
    } else {
      tile_get<El>(a, s, x0, smem, c);
      tile_get<El>(a, s, x1, smem, c ^ v.d0);
    }
    El::sub(y, x0, x1);
    El::add(x0, x0, x1);
    if (d < a.num_sub) {
      store_output<El>(a, out + ((uint64_t)k << sh), x0);
      store_output<El>(a, out + ((uint64_t)(k + half) << sh), y);
    }
  }
}

// ------------------------------------------------------------ pass kernel

// Programmatic dependent launch (the passes are launched with it): each thread
// waits here until the previous launch has completed and its memory is visible.
// No launch is released early (no griddepcontrol.launch_dependents): the next
// one's CTAs then start as ours retire.  A release at the start let waiting CTAs
// of the next launches fill the free slots of the SMs, unevenly, so that every
// launch after ran on few of them: 2^17 points 125 us a transform back to back
// and 62 alone with the release before this wait, 2^18 points 69 us with it after
// the wait and 50 without.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class F, int MODE, int MAXT>
__global__ void __launch_bounds__(MAXT, TileBounds<MAXT>::kMinBlocks)
    ntt_pass_kernel(const __grid_constant__ PassArgs a, const TileShape s, uint32_t tiles) {
  extern __shared__ uint4 smem[];
  pdl_wait();
  const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem);
  if constexpr (MAXT == 896) {
    const uint32_t group = threadIdx.x / kGroupThreads, tile = blockIdx.x * kGroups + group;
    if (tile < tiles)
      pass_tile<Elem256<F>, MODE, true>(a, s, tile, base + group * kGroupBytes, threadIdx.x % kGroupThreads, group);
  } else {
    pass_tile<Elem256<F>, MODE, false>(a, s, blockIdx.x, base, threadIdx.x, 0);
  }
}

}  // namespace gb300ntt
