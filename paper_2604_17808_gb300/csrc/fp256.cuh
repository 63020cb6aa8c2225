// fp256.cuh -- 255-bit prime-field arithmetic for sm_103a, 8 x 32-bit limbs.
//
// The paper's arithmetic baseline ("radix Mont", Sec. 2.3.2 and Tab. 1): a
// field element is D = 8 32-bit digits; a multiplication is an O(D^2) digit
// product with carry propagation followed by an O(D^2) Montgomery reduction.
// On a GPU the carry chains are native (mad.lo.cc / madc.hi.cc on the
// integer multiply-add pipe), so this is the hot loop of the butterfly path.
//
// Conventions used throughout the library:
//   * element = uint32_t[8], limb 0 least significant;
//   * data stays in STANDARD form end to end; every constant operand
//     (twiddles, coset powers, N^-1) is stored in MONTGOMERY form c*2^256, so
//     mont_mul(x, c*2^256) = x*c mod p is again standard.  No conversion
//     passes are needed at the ABI boundary;
//   * values at the ABI are canonical, in [0, p), and operations take and leave
//     canonical values where their comment does not say otherwise; inside a
//     transform pass values are lazy, in [0, 2p) or [0, 3p) (below).
//
// mont_mul is Montgomery multiplication by operand scanning (CIOS; Koc, Acar,
// Kaliski, "Analyzing and comparing Montgomery multiplication algorithms",
// IEEE Micro 1996), radix 2^32, over two accumulators.  What bounds it is the
// IMAD (fmaheavy) pipe: a 32 x 32 -> 64 bit multiply-add with carry takes four
// of its cycles per warp (measured on GB300: 30 of them per SM and clock,
// half the rate of a 32-bit one), if its two accumulator words are an aligned
// register pair.  Products a_i b_j of even i start at even word columns and
// those of odd i at odd ones, so the running value is kept as
//
//   T = sum_k E_k 2^(32 k) + sum_k O_k 2^(32 (k + 1))
//
// with the even products added into E's pairs and the odd ones into O's: no
// product straddles two pairs.  Dividing by 2^32 swaps the roles: the new E is
// the old O, the new O is the old E without its two low words, and the old
// E_1 is added into column 0, its carry entering the next odd chain.
// Measured (268 M dependent products of BN254 Fr): 66 G/s against 57-58 G/s
// for one accumulator, whose odd products ptxas split into low and high
// halves; 136 instead of 171 IMAD-pipe instructions per product.
#pragma once

#include <cstdint>

namespace gb300ntt {

constexpr uint32_t neg_inv_u32(uint32_t p0) {
  // Newton iteration for p0^-1 mod 2^32 (p0 odd); each step doubles the
  // number of correct low bits, starting from 3 (p0 * p0 = 1 mod 8).
  uint32_t inv = p0;
  for (int i = 0; i < 5; ++i) inv *= 2u - p0 * inv;
  return 0u - inv;
}

// BLS12-381 scalar field r (255 bits, 2-adicity 32, generator 7).
struct FieldBls12381Fr {
  static constexpr int kId = 0;
  static constexpr uint32_t kLazy = 2;       // values inside a transform pass stay below kLazy p
  static constexpr bool kSubtract = true;   // redc_row subtracts T_0 r
  static constexpr uint32_t P0 = 0x00000001u, P1 = 0xffffffffu, P2 = 0xfffe5bfeu, P3 = 0x53bda402u,
                            P4 = 0x09a1d805u, P5 = 0x3339d808u, P6 = 0x299d7d48u, P7 = 0x73eda753u;
  static constexpr uint32_t NP = neg_inv_u32(P0);
};

// BN254 scalar field r (254 bits, 2-adicity 28, generator 5).
struct FieldBn254Fr {
  static constexpr int kId = 1;
  static constexpr uint32_t kLazy = 3;
  static constexpr bool kSubtract = false;
  static constexpr uint32_t P0 = 0xf0000001u, P1 = 0x43e1f593u, P2 = 0x79b97091u, P3 = 0x2833e848u,
                            P4 = 0x8181585du, P5 = 0xb85045b6u, P6 = 0xe131a029u, P7 = 0x30644e72u;
  static constexpr uint32_t NP = neg_inv_u32(P0);
};

static_assert(FieldBls12381Fr::P0 * (0u - FieldBls12381Fr::NP) == 1u, "NP");
static_assert(FieldBn254Fr::P0 * (0u - FieldBn254Fr::NP) == 1u, "NP");
static_assert(FieldBls12381Fr::P0 == 1u && FieldBls12381Fr::P1 == 0xffffffffu && FieldBls12381Fr::NP == 0xffffffffu,
              "the BLS12-381 reduction rows rely on r = 2^64 - 2^32 + 1 mod 2^64");

// ------------------------------------------------------------------ helpers

// Carry chains over aligned word pairs d[0..7]; the low and high half of a
// product are adjacent, so that ptxas issues the pair as one instruction.

// d = (x0, x1, x2, x3) * y
__device__ __forceinline__ void pairs_mul4(uint32_t d[8], uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3,
                                           uint32_t y) {
  asm("mul.lo.u32 %0, %8,  %12;\n\t"
      "mul.hi.u32 %1, %8,  %12;\n\t"
      "mul.lo.u32 %2, %9,  %12;\n\t"
      "mul.hi.u32 %3, %9,  %12;\n\t"
      "mul.lo.u32 %4, %10, %12;\n\t"
      "mul.hi.u32 %5, %10, %12;\n\t"
      "mul.lo.u32 %6, %11, %12;\n\t"
      "mul.hi.u32 %7, %11, %12;"
      : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3]), "=r"(d[4]), "=r"(d[5]), "=r"(d[6]), "=r"(d[7])
      : "r"(x0), "r"(x1), "r"(x2), "r"(x3), "r"(y));
}

// d += (x0, x1, x2, x3) * y, no carry out
__device__ __forceinline__ void pairs_mad4(uint32_t d[8], uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3,
                                           uint32_t y) {
  asm("mad.lo.cc.u32  %0, %8,  %12, %0;\n\t"
      "madc.hi.cc.u32 %1, %8,  %12, %1;\n\t"
      "madc.lo.cc.u32 %2, %9,  %12, %2;\n\t"
      "madc.hi.cc.u32 %3, %9,  %12, %3;\n\t"
      "madc.lo.cc.u32 %4, %10, %12, %4;\n\t"
      "madc.hi.cc.u32 %5, %10, %12, %5;\n\t"
      "madc.lo.cc.u32 %6, %11, %12, %6;\n\t"
      "madc.hi.u32    %7, %11, %12, %7;"
      : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3]), "+r"(d[4]), "+r"(d[5]), "+r"(d[6]), "+r"(d[7])
      : "r"(x0), "r"(x1), "r"(x2), "r"(x3), "r"(y));
}

// d += (x0, x1, x2, x3) * y, carry into top
__device__ __forceinline__ void pairs_mad4_top(uint32_t d[8], uint32_t &top, uint32_t x0, uint32_t x1, uint32_t x2,
                                               uint32_t x3, uint32_t y) {
  asm("mad.lo.cc.u32  %0, %9,  %13, %0;\n\t"
      "madc.hi.cc.u32 %1, %9,  %13, %1;\n\t"
      "madc.lo.cc.u32 %2, %10, %13, %2;\n\t"
      "madc.hi.cc.u32 %3, %10, %13, %3;\n\t"
      "madc.lo.cc.u32 %4, %11, %13, %4;\n\t"
      "madc.hi.cc.u32 %5, %11, %13, %5;\n\t"
      "madc.lo.cc.u32 %6, %12, %13, %6;\n\t"
      "madc.hi.cc.u32 %7, %12, %13, %7;\n\t"
      "addc.u32       %8, %8, 0;"
      : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3]), "+r"(d[4]), "+r"(d[5]), "+r"(d[6]), "+r"(d[7]), "+r"(top)
      : "r"(x0), "r"(x1), "r"(x2), "r"(x3), "r"(y));
}

// The division by 2^32 with the next odd chain: e0 += s[1] (its carry is in
// column 1, where d starts), d = s[2..7] (then 0, top) + (x0, x1, x2, x3) * y.
__device__ __forceinline__ void pairs_shift_mad4(uint32_t &e0, uint32_t d[8], const uint32_t s[8], uint32_t top,
                                                 uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3, uint32_t y) {
  asm("add.cc.u32     %0, %0,  %9;\n\t"
      "madc.lo.cc.u32 %1, %17, %21, %10;\n\t"
      "madc.hi.cc.u32 %2, %17, %21, %11;\n\t"
      "madc.lo.cc.u32 %3, %18, %21, %12;\n\t"
      "madc.hi.cc.u32 %4, %18, %21, %13;\n\t"
      "madc.lo.cc.u32 %5, %19, %21, %14;\n\t"
      "madc.hi.cc.u32 %6, %19, %21, %15;\n\t"
      "madc.lo.cc.u32 %7, %20, %21, 0;\n\t"
      "madc.hi.u32    %8, %20, %21, %16;"
      : "+&r"(e0), "=&r"(d[0]), "=&r"(d[1]), "=&r"(d[2]), "=&r"(d[3]), "=&r"(d[4]), "=&r"(d[5]), "=&r"(d[6]),
        "=&r"(d[7])
      : "r"(s[1]), "r"(s[2]), "r"(s[3]), "r"(s[4]), "r"(s[5]), "r"(s[6]), "r"(s[7]), "r"(top), "r"(x0), "r"(x1),
        "r"(x2), "r"(x3), "r"(y));
}

// t = the value left after the last row: e + the words s[1..7] of the other
// accumulator (no carry out of eight words).
__device__ __forceinline__ void pairs_merge(uint32_t t[8], const uint32_t e[8], const uint32_t s[8]) {
  asm("add.cc.u32  %0, %8,  %16;\n\t"
      "addc.cc.u32 %1, %9,  %17;\n\t"
      "addc.cc.u32 %2, %10, %18;\n\t"
      "addc.cc.u32 %3, %11, %19;\n\t"
      "addc.cc.u32 %4, %12, %20;\n\t"
      "addc.cc.u32 %5, %13, %21;\n\t"
      "addc.cc.u32 %6, %14, %22;\n\t"
      "addc.u32    %7, %15, 0;"
      : "=&r"(t[0]), "=&r"(t[1]), "=&r"(t[2]), "=&r"(t[3]), "=&r"(t[4]), "=&r"(t[5]), "=&r"(t[6]), "=&r"(t[7])
      : "r"(e[0]), "r"(e[1]), "r"(e[2]), "r"(e[3]), "r"(e[4]), "r"(e[5]), "r"(e[6]), "r"(e[7]), "r"(s[1]),
        "r"(s[2]), "r"(s[3]), "r"(s[4]), "r"(s[5]), "r"(s[6]), "r"(s[7]));
}

// Reduction of one row: T becomes a multiple of 2^32 (E_0 is not used after).
//
// In general T += m p with m = T_0 (-p^-1 mod 2^32).
//
// BLS12-381 Fr: r = 2^64 R + (2^64 - 2^32 + 1), so T - T_0 r needs no product
// for m and six instead of eight for T_0 r:
//   T - T_0 r = T - T_0 + T_0 2^32 - T_0 (R + 1) 2^64
//             = T - T_0 + T_0 2^32 + T_0 (2^192 - R - 1) 2^64 - T_0 2^256.
// T is then a signed number (two's complement in nine words: with one factor
// below r, |T| < 2^287).  Measured: 74 G products/s against 57 G/s with the
// additive rows of one accumulator (120 against 187 IMAD-pipe instructions)
// and 57-62 G/s with additive rows over two.
template <class F>
__device__ __forceinline__ void redc_row(uint32_t E[8], uint32_t O[8]) {
  if constexpr (F::kSubtract) {
    const uint32_t t = E[0];
    asm("mad.lo.cc.u32  %0, %6, %7, %0;\n\t"
        "madc.hi.cc.u32 %1, %6, %7, %1;\n\t"
        "madc.lo.cc.u32 %2, %6, %8, %2;\n\t"
        "madc.hi.cc.u32 %3, %6, %8, %3;\n\t"
        "madc.lo.cc.u32 %4, %6, %9, %4;\n\t"
        "madc.hi.u32    %5, %6, %9, %5;"
        : "+r"(O[2]), "+r"(O[3]), "+r"(O[4]), "+r"(O[5]), "+r"(O[6]), "+r"(O[7])
        : "r"(t), "n"(~F::P3), "n"(~F::P5), "n"(~F::P7));
    O[7] -= t;
    asm("add.cc.u32     %0, %0, %8;\n\t"
        "madc.lo.cc.u32 %1, %8, %9,  %1;\n\t"
        "madc.hi.cc.u32 %2, %8, %9,  %2;\n\t"
        "madc.lo.cc.u32 %3, %8, %10, %3;\n\t"
        "madc.hi.cc.u32 %4, %8, %10, %4;\n\t"
        "madc.lo.cc.u32 %5, %8, %11, %5;\n\t"
        "madc.hi.cc.u32 %6, %8, %11, %6;\n\t"
        "addc.u32       %7, %7, 0;"
        : "+r"(E[1]), "+r"(E[2]), "+r"(E[3]), "+r"(E[4]), "+r"(E[5]), "+r"(E[6]), "+r"(E[7]), "+r"(O[7])
        : "r"(t), "n"(~F::P2), "n"(~F::P4), "n"(~F::P6));
  } else {
    const uint32_t m = E[0] * F::NP;
    pairs_mad4(O, F::P1, F::P3, F::P5, F::P7, m);
    pairs_mad4_top(E, O[7], F::P0, F::P2, F::P4, F::P6, m);
  }
}

// r += p when the mask is nonzero (mod 2^256)
template <class F>
__device__ __forceinline__ void add_p_if(uint32_t r[8], uint32_t mask) {
  asm("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %16, 0;\n\t"
      "@q add.cc.u32  %0, %0, %8;\n\t"
      "@q addc.cc.u32 %1, %1, %9;\n\t"
      "@q addc.cc.u32 %2, %2, %10;\n\t"
      "@q addc.cc.u32 %3, %3, %11;\n\t"
      "@q addc.cc.u32 %4, %4, %12;\n\t"
      "@q addc.cc.u32 %5, %5, %13;\n\t"
      "@q addc.cc.u32 %6, %6, %14;\n\t"
      "@q addc.u32    %7, %7, %15;\n\t}"
      : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])
      : "n"(F::P0), "n"(F::P1), "n"(F::P2), "n"(F::P3), "n"(F::P4), "n"(F::P5), "n"(F::P6), "n"(F::P7), "r"(mask));
}

__device__ __forceinline__ void fe_copy(uint32_t r[8], const uint32_t a[8]) {
#pragma unroll
  for (int j = 0; j < 8; ++j) r[j] = a[j];
}

// r = t - p if t >= p else t   (t < 2p).
template <class F>
__device__ __forceinline__ void reduce_once(uint32_t r[8], const uint32_t t[8]) {
  uint32_t d[8], bw;
  const uint32_t zero = 0;
  asm("sub.cc.u32  %0, %9,  %17;\n\t"
      "subc.cc.u32 %1, %10, %18;\n\t"
      "subc.cc.u32 %2, %11, %19;\n\t"
      "subc.cc.u32 %3, %12, %20;\n\t"
      "subc.cc.u32 %4, %13, %21;\n\t"
      "subc.cc.u32 %5, %14, %22;\n\t"
      "subc.cc.u32 %6, %15, %23;\n\t"
      "subc.cc.u32 %7, %16, %24;\n\t"
      "subc.u32    %8, %25, %25;"
      : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3]), "=r"(d[4]), "=r"(d[5]), "=r"(d[6]), "=r"(d[7]),
        "=r"(bw)
      : "r"(t[0]), "r"(t[1]), "r"(t[2]), "r"(t[3]), "r"(t[4]), "r"(t[5]), "r"(t[6]), "r"(t[7]), "n"(F::P0),
        "n"(F::P1), "n"(F::P2), "n"(F::P3), "n"(F::P4), "n"(F::P5), "n"(F::P6), "n"(F::P7), "r"(zero));
  // bw = all ones when t < p (keep t), zero otherwise (take t - p).
#pragma unroll
  for (int j = 0; j < 8; ++j) r[j] = (t[j] & bw) | (d[j] & ~bw);
}

// ---------------------------------------------------------------- field ops

// r = (a * b + c) * 2^(-32 N) mod p for a < p, c < p and any b of N words, N
// rows: c (nullptr: zero) is what the accumulators start from.  As a b + c <=
// (p - 1) 2^(32 N), the result (a b + c + M p) / 2^(32 N), M < 2^(32 N), is
// below 2p; with subtracted rows (- M p) it lies in (-p, p) before p is added
// to a negative one, so it is canonical.
template <class F, int N>
__device__ __forceinline__ void mont_rows(uint32_t r[8], const uint32_t a[8], const uint32_t *b, const uint32_t *c) {
  uint32_t E[8], O[8];
  if (c) {
#pragma unroll
    for (int j = 0; j < 8; ++j) E[j] = c[j];
    O[7] = 0;
    uint32_t top = 0;
    pairs_mad4_top(E, top, a[0], a[2], a[4], a[6], b[0]);
    pairs_mul4(O, a[1], a[3], a[5], a[7], b[0]);
    O[7] += top;   // column 8
  } else {
    pairs_mul4(E, a[0], a[2], a[4], a[6], b[0]);
    pairs_mul4(O, a[1], a[3], a[5], a[7], b[0]);
  }
  redc_row<F>(E, O);
#pragma unroll
  for (int i = 1; i < N; ++i) {
    uint32_t X[8];
    const uint32_t top = F::kSubtract ? (uint32_t)((int32_t)O[7] >> 31) : 0u;   // sign of T
    pairs_shift_mad4(O[0], X, E, top, a[1], a[3], a[5], a[7], b[i]);
    pairs_mad4_top(O, X[7], a[0], a[2], a[4], a[6], b[i]);
    redc_row<F>(O, X);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      E[j] = O[j];
      O[j] = X[j];
    }
  }
  pairs_merge(r, O, E);
  if constexpr (F::kSubtract) add_p_if<F>(r, (uint32_t)((int32_t)r[7] >> 31));
}

// r = a * b * 2^-256 mod p for a < p and any 256-bit b; r is canonical and may
// alias a or b.
template <class F>
__device__ __forceinline__ void mont_mul(uint32_t r[8], const uint32_t a[8], const uint32_t b[8]) {
  uint32_t t[8];
  mont_rows<F, 8>(t, a, b, nullptr);
  if constexpr (F::kSubtract) fe_copy(r, t);
  else reduce_once<F>(r, t);
}

// r = (a * b + c) * 2^-256 mod p for a, b, c < p; r canonical.
template <class F>
__device__ __forceinline__ void mont_mul_add(uint32_t r[8], const uint32_t a[8], const uint32_t b[8],
                                             const uint32_t c[8]) {
  uint32_t t[8];
  mont_rows<F, 8>(t, a, b, c);
  if constexpr (F::kSubtract) fe_copy(r, t);
  else reduce_once<F>(r, t);
}

// r = a * 2^-256 mod p for a < p; r canonical.
template <class F>
__device__ __forceinline__ void mont_redc(uint32_t r[8], const uint32_t a[8]) {
  const uint32_t one[8] = {1, 0, 0, 0, 0, 0, 0, 0};
  mont_mul<F>(r, a, one);
}

// r = a + b mod p.
template <class F>
__device__ __forceinline__ void add_mod(uint32_t r[8], const uint32_t a[8], const uint32_t b[8]) {
  uint32_t s[8];
  asm("add.cc.u32  %0, %8,  %16;\n\t"
      "addc.cc.u32 %1, %9,  %17;\n\t"
      "addc.cc.u32 %2, %10, %18;\n\t"
      "addc.cc.u32 %3, %11, %19;\n\t"
      "addc.cc.u32 %4, %12, %20;\n\t"
      "addc.cc.u32 %5, %13, %21;\n\t"
      "addc.cc.u32 %6, %14, %22;\n\t"
      "addc.u32    %7, %15, %23;"
      : "=r"(s[0]), "=r"(s[1]), "=r"(s[2]), "=r"(s[3]), "=r"(s[4]), "=r"(s[5]), "=r"(s[6]), "=r"(s[7])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]), "r"(b[0]),
        "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]));
  reduce_once<F>(r, s);
}

// r = a - b mod p.
template <class F>
__device__ __forceinline__ void sub_mod(uint32_t r[8], const uint32_t a[8], const uint32_t b[8]) {
  uint32_t d[8], bw;
  const uint32_t zero = 0;
  asm("sub.cc.u32  %0, %9,  %17;\n\t"
      "subc.cc.u32 %1, %10, %18;\n\t"
      "subc.cc.u32 %2, %11, %19;\n\t"
      "subc.cc.u32 %3, %12, %20;\n\t"
      "subc.cc.u32 %4, %13, %21;\n\t"
      "subc.cc.u32 %5, %14, %22;\n\t"
      "subc.cc.u32 %6, %15, %23;\n\t"
      "subc.cc.u32 %7, %16, %24;\n\t"
      "subc.u32    %8, %25, %25;"
      : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3]), "=r"(d[4]), "=r"(d[5]), "=r"(d[6]), "=r"(d[7]),
        "=r"(bw)
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]), "r"(b[0]),
        "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]), "r"(zero));
  // add p back when the subtraction borrowed (bw = all ones)
  add_p_if<F>(d, bw);
#pragma unroll
  for (int j = 0; j < 8; ++j) r[j] = d[j];
}

// ------------------------------------------- lazy values in [0, kLazy p)
// Inside a transform pass values stay in [0, 2p) (BLS12-381 Fr) or [0, 3p) (BN254
// Fr, where 3p < 2^256 and mul_split then ends below 3p without a subtraction).

// Limb j of kLazy p.
template <class F>
struct LazyP {
  static constexpr uint64_t k = F::kLazy;
  static constexpr uint64_t C0 = k * F::P0, C1 = k * F::P1 + (C0 >> 32), C2 = k * F::P2 + (C1 >> 32),
                            C3 = k * F::P3 + (C2 >> 32), C4 = k * F::P4 + (C3 >> 32), C5 = k * F::P5 + (C4 >> 32),
                            C6 = k * F::P6 + (C5 >> 32), C7 = k * F::P7 + (C6 >> 32);
  static_assert(C7 >> 32 == 0, "kLazy p < 2^256");
  static constexpr uint32_t W0 = (uint32_t)C0, W1 = (uint32_t)C1, W2 = (uint32_t)C2, W3 = (uint32_t)C3,
                            W4 = (uint32_t)C4, W5 = (uint32_t)C5, W6 = (uint32_t)C6, W7 = (uint32_t)C7;
};

// r = a + b mod kLazy p for a, b < kLazy p (the sum may need 257 bits).
template <class F>
__device__ __forceinline__ void add_lazy(uint32_t r[8], const uint32_t a[8], const uint32_t b[8]) {
  using P = LazyP<F>;
  uint32_t s[8], d[8], c;
  asm("add.cc.u32  %0, %9,  %17;\n\t"
      "addc.cc.u32 %1, %10, %18;\n\t"
      "addc.cc.u32 %2, %11, %19;\n\t"
      "addc.cc.u32 %3, %12, %20;\n\t"
      "addc.cc.u32 %4, %13, %21;\n\t"
      "addc.cc.u32 %5, %14, %22;\n\t"
      "addc.cc.u32 %6, %15, %23;\n\t"
      "addc.cc.u32 %7, %16, %24;\n\t"
      "addc.u32    %8, 0, 0;"
      : "=&r"(s[0]), "=&r"(s[1]), "=&r"(s[2]), "=&r"(s[3]), "=&r"(s[4]), "=&r"(s[5]), "=&r"(s[6]), "=&r"(s[7]),
        "=&r"(c)
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]), "r"(b[0]),
        "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]));
  asm("sub.cc.u32  %0, %9,  %17;\n\t"
      "subc.cc.u32 %1, %10, %18;\n\t"
      "subc.cc.u32 %2, %11, %19;\n\t"
      "subc.cc.u32 %3, %12, %20;\n\t"
      "subc.cc.u32 %4, %13, %21;\n\t"
      "subc.cc.u32 %5, %14, %22;\n\t"
      "subc.cc.u32 %6, %15, %23;\n\t"
      "subc.cc.u32 %7, %16, %24;\n\t"
      "subc.u32    %8, %8, 0;"
      : "=&r"(d[0]), "=&r"(d[1]), "=&r"(d[2]), "=&r"(d[3]), "=&r"(d[4]), "=&r"(d[5]), "=&r"(d[6]), "=&r"(d[7]),
        "+&r"(c)
      : "r"(s[0]), "r"(s[1]), "r"(s[2]), "r"(s[3]), "r"(s[4]), "r"(s[5]), "r"(s[6]), "r"(s[7]), "n"(P::W0),
        "n"(P::W1), "n"(P::W2), "n"(P::W3), "n"(P::W4), "n"(P::W5), "n"(P::W6), "n"(P::W7));
  // c: all ones when a + b < kLazy p, zero otherwise
#pragma unroll
  for (int j = 0; j < 8; ++j) r[j] = c ? s[j] : d[j];
}

// r = a - b mod kLazy p for a, b < kLazy p.
template <class F>
__device__ __forceinline__ void sub_lazy(uint32_t r[8], const uint32_t a[8], const uint32_t b[8]) {
  using P = LazyP<F>;
  asm("{\n\t.reg .pred q;\n\t.reg .u32 c;\n\t"
      "sub.cc.u32  %0, %8,  %16;\n\t"
      "subc.cc.u32 %1, %9,  %17;\n\t"
      "subc.cc.u32 %2, %10, %18;\n\t"
      "subc.cc.u32 %3, %11, %19;\n\t"
      "subc.cc.u32 %4, %12, %20;\n\t"
      "subc.cc.u32 %5, %13, %21;\n\t"
      "subc.cc.u32 %6, %14, %22;\n\t"
      "subc.cc.u32 %7, %15, %23;\n\t"
      "subc.u32    c, 0, 0;\n\t"
      "setp.ne.u32 q, c, 0;\n\t"
      "@q add.cc.u32  %0, %0, %24;\n\t"
      "@q addc.cc.u32 %1, %1, %25;\n\t"
      "@q addc.cc.u32 %2, %2, %26;\n\t"
      "@q addc.cc.u32 %3, %3, %27;\n\t"
      "@q addc.cc.u32 %4, %4, %28;\n\t"
      "@q addc.cc.u32 %5, %5, %29;\n\t"
      "@q addc.cc.u32 %6, %6, %30;\n\t"
      "@q addc.u32    %7, %7, %31;\n\t}"
      : "=&r"(r[0]), "=&r"(r[1]), "=&r"(r[2]), "=&r"(r[3]), "=&r"(r[4]), "=&r"(r[5]), "=&r"(r[6]), "=&r"(r[7])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]), "r"(b[0]),
        "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]), "n"(P::W0), "n"(P::W1),
        "n"(P::W2), "n"(P::W3), "n"(P::W4), "n"(P::W5), "n"(P::W6), "n"(P::W7));
}

// r = a * b * 2^-256 mod p for a < p and any 256-bit b, left below 2p.
template <class F>
__device__ __forceinline__ void mont_mul_lazy(uint32_t r[8], const uint32_t a[8], const uint32_t b[8]) {
  uint32_t t[8];
  mont_rows<F, 8>(t, a, b, nullptr);
  fe_copy(r, t);
}

// The subtracted rows below add two products per row: T < 2 p 2^32 + 2p is
// below 2^288, but T - T_0 r can be negative too, so the sign is a word of its
// own, s (0 or all ones, weight 2^288), which every chain that ends in column
// 8 carries into.
__device__ __forceinline__ void pairs_mad4_top_s(uint32_t d[8], uint32_t &top, uint32_t &s, uint32_t x0, uint32_t x1,
                                                 uint32_t x2, uint32_t x3, uint32_t y) {
  asm("mad.lo.cc.u32  %0, %10, %14, %0;\n\t"
      "madc.hi.cc.u32 %1, %10, %14, %1;\n\t"
      "madc.lo.cc.u32 %2, %11, %14, %2;\n\t"
      "madc.hi.cc.u32 %3, %11, %14, %3;\n\t"
      "madc.lo.cc.u32 %4, %12, %14, %4;\n\t"
      "madc.hi.cc.u32 %5, %12, %14, %5;\n\t"
      "madc.lo.cc.u32 %6, %13, %14, %6;\n\t"
      "madc.hi.cc.u32 %7, %13, %14, %7;\n\t"
      "addc.cc.u32    %8, %8, 0;\n\t"
      "addc.u32       %9, %9, 0;"
      : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3]), "+r"(d[4]), "+r"(d[5]), "+r"(d[6]), "+r"(d[7]), "+r"(top),
        "+r"(s)
      : "r"(x0), "r"(x1), "r"(x2), "r"(x3), "r"(y));
}

// pairs_shift_mad4 with s as the word above; the new s is its sign extension.
__device__ __forceinline__ void pairs_shift_mad4_s(uint32_t &e0, uint32_t d[8], uint32_t &s, const uint32_t w[8],
                                                   uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3, uint32_t y) {
  asm("add.cc.u32     %0, %0,  %10;\n\t"
      "madc.lo.cc.u32 %1, %17, %21, %11;\n\t"
      "madc.hi.cc.u32 %2, %17, %21, %12;\n\t"
      "madc.lo.cc.u32 %3, %18, %21, %13;\n\t"
      "madc.hi.cc.u32 %4, %18, %21, %14;\n\t"
      "madc.lo.cc.u32 %5, %19, %21, %15;\n\t"
      "madc.hi.cc.u32 %6, %19, %21, %16;\n\t"
      "madc.lo.cc.u32 %7, %20, %21, 0;\n\t"
      "madc.hi.cc.u32 %8, %20, %21, %9;\n\t"
      "addc.u32       %9, %9, 0;"
      : "+&r"(e0), "=&r"(d[0]), "=&r"(d[1]), "=&r"(d[2]), "=&r"(d[3]), "=&r"(d[4]), "=&r"(d[5]), "=&r"(d[6]),
        "=&r"(d[7]), "+&r"(s)
      : "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]), "r"(x0), "r"(x1), "r"(x2),
        "r"(x3), "r"(y));
}

template <class F>
__device__ __forceinline__ void redc_row_s(uint32_t E[8], uint32_t O[8], uint32_t &s) {
  const uint32_t t = E[0];
  asm("mad.lo.cc.u32  %0, %7, %8,  %0;\n\t"
      "madc.hi.cc.u32 %1, %7, %8,  %1;\n\t"
      "madc.lo.cc.u32 %2, %7, %9,  %2;\n\t"
      "madc.hi.cc.u32 %3, %7, %9,  %3;\n\t"
      "madc.lo.cc.u32 %4, %7, %10, %4;\n\t"
      "madc.hi.cc.u32 %5, %7, %10, %5;\n\t"
      "addc.u32       %6, %6, 0;\n\t"
      "sub.cc.u32     %5, %5, %7;\n\t"
      "subc.u32       %6, %6, 0;"
      : "+r"(O[2]), "+r"(O[3]), "+r"(O[4]), "+r"(O[5]), "+r"(O[6]), "+r"(O[7]), "+r"(s)
      : "r"(t), "n"(~F::P3), "n"(~F::P5), "n"(~F::P7));
  asm("add.cc.u32     %0, %0, %9;\n\t"
      "madc.lo.cc.u32 %1, %9, %10, %1;\n\t"
      "madc.hi.cc.u32 %2, %9, %10, %2;\n\t"
      "madc.lo.cc.u32 %3, %9, %11, %3;\n\t"
      "madc.hi.cc.u32 %4, %9, %11, %4;\n\t"
      "madc.lo.cc.u32 %5, %9, %12, %5;\n\t"
      "madc.hi.cc.u32 %6, %9, %12, %6;\n\t"
      "addc.cc.u32    %7, %7, 0;\n\t"
      "addc.u32       %8, %8, 0;"
      : "+r"(E[1]), "+r"(E[2]), "+r"(E[3]), "+r"(E[4]), "+r"(E[5]), "+r"(E[6]), "+r"(E[7]), "+r"(O[7]), "+r"(s)
      : "r"(t), "n"(~F::P2), "n"(~F::P4), "n"(~F::P6));
}

// Product by a constant w kept as two residues, A = w 2^128 mod p and B = w
// 2^256 mod p: x w = (x_lo A + x_hi B) 2^-128 with the 128-bit halves of x, a
// sum of 12 words instead of 16, so half of the reduction rows fall away (64 +
// 32 products instead of 64 + 64; BLS12-381 Fr 64 + 24 instead of 64 + 48).
// x < kLazy p; r = x w mod p, left below kLazy p: (x_lo A + x_hi B + M p) 2^-128
// < (1 + x 2^-256 + 1) p, which is below 2.57 p for BN254 and x < 3p; for
// BLS12-381 the subtracted rows give (-p, 1.91 p) (p added to a negative
// value).  Measured, dependent products: 93 G/s (BLS12-381 Fr) and 88 G/s
// (BN254 Fr) against 74 and 66 G/s for mont_mul.
template <class F>
__device__ __forceinline__ void mul_split(uint32_t r[8], const uint32_t x[8], const uint32_t A[8],
                                          const uint32_t B[8]) {
  uint32_t E[8], O[8], s = 0;
  pairs_mul4(E, A[0], A[2], A[4], A[6], x[0]);
  pairs_mul4(O, A[1], A[3], A[5], A[7], x[0]);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (i > 0) {
      uint32_t X[8];
      if constexpr (F::kSubtract) {
        pairs_shift_mad4_s(O[0], X, s, E, A[1], A[3], A[5], A[7], x[i]);
        pairs_mad4_top_s(O, X[7], s, A[0], A[2], A[4], A[6], x[i]);
      } else {
        pairs_shift_mad4(O[0], X, E, 0u, A[1], A[3], A[5], A[7], x[i]);
        pairs_mad4_top(O, X[7], A[0], A[2], A[4], A[6], x[i]);
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        E[j] = O[j];
        O[j] = X[j];
      }
    }
    if constexpr (F::kSubtract) {
      pairs_mad4_top(O, s, B[1], B[3], B[5], B[7], x[4 + i]);
      pairs_mad4_top_s(E, O[7], s, B[0], B[2], B[4], B[6], x[4 + i]);
      redc_row_s<F>(E, O, s);
    } else {
      pairs_mad4(O, B[1], B[3], B[5], B[7], x[4 + i]);
      pairs_mad4_top(E, O[7], B[0], B[2], B[4], B[6], x[4 + i]);
      redc_row<F>(E, O);
    }
  }
  if constexpr (F::kSubtract) {
    asm("add.cc.u32  %0, %9,  %17;\n\t"
        "addc.cc.u32 %1, %10, %18;\n\t"
        "addc.cc.u32 %2, %11, %19;\n\t"
        "addc.cc.u32 %3, %12, %20;\n\t"
        "addc.cc.u32 %4, %13, %21;\n\t"
        "addc.cc.u32 %5, %14, %22;\n\t"
        "addc.cc.u32 %6, %15, %23;\n\t"
        "addc.cc.u32 %7, %16, 0;\n\t"
        "addc.u32    %8, %8, 0;"
        : "=&r"(r[0]), "=&r"(r[1]), "=&r"(r[2]), "=&r"(r[3]), "=&r"(r[4]), "=&r"(r[5]), "=&r"(r[6]), "=&r"(r[7]),
          "+&r"(s)
        : "r"(O[0]), "r"(O[1]), "r"(O[2]), "r"(O[3]), "r"(O[4]), "r"(O[5]), "r"(O[6]), "r"(O[7]), "r"(E[1]),
          "r"(E[2]), "r"(E[3]), "r"(E[4]), "r"(E[5]), "r"(E[6]), "r"(E[7]));
    add_p_if<F>(r, s);
  } else {
    pairs_merge(r, O, E);
  }
}

// r = t mod p for t < kLazy p.
template <class F>
__device__ __forceinline__ void reduce_lazy(uint32_t r[8], const uint32_t t[8]) {
  reduce_once<F>(r, t);
  if constexpr (F::kLazy == 3) reduce_once<F>(r, r);
}

// ------------------------------------------- warp-cooperative variant
// The same CIOS Montgomery product with one element spread over 8 lanes
// (lane j of each aligned group of 8 holds limb j): every lane does the two
// 32x32 products of its limb per row, the high halves move one lane up by
// warp shuffle, the reduction factor m is broadcast from lane 0, and the
// running value is shifted one lane down per row.  Columns are kept in 64-bit
// accumulators (carries deferred); after the 8 rows the carries are
// propagated lane to lane, and the final comparison / subtraction of p uses
// a carry-lookahead on warp ballots.  Kept as a measured alternative to the
// per-thread carry chains (mont_mul), which have no shuffle traffic.
template <class F>
__device__ __forceinline__ uint32_t mont_mul_coop(uint32_t a_j, uint32_t b_j, uint32_t j) {
  constexpr uint32_t kFull = 0xffffffffu;
  const uint32_t p_j = j == 0 ? F::P0 : j == 1 ? F::P1 : j == 2 ? F::P2 : j == 3 ? F::P3
                     : j == 4 ? F::P4 : j == 5 ? F::P5 : j == 6 ? F::P6 : F::P7;
  uint64_t acc = 0, top = 0;  // top: column 8, kept by lane 7
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t bi = __shfl_sync(kFull, b_j, i, 8);
    const uint64_t pr = (uint64_t)a_j * bi;
    const uint32_t hi_in = __shfl_up_sync(kFull, (uint32_t)(pr >> 32), 1, 8);
    acc += (uint64_t)(uint32_t)pr + (j ? hi_in : 0u);
    if (j == 7) top += pr >> 32;
    const uint32_t m = __shfl_sync(kFull, (uint32_t)acc * F::NP, 0, 8);
    const uint64_t pm = (uint64_t)p_j * m;
    const uint32_t hm_in = __shfl_up_sync(kFull, (uint32_t)(pm >> 32), 1, 8);
    acc += (uint64_t)(uint32_t)pm + (j ? hm_in : 0u);
    if (j == 7) top += pm >> 32;
    // column 0 is now 0 mod 2^32: its high part carries into column 1
    const uint32_t c0 = __shfl_sync(kFull, (uint32_t)(acc >> 32), 0, 8);  // columns stay < 2^38
    if (j == 1) acc += c0;
    // divide by 2^32: every column moves one lane down
    const uint32_t nx_lo = __shfl_down_sync(kFull, (uint32_t)acc, 1, 8);
    const uint32_t nx_hi = __shfl_down_sync(kFull, (uint32_t)(acc >> 32), 1, 8);
    acc = j == 7 ? top : ((uint64_t)nx_hi << 32 | nx_lo);
    if (j == 7) top = 0;
  }
  // propagate the deferred carries (each column < 2^38)
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const uint32_t c = __shfl_up_sync(kFull, (uint32_t)(acc >> 32), 1, 8);
    acc = (acc & 0xffffffffull) + (j ? c : 0u);
  }
  const uint32_t t = (uint32_t)acc;  // t < 2p
  // t - p if t >= p: borrow lookahead over the group's 8 lanes
  const uint32_t base = (threadIdx.x & 31u) & ~7u;
  const uint32_t G = (__ballot_sync(kFull, t < p_j) >> base) & 0xffu;   // generates a borrow
  const uint32_t P = (__ballot_sync(kFull, t == p_j) >> base) & 0xffu;  // propagates one
  const uint32_t x = G | P, sum = x + G;
  const uint32_t borrow_in = ((sum ^ x ^ G) >> j) & 1u;
  const bool ge = ((sum >> 8) & 1u) == 0;  // no borrow out of the top limb
  return ge ? t - p_j - borrow_in : t;
}

// ------------------------------------------------------------- memory access

// One element = 32 bytes, moved with one 256-bit access (ld/st .v8.b32,
// sm_100 and later); element addresses are 32-byte aligned.
__device__ __forceinline__ void fe_load_global(uint32_t r[8], const uint4 *base, uint64_t elem) {
  asm("ld.global.nc.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
      : "l"(base + 2 * elem));
}

__device__ __forceinline__ void fe_store_global(uint4 *base, uint64_t elem, const uint32_t a[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
               :
               : "l"(base + 2 * elem), "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]),
                 "r"(a[6]), "r"(a[7])
               : "memory");
}

}  // namespace gb300ntt
