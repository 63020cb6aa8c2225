// fp_square.cuh -- Montgomery squares and sums of two products over the base
// fields of the curves (T: a field of ec_xyzz.cuh with L = 8 or 12 limbs of 32
// bits), sm_103a.
//
// Point additions are bound by the IMAD pipe, where each 32 x 32 + 64 product
// takes four cycles of a warp.  Of the ten products of a mixed addition two are
// squares, which need 36 limb products instead of 64 beside their reduction (78
// instead of 144 over 12 limbs), and two are only used as a difference, which
// needs one reduction instead of two.
// Bucket accumulation, 2^22 points of BN254: 10.47 -> 9.51 ms; a commitment over
// 2^20 fixed points of BLS12-381: 6.05 -> 5.50 ms.
#pragma once

#include "fp256.cuh"
#include "fp384.cuh"

namespace gb300ntt {

// d[0 .. 2N-1] += (x[0], ..., x[N-1]) * y over aligned word pairs, carry into
// top.
template <int N>
__device__ __forceinline__ void pairs_mad_chain(uint32_t *d, uint32_t &top, const uint32_t *x, uint32_t y) {
  if constexpr (N == 1) {
    asm("mad.lo.cc.u32  %0, %3, %4, %0;\n\t"
        "madc.hi.cc.u32 %1, %3, %4, %1;\n\t"
        "addc.u32       %2, %2, 0;"
        : "+r"(d[0]), "+r"(d[1]), "+r"(top)
        : "r"(x[0]), "r"(y));
  } else if constexpr (N == 2) {
    asm("mad.lo.cc.u32  %0, %5, %7, %0;\n\t"
        "madc.hi.cc.u32 %1, %5, %7, %1;\n\t"
        "madc.lo.cc.u32 %2, %6, %7, %2;\n\t"
        "madc.hi.cc.u32 %3, %6, %7, %3;\n\t"
        "addc.u32       %4, %4, 0;"
        : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3]), "+r"(top)
        : "r"(x[0]), "r"(x[1]), "r"(y));
  } else if constexpr (N == 3) {
    asm("mad.lo.cc.u32  %0, %7, %10, %0;\n\t"
        "madc.hi.cc.u32 %1, %7, %10, %1;\n\t"
        "madc.lo.cc.u32 %2, %8, %10, %2;\n\t"
        "madc.hi.cc.u32 %3, %8, %10, %3;\n\t"
        "madc.lo.cc.u32 %4, %9, %10, %4;\n\t"
        "madc.hi.cc.u32 %5, %9, %10, %5;\n\t"
        "addc.u32       %6, %6, 0;"
        : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3]), "+r"(d[4]), "+r"(d[5]), "+r"(top)
        : "r"(x[0]), "r"(x[1]), "r"(x[2]), "r"(y));
  } else if constexpr (N == 4) {
    pairs_mad4_top(d, top, x[0], x[1], x[2], x[3], y);
  } else if constexpr (N == 5) {
    asm("mad.lo.cc.u32  %0, %11, %16, %0;\n\t"
        "madc.hi.cc.u32 %1, %11, %16, %1;\n\t"
        "madc.lo.cc.u32 %2, %12, %16, %2;\n\t"
        "madc.hi.cc.u32 %3, %12, %16, %3;\n\t"
        "madc.lo.cc.u32 %4, %13, %16, %4;\n\t"
        "madc.hi.cc.u32 %5, %13, %16, %5;\n\t"
        "madc.lo.cc.u32 %6, %14, %16, %6;\n\t"
        "madc.hi.cc.u32 %7, %14, %16, %7;\n\t"
        "madc.lo.cc.u32 %8, %15, %16, %8;\n\t"
        "madc.hi.cc.u32 %9, %15, %16, %9;\n\t"
        "addc.u32       %10, %10, 0;"
        : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3]), "+r"(d[4]), "+r"(d[5]), "+r"(d[6]), "+r"(d[7]), "+r"(d[8]),
          "+r"(d[9]), "+r"(top)
        : "r"(x[0]), "r"(x[1]), "r"(x[2]), "r"(x[3]), "r"(x[4]), "r"(y));
  } else if constexpr (N == 6) {
    fp384::pairs_mad6_top(d, top, x[0], x[1], x[2], x[3], x[4], x[5], y);
  } else {
    static_assert(N >= 1 && N <= 6, "chain length");
  }
}

// u = a + b, no carry out of L words
template <int L>
__device__ __forceinline__ void words_add(uint32_t u[L], const uint32_t a[L], const uint32_t b[L]) {
  static_assert(L == 8 || L == 12, "limbs");
  if constexpr (L == 8) {
    asm("add.cc.u32  %0, %8, %16;\n\t"
        "addc.cc.u32 %1, %9, %17;\n\t"
        "addc.cc.u32 %2, %10, %18;\n\t"
        "addc.cc.u32 %3, %11, %19;\n\t"
        "addc.cc.u32 %4, %12, %20;\n\t"
        "addc.cc.u32 %5, %13, %21;\n\t"
        "addc.cc.u32 %6, %14, %22;\n\t"
        "addc.u32    %7, %15, %23;"
        : "=&r"(u[0]), "=&r"(u[1]), "=&r"(u[2]), "=&r"(u[3]), "=&r"(u[4]), "=&r"(u[5]), "=&r"(u[6]), "=&r"(u[7])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]), "r"(b[0]), "r"(b[1]),
          "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]));
  } else {
    asm("add.cc.u32  %0, %12, %24;\n\t"
        "addc.cc.u32 %1, %13, %25;\n\t"
        "addc.cc.u32 %2, %14, %26;\n\t"
        "addc.cc.u32 %3, %15, %27;\n\t"
        "addc.cc.u32 %4, %16, %28;\n\t"
        "addc.cc.u32 %5, %17, %29;\n\t"
        "addc.cc.u32 %6, %18, %30;\n\t"
        "addc.cc.u32 %7, %19, %31;\n\t"
        "addc.cc.u32 %8, %20, %32;\n\t"
        "addc.cc.u32 %9, %21, %33;\n\t"
        "addc.cc.u32 %10, %22, %34;\n\t"
        "addc.u32    %11, %23, %35;"
        : "=&r"(u[0]), "=&r"(u[1]), "=&r"(u[2]), "=&r"(u[3]), "=&r"(u[4]), "=&r"(u[5]), "=&r"(u[6]), "=&r"(u[7]),
          "=&r"(u[8]), "=&r"(u[9]), "=&r"(u[10]), "=&r"(u[11])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]), "r"(a[8]), "r"(a[9]),
          "r"(a[10]), "r"(a[11]), "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]),
          "r"(b[7]), "r"(b[8]), "r"(b[9]), "r"(b[10]), "r"(b[11]));
  }
}

// u = a - b for a >= b
template <int L>
__device__ __forceinline__ void words_sub(uint32_t u[L], const uint32_t a[L], const uint32_t b[L]) {
  static_assert(L == 8 || L == 12, "limbs");
  if constexpr (L == 8) {
    asm("sub.cc.u32  %0, %8, %16;\n\t"
        "subc.cc.u32 %1, %9, %17;\n\t"
        "subc.cc.u32 %2, %10, %18;\n\t"
        "subc.cc.u32 %3, %11, %19;\n\t"
        "subc.cc.u32 %4, %12, %20;\n\t"
        "subc.cc.u32 %5, %13, %21;\n\t"
        "subc.cc.u32 %6, %14, %22;\n\t"
        "subc.u32    %7, %15, %23;"
        : "=&r"(u[0]), "=&r"(u[1]), "=&r"(u[2]), "=&r"(u[3]), "=&r"(u[4]), "=&r"(u[5]), "=&r"(u[6]), "=&r"(u[7])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]), "r"(b[0]), "r"(b[1]),
          "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]));
  } else {
    asm("sub.cc.u32  %0, %12, %24;\n\t"
        "subc.cc.u32 %1, %13, %25;\n\t"
        "subc.cc.u32 %2, %14, %26;\n\t"
        "subc.cc.u32 %3, %15, %27;\n\t"
        "subc.cc.u32 %4, %16, %28;\n\t"
        "subc.cc.u32 %5, %17, %29;\n\t"
        "subc.cc.u32 %6, %18, %30;\n\t"
        "subc.cc.u32 %7, %19, %31;\n\t"
        "subc.cc.u32 %8, %20, %32;\n\t"
        "subc.cc.u32 %9, %21, %33;\n\t"
        "subc.cc.u32 %10, %22, %34;\n\t"
        "subc.u32    %11, %23, %35;"
        : "=&r"(u[0]), "=&r"(u[1]), "=&r"(u[2]), "=&r"(u[3]), "=&r"(u[4]), "=&r"(u[5]), "=&r"(u[6]), "=&r"(u[7]),
          "=&r"(u[8]), "=&r"(u[9]), "=&r"(u[10]), "=&r"(u[11])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]), "r"(a[8]), "r"(a[9]),
          "r"(a[10]), "r"(a[11]), "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]),
          "r"(b[7]), "r"(b[8]), "r"(b[9]), "r"(b[10]), "r"(b[11]));
  }
}

// The division by 2^32 with the next row's factor and odd chain: e0 += s[1] (its
// carry is in column 1, where d starts), m = e0 np, d = s[2 .. L-1], u, 0 + p m
// for the odd limbs p of the modulus.
template <int L>
__device__ __forceinline__ void shift_redc_odd(uint32_t &e0, uint32_t d[L], uint32_t &m, const uint32_t s[L],
                                               uint32_t u, const uint32_t p[L / 2], uint32_t np) {
  if constexpr (L == 8) {
    asm("add.cc.u32     %0, %0, %10;\n\t"
        "mul.lo.u32     %9, %0, %22;\n\t"
        "madc.lo.cc.u32 %1, %18, %9, %11;\n\t"
        "madc.hi.cc.u32 %2, %18, %9, %12;\n\t"
        "madc.lo.cc.u32 %3, %19, %9, %13;\n\t"
        "madc.hi.cc.u32 %4, %19, %9, %14;\n\t"
        "madc.lo.cc.u32 %5, %20, %9, %15;\n\t"
        "madc.hi.cc.u32 %6, %20, %9, %16;\n\t"
        "madc.lo.cc.u32 %7, %21, %9, %17;\n\t"
        "madc.hi.u32    %8, %21, %9, 0;"
        : "+&r"(e0), "=&r"(d[0]), "=&r"(d[1]), "=&r"(d[2]), "=&r"(d[3]), "=&r"(d[4]), "=&r"(d[5]), "=&r"(d[6]),
          "=&r"(d[7]), "=&r"(m)
        : "r"(s[1]), "r"(s[2]), "r"(s[3]), "r"(s[4]), "r"(s[5]), "r"(s[6]), "r"(s[7]), "r"(u), "r"(p[0]), "r"(p[1]),
          "r"(p[2]), "r"(p[3]), "r"(np));
  } else {
    asm("add.cc.u32     %0, %0, %14;\n\t"
        "mul.lo.u32     %13, %0, %32;\n\t"
        "madc.lo.cc.u32 %1, %26, %13, %15;\n\t"
        "madc.hi.cc.u32 %2, %26, %13, %16;\n\t"
        "madc.lo.cc.u32 %3, %27, %13, %17;\n\t"
        "madc.hi.cc.u32 %4, %27, %13, %18;\n\t"
        "madc.lo.cc.u32 %5, %28, %13, %19;\n\t"
        "madc.hi.cc.u32 %6, %28, %13, %20;\n\t"
        "madc.lo.cc.u32 %7, %29, %13, %21;\n\t"
        "madc.hi.cc.u32 %8, %29, %13, %22;\n\t"
        "madc.lo.cc.u32 %9, %30, %13, %23;\n\t"
        "madc.hi.cc.u32 %10, %30, %13, %24;\n\t"
        "madc.lo.cc.u32 %11, %31, %13, %25;\n\t"
        "madc.hi.u32    %12, %31, %13, 0;"
        : "+&r"(e0), "=&r"(d[0]), "=&r"(d[1]), "=&r"(d[2]), "=&r"(d[3]), "=&r"(d[4]), "=&r"(d[5]), "=&r"(d[6]),
          "=&r"(d[7]), "=&r"(d[8]), "=&r"(d[9]), "=&r"(d[10]), "=&r"(d[11]), "=&r"(m)
        : "r"(s[1]), "r"(s[2]), "r"(s[3]), "r"(s[4]), "r"(s[5]), "r"(s[6]), "r"(s[7]), "r"(s[8]), "r"(s[9]),
          "r"(s[10]), "r"(s[11]), "r"(u), "r"(p[0]), "r"(p[1]), "r"(p[2]), "r"(p[3]), "r"(p[4]), "r"(p[5]), "r"(np));
  }
}

// d = s[2 .. L-1], 0, 0 + x y after e0 += s[1]
template <int L>
__device__ __forceinline__ void shift_mad_odd(uint32_t &e0, uint32_t d[L], const uint32_t s[L], const uint32_t x[L / 2],
                                              uint32_t y) {
  if constexpr (L == 8) pairs_shift_mad4(e0, d, s, 0u, x[0], x[1], x[2], x[3], y);
  else fp384::pairs_shift_mad6(e0, d, s, x[0], x[1], x[2], x[3], x[4], x[5], y);
}

// The modulus by even and odd limbs.
template <class T>
struct ModulusPairs {
  uint32_t even[T::L / 2], odd[T::L / 2];
  __device__ __forceinline__ ModulusPairs() {
#pragma unroll
    for (int j = 0; j < T::L / 2; ++j) {
      even[j] = T::modulus(2 * j);
      odd[j] = T::modulus(2 * j + 1);
    }
  }
};

// Row I of a square: a_I^2 2^(64 I) + a_I 2^(32 I) 2 (sum of a_j 2^(32 j), j > I).
// The limbs of the doubled tail are those of dbl = 2 a but the lowest, which has
// no bit of a_I below it.  te collects the products at even columns, to those at
// odd ones (te[k], to[k]: column k).
template <class T, int I>
__device__ __forceinline__ void square_row(uint32_t *te, uint32_t *to, const uint32_t *a, const uint32_t *dbl) {
  constexpr int L = T::L, NE = 1 + (L - 1 - I) / 2, NO = (L - I) / 2;
  uint32_t x[NE];
  x[0] = a[I];
#pragma unroll
  for (int k = 1; k < NE; ++k) x[k] = dbl[I + 2 * k];
  pairs_mad_chain<NE>(te + 2 * I, te[2 * I + 2 * NE], x, a[I]);
  if constexpr (NO > 0) {
    x[0] = a[I + 1] << 1;
#pragma unroll
    for (int k = 1; k < NO; ++k) x[k] = dbl[I + 1 + 2 * k];
    pairs_mad_chain<NO>(to + 2 * I + 1, to[2 * I + 1 + 2 * NO], x, a[I]);
  }
  if constexpr (I + 1 < L) square_row<T, I + 1>(te, to, a, dbl);
}

// r = a^2 2^(-32 L) mod p for a < 2p (4 p < 2^(32 L)); r canonical, may alias a.
// The low half of the square starts the reduction's accumulators; word i of the
// high half enters at the top column after row i, so that the running value
// stays below 2^(32 L) + p before each row and every chain ends without a carry.
template <class T>
__device__ __forceinline__ void field_square(uint32_t r[T::L], const uint32_t a[T::L]) {
  constexpr int L = T::L, H = L / 2;
  uint32_t te[2 * L + 2], to[2 * L + 2], dbl[L];
#pragma unroll
  for (int j = 0; j < 2 * L + 2; ++j) te[j] = to[j] = 0u;
  dbl[0] = a[0] << 1;
#pragma unroll
  for (int j = 1; j < L; ++j) dbl[j] = __funnelshift_l(a[j - 1], a[j], 1);
  square_row<T, 0>(te, to, a, dbl);
  uint32_t high[L], E[L], O[L];
  words_add<L>(high, te + L, to + L);
#pragma unroll
  for (int j = 0; j < L; ++j) {
    E[j] = te[j];
    O[j] = j + 1 < L ? to[j + 1] : 0u;
  }
  const ModulusPairs<T> p;
  uint32_t m = E[0] * T::F::NP, none = 0u;
  pairs_mad_chain<H>(O, none, p.odd, m);
  pairs_mad_chain<H>(E, O[L - 1], p.even, m);
#pragma unroll
  for (int i = 1; i < L; ++i) {
    uint32_t X[L];
    shift_redc_odd<L>(O[0], X, m, E, high[i - 1], p.odd, T::F::NP);
    pairs_mad_chain<H>(O, X[L - 1], p.even, m);
#pragma unroll
    for (int j = 0; j < L; ++j) {
      E[j] = O[j];
      O[j] = X[j];
    }
  }
  uint32_t s[L], t[L];
#pragma unroll
  for (int j = 0; j < L; ++j) s[j] = j + 1 < L ? E[j + 1] : high[L - 1];
  words_add<L>(t, O, s);
  T::reduce(r, t);
}

// r = (a b + c d) 2^(-32 L) mod p for a, c <= p and b, d < p; r canonical, may
// alias any.  A row adds less than 3 p 2^32 to a running value that stays below
// 4 p < 2^(32 L); the result is below 2 p as 2 p < 2^(32 L).
template <class T>
__device__ __forceinline__ void field_mul2(uint32_t r[T::L], const uint32_t a[T::L], const uint32_t b[T::L],
                                           const uint32_t c[T::L], const uint32_t d[T::L]) {
  constexpr int L = T::L, H = L / 2;
  uint32_t E[L], O[L], ae[H], ao[H], ce[H], co[H], none = 0u;
#pragma unroll
  for (int j = 0; j < H; ++j) {
    ae[j] = a[2 * j];
    ao[j] = a[2 * j + 1];
    ce[j] = c[2 * j];
    co[j] = c[2 * j + 1];
  }
#pragma unroll
  for (int j = 0; j < L; ++j) E[j] = O[j] = 0u;
  const ModulusPairs<T> p;
#pragma unroll
  for (int i = 0; i < L; ++i) {
    uint32_t X[L];
    if (i == 0) {
#pragma unroll
      for (int j = 0; j < L; ++j) X[j] = 0u;
      pairs_mad_chain<H>(X, none, ao, b[0]);
    } else {
      shift_mad_odd<L>(O[0], X, E, ao, b[i]);
    }
    pairs_mad_chain<H>(X, none, co, d[i]);
    pairs_mad_chain<H>(O, X[L - 1], ae, b[i]);
    pairs_mad_chain<H>(O, X[L - 1], ce, d[i]);
    const uint32_t m = O[0] * T::F::NP;
    pairs_mad_chain<H>(X, none, p.odd, m);
    pairs_mad_chain<H>(O, X[L - 1], p.even, m);
#pragma unroll
    for (int j = 0; j < L; ++j) {
      E[j] = O[j];
      O[j] = X[j];
    }
  }
  uint32_t s[L], t[L];
#pragma unroll
  for (int j = 0; j < L; ++j) s[j] = j + 1 < L ? E[j + 1] : 0u;
  words_add<L>(t, O, s);
  T::reduce(r, t);
}

}  // namespace gb300ntt
