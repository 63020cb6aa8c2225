// fp_wide.cuh -- arithmetic of the 377- and 753-bit fields for sm_103a, 12 and 24
// 32-bit words.
//
// Both moduli are p = C 2^32 + 1, so Montgomery's reduction row (fp256.cuh) needs
// no product for m: T - T_0 p drops column 0 and subtracts T_0 C, 11 or 23
// products, written as T_0 (2^(32 (L - 1)) - C) 2^32 - T_0 2^(32 L).  T is a signed
// number of L + 1 words; the moduli leave 7 and 15 bits of the top word free, so
// its sign is never in doubt and values may be left in [0, 2p).
//
// What bounds these fields is the IMAD pipe at four cycles per 32 x 32 bit
// multiply-add of a carry chain, as for the 256-bit ones.  29-bit limbs in 64-bit
// accumulators without carries take the same four cycles each and need 14^2 2 =
// 392 and 26^2 2 = 1352 of them; 32-bit words need 276 and 1128, and a product by
// a constant kept as two residues (mul_split) 210 and 852.
#pragma once

#include <cstdint>

#include "fp256.cuh"

namespace gb300ntt {

template <int L>
struct Words {};

// Word j of the modulus and of D = 2^(32 (L - 1)) - (p >> 32).
struct FieldW377 {
  static constexpr int L = 12;
  static constexpr int kGenerator = 7;
  __host__ __device__ static constexpr uint32_t p(int j) {
    constexpr uint32_t v[12] = {0x00000001u, 0xBBDF2BD5u, 0xF31C6809u, 0x44A29410u, 0x4C762736u, 0xE804177Du,
                                0x1114CF98u, 0xA252049Cu, 0x1701B839u, 0x69898CC5u, 0x4442D184u, 0x01921FB5u};
    return v[j];
  }
  __host__ __device__ static constexpr uint32_t d(int j) { return j == 0 ? 0u - p(1) : ~p(j + 1); }
};

struct FieldW753 {
  static constexpr int L = 24;
  static constexpr int kGenerator = 11;
  __host__ __device__ static constexpr uint32_t p(int j) {
    constexpr uint32_t v[24] = {0x00000001u, 0x6FDBDCD3u, 0xB96DE80Du, 0xDAD617FEu, 0x85D34C6Fu, 0xFD8DE898u,
                                0x6AECC4BCu, 0x848BC90Bu, 0x6ADADAA3u, 0x286E9FC2u, 0x14DBE4BEu, 0x86366056u,
                                0x33679A74u, 0x09BBDF2Au, 0x10F31C68u, 0x3644A294u, 0x7D4C7627u, 0x98E80417u,
                                0x9C1114CFu, 0x39A25204u, 0xC51701B8u, 0x8469898Cu, 0xB54442D1u, 0x0001921Fu};
    return v[j];
  }
  __host__ __device__ static constexpr uint32_t d(int j) { return j == 0 ? 0u - p(1) : ~p(j + 1); }
};

// ------------------------------------------------------------- carry chains
// As in fp256.cuh, over L / 2 aligned word pairs; x is read at every second
// word (x[0], x[2], ...).

__device__ __forceinline__ void chain_mul(Words<12>, uint32_t *d, const uint32_t *x, uint32_t y) {
  asm("mul.lo.u32 %0, %12, %18;\n\t"
      "mul.hi.u32 %1, %12, %18;\n\t"
      "mul.lo.u32 %2, %13, %18;\n\t"
      "mul.hi.u32 %3, %13, %18;\n\t"
      "mul.lo.u32 %4, %14, %18;\n\t"
      "mul.hi.u32 %5, %14, %18;\n\t"
      "mul.lo.u32 %6, %15, %18;\n\t"
      "mul.hi.u32 %7, %15, %18;\n\t"
      "mul.lo.u32 %8, %16, %18;\n\t"
      "mul.hi.u32 %9, %16, %18;\n\t"
      "mul.lo.u32 %10, %17, %18;\n\t"
      "mul.hi.u32 %11, %17, %18;"
      : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3]), "=r"(d[4]), "=r"(d[5]), "=r"(d[6]), "=r"(d[7]), "=r"(d[8]),
        "=r"(d[9]), "=r"(d[10]), "=r"(d[11])
      : "r"(x[0]), "r"(x[2]), "r"(x[4]), "r"(x[6]), "r"(x[8]), "r"(x[10]), "r"(y));
}

__device__ __forceinline__ void chain_mad(Words<12>, uint32_t *d, const uint32_t *x, uint32_t y) {
  asm("mad.lo.cc.u32 %0, %12, %18, %0;\n\t"
      "madc.hi.cc.u32 %1, %12, %18, %1;\n\t"
      "madc.lo.cc.u32 %2, %13, %18, %2;\n\t"
      "madc.hi.cc.u32 %3, %13, %18, %3;\n\t"
      "madc.lo.cc.u32 %4, %14, %18, %4;\n\t"
      "madc.hi.cc.u32 %5, %14, %18, %5;\n\t"
      "madc.lo.cc.u32 %6, %15, %18, %6;\n\t"
      "madc.hi.cc.u32 %7, %15, %18, %7;\n\t"
      "madc.lo.cc.u32 %8, %16, %18, %8;\n\t"
      "madc.hi.cc.u32 %9, %16, %18, %9;\n\t"
      "madc.lo.cc.u32 %10, %17, %18, %10;\n\t"
      "madc.hi.u32 %11, %17, %18, %11;"
      : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3]), "+r"(d[4]), "+r"(d[5]), "+r"(d[6]), "+r"(d[7]), "+r"(d[8]),
        "+r"(d[9]), "+r"(d[10]), "+r"(d[11])
      : "r"(x[0]), "r"(x[2]), "r"(x[4]), "r"(x[6]), "r"(x[8]), "r"(x[10]), "r"(y));
}

__device__ __forceinline__ void chain_mad_top(Words<12>, uint32_t *d, uint32_t &top, const uint32_t *x, uint32_t y) {
  asm("mad.lo.cc.u32 %0, %13, %19, %0;\n\t"
      "madc.hi.cc.u32 %1, %13, %19, %1;\n\t"
      "madc.lo.cc.u32 %2, %14, %19, %2;\n\t"
      "madc.hi.cc.u32 %3, %14, %19, %3;\n\t"
      "madc.lo.cc.u32 %4, %15, %19, %4;\n\t"
      "madc.hi.cc.u32 %5, %15, %19, %5;\n\t"
      "madc.lo.cc.u32 %6, %16, %19, %6;\n\t"
      "madc.hi.cc.u32 %7, %16, %19, %7;\n\t"
      "madc.lo.cc.u32 %8, %17, %19, %8;\n\t"
      "madc.hi.cc.u32 %9, %17, %19, %9;\n\t"
      "madc.lo.cc.u32 %10, %18, %19, %10;\n\t"
      "madc.hi.cc.u32 %11, %18, %19, %11;\n\t"
      "addc.u32 %12, %12, 0;"
      : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3]), "+r"(d[4]), "+r"(d[5]), "+r"(d[6]), "+r"(d[7]), "+r"(d[8]),
        "+r"(d[9]), "+r"(d[10]), "+r"(d[11]), "+r"(top)
      : "r"(x[0]), "r"(x[2]), "r"(x[4]), "r"(x[6]), "r"(x[8]), "r"(x[10]), "r"(y));
}

__device__ __forceinline__ void chain_shift_mad(Words<12>, uint32_t &e0, uint32_t *d, const uint32_t *s, uint32_t top,
                                                const uint32_t *x, uint32_t y) {
  asm("add.cc.u32 %0, %0, %13;\n\t"
      "madc.lo.cc.u32 %1, %25, %31, %14;\n\t"
      "madc.hi.cc.u32 %2, %25, %31, %15;\n\t"
      "madc.lo.cc.u32 %3, %26, %31, %16;\n\t"
      "madc.hi.cc.u32 %4, %26, %31, %17;\n\t"
      "madc.lo.cc.u32 %5, %27, %31, %18;\n\t"
      "madc.hi.cc.u32 %6, %27, %31, %19;\n\t"
      "madc.lo.cc.u32 %7, %28, %31, %20;\n\t"
      "madc.hi.cc.u32 %8, %28, %31, %21;\n\t"
      "madc.lo.cc.u32 %9, %29, %31, %22;\n\t"
      "madc.hi.cc.u32 %10, %29, %31, %23;\n\t"
      "madc.lo.cc.u32 %11, %30, %31, 0;\n\t"
      "madc.hi.u32 %12, %30, %31, %24;"
      : "+&r"(e0), "=&r"(d[0]), "=&r"(d[1]), "=&r"(d[2]), "=&r"(d[3]), "=&r"(d[4]), "=&r"(d[5]), "=&r"(d[6]),
        "=&r"(d[7]), "=&r"(d[8]), "=&r"(d[9]), "=&r"(d[10]), "=&r"(d[11])
      : "r"(s[1]), "r"(s[2]), "r"(s[3]), "r"(s[4]), "r"(s[5]), "r"(s[6]), "r"(s[7]), "r"(s[8]), "r"(s[9]),
        "r"(s[10]), "r"(s[11]), "r"(top), "r"(x[0]), "r"(x[2]), "r"(x[4]), "r"(x[6]), "r"(x[8]), "r"(x[10]), "r"(y));
}

template <class F>
__device__ __forceinline__ void chain_redc(Words<12>, uint32_t *E, uint32_t *O) {
  const uint32_t t = E[0];
  asm("mad.lo.cc.u32 %0, %12, %13, %0;\n\t"
      "madc.hi.cc.u32 %1, %12, %13, %1;\n\t"
      "madc.lo.cc.u32 %2, %12, %14, %2;\n\t"
      "madc.hi.cc.u32 %3, %12, %14, %3;\n\t"
      "madc.lo.cc.u32 %4, %12, %15, %4;\n\t"
      "madc.hi.cc.u32 %5, %12, %15, %5;\n\t"
      "madc.lo.cc.u32 %6, %12, %16, %6;\n\t"
      "madc.hi.cc.u32 %7, %12, %16, %7;\n\t"
      "madc.lo.cc.u32 %8, %12, %17, %8;\n\t"
      "madc.hi.cc.u32 %9, %12, %17, %9;\n\t"
      "madc.lo.cc.u32 %10, %12, %18, %10;\n\t"
      "madc.hi.u32 %11, %12, %18, %11;"
      : "+r"(O[0]), "+r"(O[1]), "+r"(O[2]), "+r"(O[3]), "+r"(O[4]), "+r"(O[5]), "+r"(O[6]), "+r"(O[7]), "+r"(O[8]),
        "+r"(O[9]), "+r"(O[10]), "+r"(O[11])
      : "r"(t), "n"(F::d(0)), "n"(F::d(2)), "n"(F::d(4)), "n"(F::d(6)), "n"(F::d(8)), "n"(F::d(10)));
  O[11] -= t;
  asm("mad.lo.cc.u32 %0, %11, %12, %0;\n\t"
      "madc.hi.cc.u32 %1, %11, %12, %1;\n\t"
      "madc.lo.cc.u32 %2, %11, %13, %2;\n\t"
      "madc.hi.cc.u32 %3, %11, %13, %3;\n\t"
      "madc.lo.cc.u32 %4, %11, %14, %4;\n\t"
      "madc.hi.cc.u32 %5, %11, %14, %5;\n\t"
      "madc.lo.cc.u32 %6, %11, %15, %6;\n\t"
      "madc.hi.cc.u32 %7, %11, %15, %7;\n\t"
      "madc.lo.cc.u32 %8, %11, %16, %8;\n\t"
      "madc.hi.cc.u32 %9, %11, %16, %9;\n\t"
      "addc.u32 %10, %10, 0;"
      : "+r"(E[2]), "+r"(E[3]), "+r"(E[4]), "+r"(E[5]), "+r"(E[6]), "+r"(E[7]), "+r"(E[8]), "+r"(E[9]),
        "+r"(E[10]), "+r"(E[11]), "+r"(O[11])
      : "r"(t), "n"(F::d(1)), "n"(F::d(3)), "n"(F::d(5)), "n"(F::d(7)), "n"(F::d(9)));
}

__device__ __forceinline__ void chain_merge(Words<12>, uint32_t *d, const uint32_t *e, const uint32_t *s) {
  asm("add.cc.u32 %0, %12, %24;\n\t"
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
      "addc.u32 %11, %23, 0;"
      : "=&r"(d[0]), "=&r"(d[1]), "=&r"(d[2]), "=&r"(d[3]), "=&r"(d[4]), "=&r"(d[5]), "=&r"(d[6]), "=&r"(d[7]),
        "=&r"(d[8]), "=&r"(d[9]), "=&r"(d[10]), "=&r"(d[11])
      : "r"(e[0]), "r"(e[1]), "r"(e[2]), "r"(e[3]), "r"(e[4]), "r"(e[5]), "r"(e[6]), "r"(e[7]), "r"(e[8]),
        "r"(e[9]), "r"(e[10]), "r"(e[11]), "r"(s[1]), "r"(s[2]), "r"(s[3]), "r"(s[4]), "r"(s[5]), "r"(s[6]),
        "r"(s[7]), "r"(s[8]), "r"(s[9]), "r"(s[10]), "r"(s[11]));
}

__device__ __forceinline__ void chain_add(Words<12>, uint32_t *d, const uint32_t *a, const uint32_t *b) {
  asm("add.cc.u32 %0, %12, %24;\n\t"
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
      "addc.u32 %11, %23, %35;"
      : "=&r"(d[0]), "=&r"(d[1]), "=&r"(d[2]), "=&r"(d[3]), "=&r"(d[4]), "=&r"(d[5]), "=&r"(d[6]), "=&r"(d[7]),
        "=&r"(d[8]), "=&r"(d[9]), "=&r"(d[10]), "=&r"(d[11])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]), "r"(a[8]),
        "r"(a[9]), "r"(a[10]), "r"(a[11]), "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]),
        "r"(b[6]), "r"(b[7]), "r"(b[8]), "r"(b[9]), "r"(b[10]), "r"(b[11]));
}

// returns all ones when a < b
__device__ __forceinline__ uint32_t chain_sub(Words<12>, uint32_t *d, const uint32_t *a, const uint32_t *b) {
  uint32_t borrow;
  asm("sub.cc.u32 %0, %13, %25;\n\t"
      "subc.cc.u32 %1, %14, %26;\n\t"
      "subc.cc.u32 %2, %15, %27;\n\t"
      "subc.cc.u32 %3, %16, %28;\n\t"
      "subc.cc.u32 %4, %17, %29;\n\t"
      "subc.cc.u32 %5, %18, %30;\n\t"
      "subc.cc.u32 %6, %19, %31;\n\t"
      "subc.cc.u32 %7, %20, %32;\n\t"
      "subc.cc.u32 %8, %21, %33;\n\t"
      "subc.cc.u32 %9, %22, %34;\n\t"
      "subc.cc.u32 %10, %23, %35;\n\t"
      "subc.cc.u32 %11, %24, %36;\n\t"
      "subc.u32 %12, 0, 0;"
      : "=&r"(d[0]), "=&r"(d[1]), "=&r"(d[2]), "=&r"(d[3]), "=&r"(d[4]), "=&r"(d[5]), "=&r"(d[6]), "=&r"(d[7]),
        "=&r"(d[8]), "=&r"(d[9]), "=&r"(d[10]), "=&r"(d[11]), "=&r"(borrow)
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]), "r"(a[8]),
        "r"(a[9]), "r"(a[10]), "r"(a[11]), "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]),
        "r"(b[6]), "r"(b[7]), "r"(b[8]), "r"(b[9]), "r"(b[10]), "r"(b[11]));
  return borrow;
}

__device__ __forceinline__ void chain_mul(Words<24>, uint32_t *d, const uint32_t *x, uint32_t y) {
  asm("mul.lo.u32 %0, %24, %36;\n\t"
      "mul.hi.u32 %1, %24, %36;\n\t"
      "mul.lo.u32 %2, %25, %36;\n\t"
      "mul.hi.u32 %3, %25, %36;\n\t"
      "mul.lo.u32 %4, %26, %36;\n\t"
      "mul.hi.u32 %5, %26, %36;\n\t"
      "mul.lo.u32 %6, %27, %36;\n\t"
      "mul.hi.u32 %7, %27, %36;\n\t"
      "mul.lo.u32 %8, %28, %36;\n\t"
      "mul.hi.u32 %9, %28, %36;\n\t"
      "mul.lo.u32 %10, %29, %36;\n\t"
      "mul.hi.u32 %11, %29, %36;\n\t"
      "mul.lo.u32 %12, %30, %36;\n\t"
      "mul.hi.u32 %13, %30, %36;\n\t"
      "mul.lo.u32 %14, %31, %36;\n\t"
      "mul.hi.u32 %15, %31, %36;\n\t"
      "mul.lo.u32 %16, %32, %36;\n\t"
      "mul.hi.u32 %17, %32, %36;\n\t"
      "mul.lo.u32 %18, %33, %36;\n\t"
      "mul.hi.u32 %19, %33, %36;\n\t"
      "mul.lo.u32 %20, %34, %36;\n\t"
      "mul.hi.u32 %21, %34, %36;\n\t"
      "mul.lo.u32 %22, %35, %36;\n\t"
      "mul.hi.u32 %23, %35, %36;"
      : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3]), "=r"(d[4]), "=r"(d[5]), "=r"(d[6]), "=r"(d[7]), "=r"(d[8]),
        "=r"(d[9]), "=r"(d[10]), "=r"(d[11]), "=r"(d[12]), "=r"(d[13]), "=r"(d[14]), "=r"(d[15]), "=r"(d[16]),
        "=r"(d[17]), "=r"(d[18]), "=r"(d[19]), "=r"(d[20]), "=r"(d[21]), "=r"(d[22]), "=r"(d[23])
      : "r"(x[0]), "r"(x[2]), "r"(x[4]), "r"(x[6]), "r"(x[8]), "r"(x[10]), "r"(x[12]), "r"(x[14]), "r"(x[16]),
        "r"(x[18]), "r"(x[20]), "r"(x[22]), "r"(y));
}

__device__ __forceinline__ void chain_mad(Words<24>, uint32_t *d, const uint32_t *x, uint32_t y) {
  asm("mad.lo.cc.u32 %0, %24, %36, %0;\n\t"
      "madc.hi.cc.u32 %1, %24, %36, %1;\n\t"
      "madc.lo.cc.u32 %2, %25, %36, %2;\n\t"
      "madc.hi.cc.u32 %3, %25, %36, %3;\n\t"
      "madc.lo.cc.u32 %4, %26, %36, %4;\n\t"
      "madc.hi.cc.u32 %5, %26, %36, %5;\n\t"
      "madc.lo.cc.u32 %6, %27, %36, %6;\n\t"
      "madc.hi.cc.u32 %7, %27, %36, %7;\n\t"
      "madc.lo.cc.u32 %8, %28, %36, %8;\n\t"
      "madc.hi.cc.u32 %9, %28, %36, %9;\n\t"
      "madc.lo.cc.u32 %10, %29, %36, %10;\n\t"
      "madc.hi.cc.u32 %11, %29, %36, %11;\n\t"
      "madc.lo.cc.u32 %12, %30, %36, %12;\n\t"
      "madc.hi.cc.u32 %13, %30, %36, %13;\n\t"
      "madc.lo.cc.u32 %14, %31, %36, %14;\n\t"
      "madc.hi.cc.u32 %15, %31, %36, %15;\n\t"
      "madc.lo.cc.u32 %16, %32, %36, %16;\n\t"
      "madc.hi.cc.u32 %17, %32, %36, %17;\n\t"
      "madc.lo.cc.u32 %18, %33, %36, %18;\n\t"
      "madc.hi.cc.u32 %19, %33, %36, %19;\n\t"
      "madc.lo.cc.u32 %20, %34, %36, %20;\n\t"
      "madc.hi.cc.u32 %21, %34, %36, %21;\n\t"
      "madc.lo.cc.u32 %22, %35, %36, %22;\n\t"
      "madc.hi.u32 %23, %35, %36, %23;"
      : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3]), "+r"(d[4]), "+r"(d[5]), "+r"(d[6]), "+r"(d[7]), "+r"(d[8]),
        "+r"(d[9]), "+r"(d[10]), "+r"(d[11]), "+r"(d[12]), "+r"(d[13]), "+r"(d[14]), "+r"(d[15]), "+r"(d[16]),
        "+r"(d[17]), "+r"(d[18]), "+r"(d[19]), "+r"(d[20]), "+r"(d[21]), "+r"(d[22]), "+r"(d[23])
      : "r"(x[0]), "r"(x[2]), "r"(x[4]), "r"(x[6]), "r"(x[8]), "r"(x[10]), "r"(x[12]), "r"(x[14]), "r"(x[16]),
        "r"(x[18]), "r"(x[20]), "r"(x[22]), "r"(y));
}

__device__ __forceinline__ void chain_mad_top(Words<24>, uint32_t *d, uint32_t &top, const uint32_t *x, uint32_t y) {
  asm("mad.lo.cc.u32 %0, %25, %37, %0;\n\t"
      "madc.hi.cc.u32 %1, %25, %37, %1;\n\t"
      "madc.lo.cc.u32 %2, %26, %37, %2;\n\t"
      "madc.hi.cc.u32 %3, %26, %37, %3;\n\t"
      "madc.lo.cc.u32 %4, %27, %37, %4;\n\t"
      "madc.hi.cc.u32 %5, %27, %37, %5;\n\t"
      "madc.lo.cc.u32 %6, %28, %37, %6;\n\t"
      "madc.hi.cc.u32 %7, %28, %37, %7;\n\t"
      "madc.lo.cc.u32 %8, %29, %37, %8;\n\t"
      "madc.hi.cc.u32 %9, %29, %37, %9;\n\t"
      "madc.lo.cc.u32 %10, %30, %37, %10;\n\t"
      "madc.hi.cc.u32 %11, %30, %37, %11;\n\t"
      "madc.lo.cc.u32 %12, %31, %37, %12;\n\t"
      "madc.hi.cc.u32 %13, %31, %37, %13;\n\t"
      "madc.lo.cc.u32 %14, %32, %37, %14;\n\t"
      "madc.hi.cc.u32 %15, %32, %37, %15;\n\t"
      "madc.lo.cc.u32 %16, %33, %37, %16;\n\t"
      "madc.hi.cc.u32 %17, %33, %37, %17;\n\t"
      "madc.lo.cc.u32 %18, %34, %37, %18;\n\t"
      "madc.hi.cc.u32 %19, %34, %37, %19;\n\t"
      "madc.lo.cc.u32 %20, %35, %37, %20;\n\t"
      "madc.hi.cc.u32 %21, %35, %37, %21;\n\t"
      "madc.lo.cc.u32 %22, %36, %37, %22;\n\t"
      "madc.hi.cc.u32 %23, %36, %37, %23;\n\t"
      "addc.u32 %24, %24, 0;"
      : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3]), "+r"(d[4]), "+r"(d[5]), "+r"(d[6]), "+r"(d[7]), "+r"(d[8]),
        "+r"(d[9]), "+r"(d[10]), "+r"(d[11]), "+r"(d[12]), "+r"(d[13]), "+r"(d[14]), "+r"(d[15]), "+r"(d[16]),
        "+r"(d[17]), "+r"(d[18]), "+r"(d[19]), "+r"(d[20]), "+r"(d[21]), "+r"(d[22]), "+r"(d[23]), "+r"(top)
      : "r"(x[0]), "r"(x[2]), "r"(x[4]), "r"(x[6]), "r"(x[8]), "r"(x[10]), "r"(x[12]), "r"(x[14]), "r"(x[16]),
        "r"(x[18]), "r"(x[20]), "r"(x[22]), "r"(y));
}

__device__ __forceinline__ void chain_shift_mad(Words<24>, uint32_t &e0, uint32_t *d, const uint32_t *s, uint32_t top,
                                                const uint32_t *x, uint32_t y) {
  asm("add.cc.u32 %0, %0, %25;\n\t"
      "madc.lo.cc.u32 %1, %49, %61, %26;\n\t"
      "madc.hi.cc.u32 %2, %49, %61, %27;\n\t"
      "madc.lo.cc.u32 %3, %50, %61, %28;\n\t"
      "madc.hi.cc.u32 %4, %50, %61, %29;\n\t"
      "madc.lo.cc.u32 %5, %51, %61, %30;\n\t"
      "madc.hi.cc.u32 %6, %51, %61, %31;\n\t"
      "madc.lo.cc.u32 %7, %52, %61, %32;\n\t"
      "madc.hi.cc.u32 %8, %52, %61, %33;\n\t"
      "madc.lo.cc.u32 %9, %53, %61, %34;\n\t"
      "madc.hi.cc.u32 %10, %53, %61, %35;\n\t"
      "madc.lo.cc.u32 %11, %54, %61, %36;\n\t"
      "madc.hi.cc.u32 %12, %54, %61, %37;\n\t"
      "madc.lo.cc.u32 %13, %55, %61, %38;\n\t"
      "madc.hi.cc.u32 %14, %55, %61, %39;\n\t"
      "madc.lo.cc.u32 %15, %56, %61, %40;\n\t"
      "madc.hi.cc.u32 %16, %56, %61, %41;\n\t"
      "madc.lo.cc.u32 %17, %57, %61, %42;\n\t"
      "madc.hi.cc.u32 %18, %57, %61, %43;\n\t"
      "madc.lo.cc.u32 %19, %58, %61, %44;\n\t"
      "madc.hi.cc.u32 %20, %58, %61, %45;\n\t"
      "madc.lo.cc.u32 %21, %59, %61, %46;\n\t"
      "madc.hi.cc.u32 %22, %59, %61, %47;\n\t"
      "madc.lo.cc.u32 %23, %60, %61, 0;\n\t"
      "madc.hi.u32 %24, %60, %61, %48;"
      : "+&r"(e0), "=&r"(d[0]), "=&r"(d[1]), "=&r"(d[2]), "=&r"(d[3]), "=&r"(d[4]), "=&r"(d[5]), "=&r"(d[6]),
        "=&r"(d[7]), "=&r"(d[8]), "=&r"(d[9]), "=&r"(d[10]), "=&r"(d[11]), "=&r"(d[12]), "=&r"(d[13]),
        "=&r"(d[14]), "=&r"(d[15]), "=&r"(d[16]), "=&r"(d[17]), "=&r"(d[18]), "=&r"(d[19]), "=&r"(d[20]),
        "=&r"(d[21]), "=&r"(d[22]), "=&r"(d[23])
      : "r"(s[1]), "r"(s[2]), "r"(s[3]), "r"(s[4]), "r"(s[5]), "r"(s[6]), "r"(s[7]), "r"(s[8]), "r"(s[9]),
        "r"(s[10]), "r"(s[11]), "r"(s[12]), "r"(s[13]), "r"(s[14]), "r"(s[15]), "r"(s[16]), "r"(s[17]), "r"(s[18]),
        "r"(s[19]), "r"(s[20]), "r"(s[21]), "r"(s[22]), "r"(s[23]), "r"(top), "r"(x[0]), "r"(x[2]), "r"(x[4]),
        "r"(x[6]), "r"(x[8]), "r"(x[10]), "r"(x[12]), "r"(x[14]), "r"(x[16]), "r"(x[18]), "r"(x[20]), "r"(x[22]),
        "r"(y));
}

template <class F>
__device__ __forceinline__ void chain_redc(Words<24>, uint32_t *E, uint32_t *O) {
  const uint32_t t = E[0];
  asm("mad.lo.cc.u32 %0, %24, %25, %0;\n\t"
      "madc.hi.cc.u32 %1, %24, %25, %1;\n\t"
      "madc.lo.cc.u32 %2, %24, %26, %2;\n\t"
      "madc.hi.cc.u32 %3, %24, %26, %3;\n\t"
      "madc.lo.cc.u32 %4, %24, %27, %4;\n\t"
      "madc.hi.cc.u32 %5, %24, %27, %5;\n\t"
      "madc.lo.cc.u32 %6, %24, %28, %6;\n\t"
      "madc.hi.cc.u32 %7, %24, %28, %7;\n\t"
      "madc.lo.cc.u32 %8, %24, %29, %8;\n\t"
      "madc.hi.cc.u32 %9, %24, %29, %9;\n\t"
      "madc.lo.cc.u32 %10, %24, %30, %10;\n\t"
      "madc.hi.cc.u32 %11, %24, %30, %11;\n\t"
      "madc.lo.cc.u32 %12, %24, %31, %12;\n\t"
      "madc.hi.cc.u32 %13, %24, %31, %13;\n\t"
      "madc.lo.cc.u32 %14, %24, %32, %14;\n\t"
      "madc.hi.cc.u32 %15, %24, %32, %15;\n\t"
      "madc.lo.cc.u32 %16, %24, %33, %16;\n\t"
      "madc.hi.cc.u32 %17, %24, %33, %17;\n\t"
      "madc.lo.cc.u32 %18, %24, %34, %18;\n\t"
      "madc.hi.cc.u32 %19, %24, %34, %19;\n\t"
      "madc.lo.cc.u32 %20, %24, %35, %20;\n\t"
      "madc.hi.cc.u32 %21, %24, %35, %21;\n\t"
      "madc.lo.cc.u32 %22, %24, %36, %22;\n\t"
      "madc.hi.u32 %23, %24, %36, %23;"
      : "+r"(O[0]), "+r"(O[1]), "+r"(O[2]), "+r"(O[3]), "+r"(O[4]), "+r"(O[5]), "+r"(O[6]), "+r"(O[7]), "+r"(O[8]),
        "+r"(O[9]), "+r"(O[10]), "+r"(O[11]), "+r"(O[12]), "+r"(O[13]), "+r"(O[14]), "+r"(O[15]), "+r"(O[16]),
        "+r"(O[17]), "+r"(O[18]), "+r"(O[19]), "+r"(O[20]), "+r"(O[21]), "+r"(O[22]), "+r"(O[23])
      : "r"(t), "n"(F::d(0)), "n"(F::d(2)), "n"(F::d(4)), "n"(F::d(6)), "n"(F::d(8)), "n"(F::d(10)), "n"(F::d(12)),
        "n"(F::d(14)), "n"(F::d(16)), "n"(F::d(18)), "n"(F::d(20)), "n"(F::d(22)));
  O[23] -= t;
  asm("mad.lo.cc.u32 %0, %23, %24, %0;\n\t"
      "madc.hi.cc.u32 %1, %23, %24, %1;\n\t"
      "madc.lo.cc.u32 %2, %23, %25, %2;\n\t"
      "madc.hi.cc.u32 %3, %23, %25, %3;\n\t"
      "madc.lo.cc.u32 %4, %23, %26, %4;\n\t"
      "madc.hi.cc.u32 %5, %23, %26, %5;\n\t"
      "madc.lo.cc.u32 %6, %23, %27, %6;\n\t"
      "madc.hi.cc.u32 %7, %23, %27, %7;\n\t"
      "madc.lo.cc.u32 %8, %23, %28, %8;\n\t"
      "madc.hi.cc.u32 %9, %23, %28, %9;\n\t"
      "madc.lo.cc.u32 %10, %23, %29, %10;\n\t"
      "madc.hi.cc.u32 %11, %23, %29, %11;\n\t"
      "madc.lo.cc.u32 %12, %23, %30, %12;\n\t"
      "madc.hi.cc.u32 %13, %23, %30, %13;\n\t"
      "madc.lo.cc.u32 %14, %23, %31, %14;\n\t"
      "madc.hi.cc.u32 %15, %23, %31, %15;\n\t"
      "madc.lo.cc.u32 %16, %23, %32, %16;\n\t"
      "madc.hi.cc.u32 %17, %23, %32, %17;\n\t"
      "madc.lo.cc.u32 %18, %23, %33, %18;\n\t"
      "madc.hi.cc.u32 %19, %23, %33, %19;\n\t"
      "madc.lo.cc.u32 %20, %23, %34, %20;\n\t"
      "madc.hi.cc.u32 %21, %23, %34, %21;\n\t"
      "addc.u32 %22, %22, 0;"
      : "+r"(E[2]), "+r"(E[3]), "+r"(E[4]), "+r"(E[5]), "+r"(E[6]), "+r"(E[7]), "+r"(E[8]), "+r"(E[9]),
        "+r"(E[10]), "+r"(E[11]), "+r"(E[12]), "+r"(E[13]), "+r"(E[14]), "+r"(E[15]), "+r"(E[16]), "+r"(E[17]),
        "+r"(E[18]), "+r"(E[19]), "+r"(E[20]), "+r"(E[21]), "+r"(E[22]), "+r"(E[23]), "+r"(O[23])
      : "r"(t), "n"(F::d(1)), "n"(F::d(3)), "n"(F::d(5)), "n"(F::d(7)), "n"(F::d(9)), "n"(F::d(11)), "n"(F::d(13)),
        "n"(F::d(15)), "n"(F::d(17)), "n"(F::d(19)), "n"(F::d(21)));
}

__device__ __forceinline__ void chain_merge(Words<24>, uint32_t *d, const uint32_t *e, const uint32_t *s) {
  asm("add.cc.u32 %0, %24, %48;\n\t"
      "addc.cc.u32 %1, %25, %49;\n\t"
      "addc.cc.u32 %2, %26, %50;\n\t"
      "addc.cc.u32 %3, %27, %51;\n\t"
      "addc.cc.u32 %4, %28, %52;\n\t"
      "addc.cc.u32 %5, %29, %53;\n\t"
      "addc.cc.u32 %6, %30, %54;\n\t"
      "addc.cc.u32 %7, %31, %55;\n\t"
      "addc.cc.u32 %8, %32, %56;\n\t"
      "addc.cc.u32 %9, %33, %57;\n\t"
      "addc.cc.u32 %10, %34, %58;\n\t"
      "addc.cc.u32 %11, %35, %59;\n\t"
      "addc.cc.u32 %12, %36, %60;\n\t"
      "addc.cc.u32 %13, %37, %61;\n\t"
      "addc.cc.u32 %14, %38, %62;\n\t"
      "addc.cc.u32 %15, %39, %63;\n\t"
      "addc.cc.u32 %16, %40, %64;\n\t"
      "addc.cc.u32 %17, %41, %65;\n\t"
      "addc.cc.u32 %18, %42, %66;\n\t"
      "addc.cc.u32 %19, %43, %67;\n\t"
      "addc.cc.u32 %20, %44, %68;\n\t"
      "addc.cc.u32 %21, %45, %69;\n\t"
      "addc.cc.u32 %22, %46, %70;\n\t"
      "addc.u32 %23, %47, 0;"
      : "=&r"(d[0]), "=&r"(d[1]), "=&r"(d[2]), "=&r"(d[3]), "=&r"(d[4]), "=&r"(d[5]), "=&r"(d[6]), "=&r"(d[7]),
        "=&r"(d[8]), "=&r"(d[9]), "=&r"(d[10]), "=&r"(d[11]), "=&r"(d[12]), "=&r"(d[13]), "=&r"(d[14]),
        "=&r"(d[15]), "=&r"(d[16]), "=&r"(d[17]), "=&r"(d[18]), "=&r"(d[19]), "=&r"(d[20]), "=&r"(d[21]),
        "=&r"(d[22]), "=&r"(d[23])
      : "r"(e[0]), "r"(e[1]), "r"(e[2]), "r"(e[3]), "r"(e[4]), "r"(e[5]), "r"(e[6]), "r"(e[7]), "r"(e[8]),
        "r"(e[9]), "r"(e[10]), "r"(e[11]), "r"(e[12]), "r"(e[13]), "r"(e[14]), "r"(e[15]), "r"(e[16]), "r"(e[17]),
        "r"(e[18]), "r"(e[19]), "r"(e[20]), "r"(e[21]), "r"(e[22]), "r"(e[23]), "r"(s[1]), "r"(s[2]), "r"(s[3]),
        "r"(s[4]), "r"(s[5]), "r"(s[6]), "r"(s[7]), "r"(s[8]), "r"(s[9]), "r"(s[10]), "r"(s[11]), "r"(s[12]),
        "r"(s[13]), "r"(s[14]), "r"(s[15]), "r"(s[16]), "r"(s[17]), "r"(s[18]), "r"(s[19]), "r"(s[20]), "r"(s[21]),
        "r"(s[22]), "r"(s[23]));
}

__device__ __forceinline__ void chain_add(Words<24>, uint32_t *d, const uint32_t *a, const uint32_t *b) {
  asm("add.cc.u32 %0, %24, %48;\n\t"
      "addc.cc.u32 %1, %25, %49;\n\t"
      "addc.cc.u32 %2, %26, %50;\n\t"
      "addc.cc.u32 %3, %27, %51;\n\t"
      "addc.cc.u32 %4, %28, %52;\n\t"
      "addc.cc.u32 %5, %29, %53;\n\t"
      "addc.cc.u32 %6, %30, %54;\n\t"
      "addc.cc.u32 %7, %31, %55;\n\t"
      "addc.cc.u32 %8, %32, %56;\n\t"
      "addc.cc.u32 %9, %33, %57;\n\t"
      "addc.cc.u32 %10, %34, %58;\n\t"
      "addc.cc.u32 %11, %35, %59;\n\t"
      "addc.cc.u32 %12, %36, %60;\n\t"
      "addc.cc.u32 %13, %37, %61;\n\t"
      "addc.cc.u32 %14, %38, %62;\n\t"
      "addc.cc.u32 %15, %39, %63;\n\t"
      "addc.cc.u32 %16, %40, %64;\n\t"
      "addc.cc.u32 %17, %41, %65;\n\t"
      "addc.cc.u32 %18, %42, %66;\n\t"
      "addc.cc.u32 %19, %43, %67;\n\t"
      "addc.cc.u32 %20, %44, %68;\n\t"
      "addc.cc.u32 %21, %45, %69;\n\t"
      "addc.cc.u32 %22, %46, %70;\n\t"
      "addc.u32 %23, %47, %71;"
      : "=&r"(d[0]), "=&r"(d[1]), "=&r"(d[2]), "=&r"(d[3]), "=&r"(d[4]), "=&r"(d[5]), "=&r"(d[6]), "=&r"(d[7]),
        "=&r"(d[8]), "=&r"(d[9]), "=&r"(d[10]), "=&r"(d[11]), "=&r"(d[12]), "=&r"(d[13]), "=&r"(d[14]),
        "=&r"(d[15]), "=&r"(d[16]), "=&r"(d[17]), "=&r"(d[18]), "=&r"(d[19]), "=&r"(d[20]), "=&r"(d[21]),
        "=&r"(d[22]), "=&r"(d[23])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]), "r"(a[8]),
        "r"(a[9]), "r"(a[10]), "r"(a[11]), "r"(a[12]), "r"(a[13]), "r"(a[14]), "r"(a[15]), "r"(a[16]), "r"(a[17]),
        "r"(a[18]), "r"(a[19]), "r"(a[20]), "r"(a[21]), "r"(a[22]), "r"(a[23]), "r"(b[0]), "r"(b[1]), "r"(b[2]),
        "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]), "r"(b[8]), "r"(b[9]), "r"(b[10]), "r"(b[11]),
        "r"(b[12]), "r"(b[13]), "r"(b[14]), "r"(b[15]), "r"(b[16]), "r"(b[17]), "r"(b[18]), "r"(b[19]), "r"(b[20]),
        "r"(b[21]), "r"(b[22]), "r"(b[23]));
}

// returns all ones when a < b
__device__ __forceinline__ uint32_t chain_sub(Words<24>, uint32_t *d, const uint32_t *a, const uint32_t *b) {
  uint32_t borrow;
  asm("sub.cc.u32 %0, %25, %49;\n\t"
      "subc.cc.u32 %1, %26, %50;\n\t"
      "subc.cc.u32 %2, %27, %51;\n\t"
      "subc.cc.u32 %3, %28, %52;\n\t"
      "subc.cc.u32 %4, %29, %53;\n\t"
      "subc.cc.u32 %5, %30, %54;\n\t"
      "subc.cc.u32 %6, %31, %55;\n\t"
      "subc.cc.u32 %7, %32, %56;\n\t"
      "subc.cc.u32 %8, %33, %57;\n\t"
      "subc.cc.u32 %9, %34, %58;\n\t"
      "subc.cc.u32 %10, %35, %59;\n\t"
      "subc.cc.u32 %11, %36, %60;\n\t"
      "subc.cc.u32 %12, %37, %61;\n\t"
      "subc.cc.u32 %13, %38, %62;\n\t"
      "subc.cc.u32 %14, %39, %63;\n\t"
      "subc.cc.u32 %15, %40, %64;\n\t"
      "subc.cc.u32 %16, %41, %65;\n\t"
      "subc.cc.u32 %17, %42, %66;\n\t"
      "subc.cc.u32 %18, %43, %67;\n\t"
      "subc.cc.u32 %19, %44, %68;\n\t"
      "subc.cc.u32 %20, %45, %69;\n\t"
      "subc.cc.u32 %21, %46, %70;\n\t"
      "subc.cc.u32 %22, %47, %71;\n\t"
      "subc.cc.u32 %23, %48, %72;\n\t"
      "subc.u32 %24, 0, 0;"
      : "=&r"(d[0]), "=&r"(d[1]), "=&r"(d[2]), "=&r"(d[3]), "=&r"(d[4]), "=&r"(d[5]), "=&r"(d[6]), "=&r"(d[7]),
        "=&r"(d[8]), "=&r"(d[9]), "=&r"(d[10]), "=&r"(d[11]), "=&r"(d[12]), "=&r"(d[13]), "=&r"(d[14]),
        "=&r"(d[15]), "=&r"(d[16]), "=&r"(d[17]), "=&r"(d[18]), "=&r"(d[19]), "=&r"(d[20]), "=&r"(d[21]),
        "=&r"(d[22]), "=&r"(d[23]), "=&r"(borrow)
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]), "r"(a[8]),
        "r"(a[9]), "r"(a[10]), "r"(a[11]), "r"(a[12]), "r"(a[13]), "r"(a[14]), "r"(a[15]), "r"(a[16]), "r"(a[17]),
        "r"(a[18]), "r"(a[19]), "r"(a[20]), "r"(a[21]), "r"(a[22]), "r"(a[23]), "r"(b[0]), "r"(b[1]), "r"(b[2]),
        "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]), "r"(b[8]), "r"(b[9]), "r"(b[10]), "r"(b[11]),
        "r"(b[12]), "r"(b[13]), "r"(b[14]), "r"(b[15]), "r"(b[16]), "r"(b[17]), "r"(b[18]), "r"(b[19]), "r"(b[20]),
        "r"(b[21]), "r"(b[22]), "r"(b[23]));
  return borrow;
}

// r += p 2^k (k = 0, 1) when mask is nonzero
template <class F, int K>
__device__ __forceinline__ void wide_add_p_if(uint32_t *r, uint32_t mask) {
  uint32_t q[F::L];
#pragma unroll
  for (int j = 0; j < F::L; ++j) q[j] = mask & (K ? F::p(j) << 1 | (j ? F::p(j - 1) >> 31 : 0u) : F::p(j));
  uint32_t s[F::L];
  chain_add(Words<F::L>{}, s, r, q);
#pragma unroll
  for (int j = 0; j < F::L; ++j) r[j] = s[j];
}

// r = a b 2^(-32 L) mod p for a < p and any b of L words; canonical; r may alias.
template <class F>
__device__ __forceinline__ void wide_mul(uint32_t *r, const uint32_t *a, const uint32_t *b) {
  constexpr int L = F::L;
  constexpr Words<L> W{};
  uint32_t E[L], O[L];
  chain_mul(W, E, a, b[0]);
  chain_mul(W, O, a + 1, b[0]);
  chain_redc<F>(W, E, O);
#pragma unroll
  for (int i = 1; i < L; ++i) {
    uint32_t X[L];
    chain_shift_mad(W, O[0], X, E, (uint32_t)((int32_t)O[L - 1] >> 31), a + 1, b[i]);
    chain_mad_top(W, O, X[L - 1], a, b[i]);
    chain_redc<F>(W, O, X);
#pragma unroll
    for (int j = 0; j < L; ++j) {
      E[j] = O[j];
      O[j] = X[j];
    }
  }
  uint32_t t[L];
  chain_merge(W, t, O, E);   // in (-p, p)
  wide_add_p_if<F, 0>(t, (uint32_t)((int32_t)t[L - 1] >> 31));
#pragma unroll
  for (int j = 0; j < L; ++j) r[j] = t[j];
}

// r = x w mod p, below 2p, for x < 2p and w as the residues A = w 2^(16 L), B = w
// 2^(32 L): (x_lo A + x_hi B - M p) 2^(-16 L) lies in (-p, 1.02 p).
template <class F>
__device__ __forceinline__ void wide_mul_split(uint32_t *r, const uint32_t *x, const uint32_t *A, const uint32_t *B) {
  constexpr int L = F::L, H = L / 2;
  constexpr Words<L> W{};
  uint32_t E[L], O[L];
#pragma unroll
  for (int i = 0; i < H; ++i) {
    if (i == 0) {
      chain_mul(W, E, A, x[0]);
      chain_mul(W, O, A + 1, x[0]);
    } else {
      uint32_t X[L];
      chain_shift_mad(W, O[0], X, E, (uint32_t)((int32_t)O[L - 1] >> 31), A + 1, x[i]);
      chain_mad_top(W, O, X[L - 1], A, x[i]);
#pragma unroll
      for (int j = 0; j < L; ++j) {
        E[j] = O[j];
        O[j] = X[j];
      }
    }
    chain_mad(W, O, B + 1, x[H + i]);
    chain_mad_top(W, E, O[L - 1], B, x[H + i]);
    chain_redc<F>(W, E, O);
  }
  uint32_t t[L];
  chain_merge(W, t, O, E);
  wide_add_p_if<F, 0>(t, (uint32_t)((int32_t)t[L - 1] >> 31));
#pragma unroll
  for (int j = 0; j < L; ++j) r[j] = t[j];
}

// r - 2^K p when that is not negative
template <class F, int K>
__device__ __forceinline__ void wide_reduce_once(uint32_t *r) {
  constexpr int L = F::L;
  uint32_t q[L], d[L];
#pragma unroll
  for (int j = 0; j < L; ++j) q[j] = K ? F::p(j) << 1 | (j ? F::p(j - 1) >> 31 : 0u) : F::p(j);
  const uint32_t borrow = chain_sub(Words<L>{}, d, r, q);
#pragma unroll
  for (int j = 0; j < L; ++j) r[j] = borrow ? r[j] : d[j];
}

// r = a + b, a - b mod 2p for a, b < 2p
template <class F>
__device__ __forceinline__ void wide_add_lazy(uint32_t *r, const uint32_t *a, const uint32_t *b) {
  uint32_t s[F::L];
  chain_add(Words<F::L>{}, s, a, b);
  wide_reduce_once<F, 1>(s);
#pragma unroll
  for (int j = 0; j < F::L; ++j) r[j] = s[j];
}

template <class F>
__device__ __forceinline__ void wide_sub_lazy(uint32_t *r, const uint32_t *a, const uint32_t *b) {
  uint32_t d[F::L];
  const uint32_t borrow = chain_sub(Words<F::L>{}, d, a, b);
  wide_add_p_if<F, 1>(d, borrow);
#pragma unroll
  for (int j = 0; j < F::L; ++j) r[j] = d[j];
}

}  // namespace gb300ntt
