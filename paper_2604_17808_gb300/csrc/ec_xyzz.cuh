// ec_xyzz.cuh -- short-Weierstrass point arithmetic (y^2 = x^3 + b) for the
// multi-scalar multiplication, sm_103a, generic over the base field.
//
// Curves (MORPH, Sec. 2.3.1 and Algorithm 2; the paper's 256-bit MSM column
// read as BN254 G1): BN254 G1 (y^2 = x^3 + 3 over a 254-bit field) and
// BLS12-381 G1 (y^2 = x^3 + 4 over a 381-bit field).  Neither has a twisted
// Edwards model over its base field (no point of order two in the group the
// MSM uses), so the buckets use XYZZ coordinates: (X, Y, ZZ, ZZZ) stands for
// the affine point (X / ZZ, Y / ZZZ) with ZZ^3 = ZZZ^2, and ZZ = 0 marks the
// point at infinity O.  The formulas are the "xyzz" ones of the
// Explicit-Formulas Database (Bernstein and Lange): madd-2008-s (bucket +=
// affine point, 8M + 2S), add-2008-s (12M + 2S), dbl-2008-s-1 (6M + 3S) and
// mdbl-2008-s-1, with the cases the formulas exclude (an operand O, P = Q,
// P = -Q) taken explicitly.
//
// Every coordinate is in Montgomery form and canonical.  A field "traits"
// type T supplies the limb count T::L and the operations (product, sum,
// difference, reduction, canonical check, 32-byte or 48-byte memory access).
#pragma once

#include "fp256.cuh"
#include "fp384.cuh"
#include "fp_square.cuh"

namespace gb300ntt {

// BN254 base field q (254 bits).
struct FieldBn254Fq {
  static constexpr int kId = 2;
  static constexpr bool kSubtract = false;
  static constexpr uint32_t P0 = 0xd87cfd47u, P1 = 0x3c208c16u, P2 = 0x6871ca8du, P3 = 0x97816a91u,
                            P4 = 0x8181585du, P5 = 0xb85045b6u, P6 = 0xe131a029u, P7 = 0x30644e72u;
  static constexpr uint32_t NP = neg_inv_u32(P0);
};
static_assert(FieldBn254Fq::P0 * (0u - FieldBn254Fq::NP) == 1u, "NP");

// ------------------------------------------------------------ field traits

struct FqBn254 {
  static constexpr int L = 8;
  using F = FieldBn254Fq;
  __device__ static void mul(uint32_t r[8], const uint32_t a[8], const uint32_t b[8]) { mont_mul<F>(r, a, b); }
  __device__ static void add(uint32_t r[8], const uint32_t a[8], const uint32_t b[8]) { add_mod<F>(r, a, b); }
  __device__ static void sub(uint32_t r[8], const uint32_t a[8], const uint32_t b[8]) { sub_mod<F>(r, a, b); }
  __device__ static void redc(uint32_t r[8], const uint32_t a[8]) { mont_redc<F>(r, a); }
  __device__ static void reduce(uint32_t r[8], const uint32_t t[8]) { reduce_once<F>(r, t); }   // t < 2p
  __device__ static bool canonical(const uint32_t a[8]) {
    const uint32_t p[8] = {F::P0, F::P1, F::P2, F::P3, F::P4, F::P5, F::P6, F::P7};
#pragma unroll
    for (int j = 7; j >= 0; --j)
      if (a[j] != p[j]) return a[j] < p[j];
    return false;
  }
  __device__ static constexpr uint32_t modulus(int j) {
    return j == 0 ? F::P0 : j == 1 ? F::P1 : j == 2 ? F::P2 : j == 3 ? F::P3 : j == 4 ? F::P4 : j == 5 ? F::P5
         : j == 6 ? F::P6 : F::P7;
  }
  __device__ static void load(uint32_t r[8], const uint4 *base, uint64_t e) { fe_load_global(r, base, e); }
  __device__ static void store(uint4 *base, uint64_t e, const uint32_t a[8]) { fe_store_global(base, e, a); }
};

struct FqBls381 {
  static constexpr int L = 12;
  using F = FieldBls12381Fq;
  __device__ static void mul(uint32_t r[12], const uint32_t a[12], const uint32_t b[12]) { fp384::mont_mul(r, a, b); }
  __device__ static void add(uint32_t r[12], const uint32_t a[12], const uint32_t b[12]) { fp384::add_mod(r, a, b); }
  __device__ static void sub(uint32_t r[12], const uint32_t a[12], const uint32_t b[12]) { fp384::sub_mod(r, a, b); }
  __device__ static void redc(uint32_t r[12], const uint32_t a[12]) { fp384::mont_redc(r, a); }
  __device__ static void reduce(uint32_t r[12], const uint32_t t[12]) { fp384::reduce_once(r, t); }   // t < 2p
  __device__ static bool canonical(const uint32_t a[12]) { return fp384::is_canonical(a); }
  __device__ static constexpr uint32_t modulus(int j) {
    return j == 0 ? F::P0 : j == 1 ? F::P1 : j == 2 ? F::P2 : j == 3 ? F::P3 : j == 4 ? F::P4 : j == 5 ? F::P5
         : j == 6 ? F::P6 : j == 7 ? F::P7 : j == 8 ? F::P8 : j == 9 ? F::P9 : j == 10 ? F::P10 : F::P11;
  }
  __device__ static void load(uint32_t r[12], const uint4 *base, uint64_t e) { fp384::load(r, base, e); }
  __device__ static void store(uint4 *base, uint64_t e, const uint32_t a[12]) { fp384::store(base, e, a); }
};

// ------------------------------------------------------ generic limb helpers

template <int L>
__device__ __forceinline__ bool fv_is_zero(const uint32_t a[L]) {
  uint32_t o = 0;
#pragma unroll
  for (int j = 0; j < L; ++j) o |= a[j];
  return o == 0u;
}

template <int L>
__device__ __forceinline__ bool fv_equal(const uint32_t a[L], const uint32_t b[L]) {
  uint32_t o = 0;
#pragma unroll
  for (int j = 0; j < L; ++j) o |= a[j] ^ b[j];
  return o == 0u;
}

template <int L>
__device__ __forceinline__ void fv_zero(uint32_t a[L]) {
#pragma unroll
  for (int j = 0; j < L; ++j) a[j] = 0u;
}

template <int L>
__device__ __forceinline__ void fv_copy(uint32_t r[L], const uint32_t a[L]) {
#pragma unroll
  for (int j = 0; j < L; ++j) r[j] = a[j];
}

// The field product as an out-of-line call with the operands passed by value
// (they travel in registers; no stack frame).  The mixed addition of the
// bucket-accumulation loop uses it: one shared copy of the product instead
// of ten inlined copies keeps the loop inside the instruction cache
// (measured on GB300, BN254: the whole MSM at 2^24 points 9% faster).
// xyzz_add / xyzz_dbl take the call when kCall is set (the reduction-tree
// and combine kernels, where it also measured faster); elsewhere the product
// is inlined.
template <class T>
struct FeV {
  uint32_t v[T::L];
};

template <class T>
__device__ __noinline__ FeV<T> f_mul_call(FeV<T> a, FeV<T> b) {
  FeV<T> r;
  T::mul(r.v, a.v, b.v);
  return r;
}

template <class T, bool kCall>
__device__ __forceinline__ void f_mul(uint32_t r[T::L], const uint32_t a[T::L], const uint32_t b[T::L]) {
  if constexpr (kCall) {
    FeV<T> x, y;
#pragma unroll
    for (int j = 0; j < T::L; ++j) {
      x.v[j] = a[j];
      y.v[j] = b[j];
    }
    const FeV<T> z = f_mul_call<T>(x, y);
#pragma unroll
    for (int j = 0; j < T::L; ++j) r[j] = z.v[j];
  } else {
    T::mul(r, a, b);
  }
}

// r = a^2
template <class T>
__device__ __noinline__ FeV<T> f_sqr_call(FeV<T> a) {
  FeV<T> r;
  field_square<T>(r.v, a.v);
  return r;
}

template <class T, bool kCall>
__device__ __forceinline__ void f_sqr(uint32_t r[T::L], const uint32_t a[T::L]) {
  if constexpr (kCall) {
    FeV<T> x;
    fv_copy<T::L>(x.v, a);
    const FeV<T> z = f_sqr_call<T>(x);
    fv_copy<T::L>(r, z.v);
  } else {
    field_square<T>(r, a);
  }
}

// r = a b - c d
template <class T>
__device__ __forceinline__ void f_mul_sub(uint32_t r[T::L], const uint32_t a[T::L], const uint32_t b[T::L],
                                          const uint32_t c[T::L], const uint32_t d[T::L]) {
  uint32_t p[T::L], n[T::L];
#pragma unroll
  for (int j = 0; j < T::L; ++j) p[j] = T::modulus(j);
  words_sub<T::L>(n, p, c);   // p - c, p for c = 0
  field_mul2<T>(r, a, b, n, d);
}

template <class T>
struct Xyzz {
  uint32_t X[T::L], Y[T::L], ZZ[T::L], ZZZ[T::L];
};

template <class T>
__device__ __forceinline__ void xyzz_set_inf(Xyzz<T> &r) {
  fv_zero<T::L>(r.X);
  fv_zero<T::L>(r.Y);
  fv_zero<T::L>(r.ZZ);
  fv_zero<T::L>(r.ZZZ);
}

template <class T>
__device__ __forceinline__ bool xyzz_is_inf(const Xyzz<T> &p) { return fv_is_zero<T::L>(p.ZZ); }

// r = 2 (x, y) for an affine point (x, y) (mdbl-2008-s-1, a = 0).
template <class T>
__device__ __forceinline__ void xyzz_mdbl(Xyzz<T> &r, const uint32_t x[T::L], const uint32_t y[T::L]) {
  constexpr int L = T::L;
  uint32_t U[L], V[L], W[L], S[L], M[L];
  T::add(U, y, y);      // U = 2 y
  T::mul(V, U, U);      // V = U^2
  T::mul(W, U, V);      // W = U V
  T::mul(S, x, V);      // S = x V
  T::mul(M, x, x);
  T::add(U, M, M);
  T::add(M, U, M);      // M = 3 x^2
  T::mul(U, M, M);
  T::sub(U, U, S);
  T::sub(U, U, S);      // X3 = M^2 - 2 S
  T::sub(S, S, U);
  T::mul(S, M, S);      // M (S - X3)
  T::mul(M, W, y);
  T::sub(r.Y, S, M);    // Y3 = M (S - X3) - W y
  fv_copy<L>(r.X, U);
  fv_copy<L>(r.ZZ, V);  // ZZ3 = V
  fv_copy<L>(r.ZZZ, W); // ZZZ3 = W
}

// r = 2 p (dbl-2008-s-1, a = 0); r may alias p.  2 O = O follows from the
// formulas (ZZ3 = V ZZ1 = 0).
template <class T, bool kCall = false>
__device__ __forceinline__ void xyzz_dbl(Xyzz<T> &r, const Xyzz<T> &p) {
  constexpr int L = T::L;
  uint32_t U[L], V[L], W[L], S[L], M[L];
  T::add(U, p.Y, p.Y);            // U = 2 Y1
  f_sqr<T, kCall>(V, U);         // V = U^2
  f_mul<T, kCall>(W, U, V);       // W = U V
  f_mul<T, kCall>(S, p.X, V);     // S = X1 V
  f_sqr<T, kCall>(M, p.X);
  T::add(U, M, M);
  T::add(M, U, M);                // M = 3 X1^2
  f_mul<T, kCall>(r.ZZ, V, p.ZZ);    // ZZ3 = V ZZ1
  f_mul<T, kCall>(r.ZZZ, W, p.ZZZ);  // ZZZ3 = W ZZZ1
  f_sqr<T, kCall>(U, M);
  T::sub(U, U, S);
  T::sub(U, U, S);                // X3 = M^2 - 2 S
  T::sub(S, S, U);
  f_mul_sub<T>(r.Y, M, S, W, p.Y);   // Y3 = M (S - X3) - W Y1
  fv_copy<L>(r.X, U);
}

// acc += (x2, y2), an affine point that is not O (madd-2008-s).
template <class T>
__device__ __forceinline__ void xyzz_madd(Xyzz<T> &acc, const uint32_t x2[T::L], const uint32_t y2[T::L],
                                          const uint32_t one[T::L]) {
  constexpr int L = T::L;
  if (xyzz_is_inf(acc)) {
    fv_copy<L>(acc.X, x2);
    fv_copy<L>(acc.Y, y2);
    fv_copy<L>(acc.ZZ, one);
    fv_copy<L>(acc.ZZZ, one);
    return;
  }
  uint32_t P[L], R[L], PP[L], PPP[L], Q[L];
  f_mul<T, true>(P, x2, acc.ZZ);
  T::sub(P, P, acc.X);            // P = U2 - X1
  f_mul<T, true>(R, y2, acc.ZZZ);
  T::sub(R, R, acc.Y);            // R = S2 - Y1
  if (fv_is_zero<L>(P)) {
    if (fv_is_zero<L>(R)) xyzz_mdbl<T>(acc, x2, y2);  // same point
    else xyzz_set_inf(acc);                          // opposite points
    return;
  }
  f_sqr<T, true>(PP, P);
  f_mul<T, true>(PPP, P, PP);
  f_mul<T, true>(acc.ZZ, acc.ZZ, PP);     // ZZ3 = ZZ1 PP
  f_mul<T, true>(acc.ZZZ, acc.ZZZ, PPP);  // ZZZ3 = ZZZ1 PPP
  f_mul<T, true>(Q, acc.X, PP);           // Q = X1 PP
  f_sqr<T, true>(P, R);
  T::sub(P, P, PPP);
  T::sub(P, P, Q);
  T::sub(P, P, Q);                        // X3 = R^2 - PPP - 2 Q
  T::sub(Q, Q, P);
  f_mul_sub<T>(acc.Y, R, Q, acc.Y, PPP);  // Y3 = R (Q - X3) - Y1 PPP
  fv_copy<L>(acc.X, P);
}

// acc += q (add-2008-s).
template <class T, bool kCall = false>
__device__ __forceinline__ void xyzz_add(Xyzz<T> &acc, const Xyzz<T> &q) {
  constexpr int L = T::L;
  if (xyzz_is_inf(q)) return;
  if (xyzz_is_inf(acc)) {
    acc = q;
    return;
  }
  uint32_t U1[L], S1[L], P[L], R[L], PP[L], PPP[L];
  f_mul<T, kCall>(U1, acc.X, q.ZZ);       // U1 = X1 ZZ2
  f_mul<T, kCall>(S1, acc.Y, q.ZZZ);      // S1 = Y1 ZZZ2
  f_mul<T, kCall>(P, q.X, acc.ZZ);
  T::sub(P, P, U1);                       // P = U2 - U1
  f_mul<T, kCall>(R, q.Y, acc.ZZZ);
  T::sub(R, R, S1);                       // R = S2 - S1
  if (fv_is_zero<L>(P)) {
    if (fv_is_zero<L>(R)) xyzz_dbl<T, kCall>(acc, q);
    else xyzz_set_inf(acc);
    return;
  }
  f_sqr<T, kCall>(PP, P);
  f_mul<T, kCall>(PPP, P, PP);
  f_mul<T, kCall>(acc.ZZ, acc.ZZ, q.ZZ);
  f_mul<T, kCall>(acc.ZZ, acc.ZZ, PP);    // ZZ3 = ZZ1 ZZ2 PP
  f_mul<T, kCall>(acc.ZZZ, acc.ZZZ, q.ZZZ);
  f_mul<T, kCall>(acc.ZZZ, acc.ZZZ, PPP); // ZZZ3 = ZZZ1 ZZZ2 PPP
  f_mul<T, kCall>(U1, U1, PP);            // Q = U1 PP
  f_sqr<T, kCall>(P, R);
  T::sub(P, P, PPP);
  T::sub(P, P, U1);
  T::sub(P, P, U1);                       // X3 = R^2 - PPP - 2 Q
  T::sub(U1, U1, P);
  f_mul_sub<T>(acc.Y, R, U1, S1, PPP);    // Y3 = R (Q - X3) - S1 PPP
  fv_copy<L>(acc.X, P);
}

// ------------------------------------------------------------- inversion
// By division steps (Bernstein and Yang, "Fast constant-time gcd computation
// and modular inversion", TCHES 2019), 30 at a time: the steps on the low bits
// of (f, g) give a 2 x 2 matrix with entries up to 2^30, which is then applied
// to the long f, g (divided by 2^30) and to d, e mod q (divided by 2^30 mod q).
// From f = q, g = a, d = 0, e = c it ends in g = 0, f = +-1, d = +-c / a.  Long
// numbers are signed, in 30-bit limbs.  About 25 (254-bit q) or 37 (381-bit)
// batches of some 600 instructions, against 380 or 570 dependent products of
// 300 to 600 by Fermat's little theorem: one inversion alone on an SM took 571
// us over the 381-bit field that way.
template <int L>
struct Div30 {
  static constexpr int N = (32 * L + 29) / 30;   // 9 or 13 limbs: 270, 390 bits
  static constexpr uint32_t kMask = (1u << 30) - 1u;
  int32_t v[N];
};

template <int L>
__device__ __forceinline__ void div30_from_words(Div30<L> &r, const uint32_t x[L]) {
#pragma unroll
  for (int j = 0; j < Div30<L>::N; ++j) {
    const int bit = 30 * j, w = bit >> 5, sh = bit & 31;
    const uint32_t lo = w < L ? x[w] : 0u, hi = w + 1 < L ? x[w + 1] : 0u;
    r.v[j] = (int32_t)(__funnelshift_r(lo, hi, sh) & Div30<L>::kMask);
  }
}

// r = a^-1 in Montgomery form for a in Montgomery form (r2 = 2^(64 L) mod q);
// a = 0 gives 0.
template <class T>
__device__ __noinline__ void f_inverse(uint32_t r[T::L], const uint32_t a[T::L], const uint32_t r2[T::L]) {
  constexpr int L = T::L, N = Div30<L>::N;
  constexpr uint32_t kMask = Div30<L>::kMask;
  if (fv_is_zero<L>(a)) {
    fv_zero<L>(r);
    return;
  }
  Div30<L> q, f, g, d, e;
  {
    uint32_t qw[L];
#pragma unroll
    for (int j = 0; j < L; ++j) qw[j] = T::modulus(j);
    div30_from_words<L>(q, qw);
  }
  f = q;
  div30_from_words<L>(g, a);
  div30_from_words<L>(e, r2);   // a = x R: d ends as R^2 / (x R) = R / x
#pragma unroll
  for (int j = 0; j < N; ++j) d.v[j] = 0;
  int32_t delta = 1;
  // (49 * 381 + 57) / 17 = 1101 steps always suffice for 381 bits
#pragma unroll 1
  for (int batch = 0; batch < 40; ++batch) {
    int32_t u = 1, v = 0, s = 0, t = 1;   // f' = u f + v g, g' = s f + t g
    {
      // 32 low bits of f and g: the 30 steps look at 30 of them
      uint32_t fl = (uint32_t)f.v[0] | (uint32_t)f.v[1] << 30, gl = (uint32_t)g.v[0] | (uint32_t)g.v[1] << 30;
      int left = 30;
#pragma unroll 1
      for (;;) {
        const int z = min(left, __clz(__brev(gl)));   // even g: halve it
        gl >>= z;
        u = (int32_t)((uint32_t)u << z);
        v = (int32_t)((uint32_t)v << z);
        delta += z;
        left -= z;
        if (left == 0) break;
        if (delta > 0) {   // (f, g) -> (g, -f): the sum below is then g - f
          delta = -delta;
          const uint32_t x = fl;
          fl = gl;
          gl = 0u - x;
          const int32_t y = u, w = v;
          u = s;
          v = t;
          s = -y;
          t = -w;
        }
        gl += fl;
        s += u;
        t += v;
        // the halving of this step comes with the next run of zeros
      }
    }
    // f, g
    {
      int64_t cf = (int64_t)u * f.v[0] + (int64_t)v * g.v[0], cg = (int64_t)s * f.v[0] + (int64_t)t * g.v[0];
      cf >>= 30;   // the low 30 bits are zero
      cg >>= 30;
#pragma unroll
      for (int j = 1; j < N; ++j) {
        cf += (int64_t)u * f.v[j] + (int64_t)v * g.v[j];
        cg += (int64_t)s * f.v[j] + (int64_t)t * g.v[j];
        f.v[j - 1] = (int32_t)((uint32_t)cf & kMask);
        g.v[j - 1] = (int32_t)((uint32_t)cg & kMask);
        cf >>= 30;
        cg >>= 30;
      }
      f.v[N - 1] = (int32_t)cf;
      g.v[N - 1] = (int32_t)cg;
    }
    // d, e: plus the multiple of q, |m| <= 2^29, that makes the low 30 bits
    // zero; |d|, |e| grow by at most q / 2 per batch, 21 q in all, which the
    // spare bits of the top limb hold
    {
      int64_t cd = (int64_t)u * d.v[0] + (int64_t)v * e.v[0], ce = (int64_t)s * d.v[0] + (int64_t)t * e.v[0];
      const int32_t md = (int32_t)(((uint32_t)cd * T::F::NP) << 2) >> 2;
      const int32_t me = (int32_t)(((uint32_t)ce * T::F::NP) << 2) >> 2;
      cd = (cd + (int64_t)md * q.v[0]) >> 30;
      ce = (ce + (int64_t)me * q.v[0]) >> 30;
#pragma unroll
      for (int j = 1; j < N; ++j) {
        cd += (int64_t)u * d.v[j] + (int64_t)v * e.v[j];
        ce += (int64_t)s * d.v[j] + (int64_t)t * e.v[j];
        cd += (int64_t)md * q.v[j];
        ce += (int64_t)me * q.v[j];
        d.v[j - 1] = (int32_t)((uint32_t)cd & kMask);
        e.v[j - 1] = (int32_t)((uint32_t)ce & kMask);
        cd >>= 30;
        ce >>= 30;
      }
      d.v[N - 1] = (int32_t)cd;
      e.v[N - 1] = (int32_t)ce;
    }
    int32_t nz = 0;
#pragma unroll
    for (int j = 0; j < N; ++j) nz |= g.v[j];
    if (nz == 0) break;
  }
  // f = 1 or -1 (all limbs' sum: the top limb carries the sign); d f mod q
  const int32_t sign = f.v[N - 1] < 0 ? -1 : 0;
  int32_t c = 0;
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const int32_t w = (d.v[j] ^ sign) - sign + c;   // +-d, limb by limb
    c = j + 1 < N ? w >> 30 : 0;
    d.v[j] = j + 1 < N ? (int32_t)((uint32_t)w & kMask) : w;
  }
  // into [0, q): |d| < 22 q
#pragma unroll 1
  for (int k = 0; k < 48; ++k) {
    const bool neg = d.v[N - 1] < 0;
    Div30<L> w;
    c = 0;
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const int32_t x = d.v[j] + (neg ? q.v[j] : -q.v[j]) + c;
      c = j + 1 < N ? x >> 30 : 0;
      w.v[j] = j + 1 < N ? (int32_t)((uint32_t)x & kMask) : x;
    }
    if (!neg && w.v[N - 1] < 0) break;   // 0 <= d < q
    d = w;
  }
#pragma unroll
  for (int w = 0; w < L; ++w) {
    const int bit = 32 * w, j = bit / 30, sh = bit % 30;
    uint32_t x = (uint32_t)d.v[j] >> sh;
    if (j + 1 < N) x |= (uint32_t)d.v[j + 1] << (30 - sh);
    if (60 - sh < 32 && j + 2 < N) x |= (uint32_t)d.v[j + 2] << (60 - sh);
    r[w] = x;
  }
}

// Affine point of p in STANDARD form (x, y); O gives (0, 0).
template <class T>
__device__ __forceinline__ void xyzz_to_affine_std(uint32_t x[T::L], uint32_t y[T::L], const Xyzz<T> &p,
                                                   const uint32_t r2[T::L]) {
  constexpr int L = T::L;
  if (xyzz_is_inf(p)) {
    fv_zero<L>(x);
    fv_zero<L>(y);
    return;
  }
  uint32_t t[L], inv[L], zi[L];
  T::mul(t, p.ZZ, p.ZZZ);
  f_inverse<T>(inv, t, r2);  // (ZZ ZZZ)^-1
  T::mul(zi, inv, p.ZZZ);     // ZZ^-1
  T::mul(t, p.X, zi);
  T::redc(x, t);
  T::mul(zi, inv, p.ZZ);      // ZZZ^-1
  T::mul(t, p.Y, zi);
  T::redc(y, t);
}

// -------------------------------------------------- four lanes per point
// For the serial tails of the MSM (window merge, upper tree levels, long
// pieces), where too few points are left to fill the GPU and the time is the
// depth of dependent products: lane 0 of an aligned group of four holds X, lane
// 1 Y, lane 2 ZZ, lane 3 ZZZ, and each step is one product per lane, all four
// at once.  A doubling is 3 products deep instead of 9, an addition 4 instead
// of 14.  Whole warps call these together (width-4 shuffles of the full warp).

template <int L>
__device__ __forceinline__ void quad_get(uint32_t r[L], const uint32_t v[L], int src) {
#pragma unroll
  for (int j = 0; j < L; ++j) r[j] = __shfl_sync(0xffffffffu, v[j], src, 4);
}

template <int L>
__device__ __forceinline__ void quad_pick(uint32_t r[L], bool first, const uint32_t a[L], const uint32_t b[L]) {
#pragma unroll
  for (int j = 0; j < L; ++j) r[j] = first ? a[j] : b[j];
}

// v = 2 v (dbl-2008-s-1, a = 0); O stays O.  On the chain between two products
// sums are left unreduced where the product allows it: factors a p and b p give
// a result below 2p while a b < 2^(32 L) / p, which is 9.8 for the 381-bit and
// 5.2 for the 254-bit field (U < 2p, M < 3p or 2p, S - X3 < 3p or 2p).
template <class T, bool kCall = true>
__device__ __forceinline__ void quad_dbl(uint32_t v[T::L]) {
  constexpr int L = T::L;
  constexpr bool kWide = T::modulus(L - 1) < 0x1c71c71cu;   // 9 p < 2^(32 L)
  static_assert(T::modulus(L - 1) < 0x3fffffffu, "4 p < 2^(32 L)");
  const int lane = threadIdx.x & 3;
  uint32_t a[L], b[L], p[L], V[L], M[L], q[L], g[L], h[L];
  words_add<L>(a, v, v);
  quad_pick<L>(a, lane == 1, a, v);       // lane 1: U = 2 Y; lane 0: X
  f_sqr<T, kCall>(p, a);                  // lane 0: X^2, lane 1: V = U^2
  quad_get<L>(V, p, 1);
  quad_get<L>(g, p, 0);
  if constexpr (kWide) words_add<L>(M, g, g);
  else T::add(M, g, g);
  words_add<L>(M, M, g);                  // M = 3 X^2
  quad_pick<L>(a, lane == 3, M, a);
  quad_pick<L>(a, lane == 2, v, a);
  quad_pick<L>(b, lane == 3, M, V);
  f_mul<T, kCall>(q, a, b);                // S = X V, W = U V, ZZ3 = ZZ V, M^2
  quad_get<L>(g, q, lane == 0 ? 3 : 1);   // lane 0: M^2, lane 3: W
  uint32_t x3[L];
  T::sub(x3, g, q);
  T::sub(x3, x3, q);                      // lane 0: X3 = M^2 - 2 S
  T::add(b, q, q);
  if constexpr (kWide) words_add<L>(b, b, q);
  else T::add(b, b, q);
#pragma unroll
  for (int j = 0; j < L; ++j) a[j] = T::modulus(j);
  words_sub<L>(a, a, g);
  words_add<L>(b, b, a);                  // lane 0: S - X3 = 3 S - M^2
  quad_pick<L>(a, lane == 0, M, q);
  quad_pick<L>(a, lane == 3, g, a);
  quad_pick<L>(b, lane == 0, b, v);
  f_mul<T, kCall>(h, a, b);                // lane 0: M (S - X3), lane 1: W Y, lane 3: W ZZZ
  quad_get<L>(g, h, 0);
  T::sub(g, g, h);                        // lane 1: Y3
  quad_pick<L>(v, lane == 0, x3, q);
  quad_pick<L>(v, lane == 1, g, v);
  quad_pick<L>(v, lane == 3, h, v);
}

// Whether every point of the warp is O.
template <class T>
__device__ __forceinline__ bool quad_all_inf(const uint32_t v[T::L]) {
  return __all_sync(0xffffffffu, (threadIdx.x & 3) != 2 || fv_is_zero<T::L>(v));
}

// v += w (add-2008-s, with the cases it excludes).  With kSkip a warp in which every
// addition has an operand O skips the products: for buckets and windows, most of
// which zero, small and sparse scalars leave empty, but not for pieces, which have
// a point each (2% of a tree's time for the vote).
template <class T, bool kSkip = false>
__device__ __forceinline__ void quad_add(uint32_t v[T::L], const uint32_t w[T::L]) {
  constexpr int L = T::L;
  const int lane = threadIdx.x & 3;
  const bool v_inf = __shfl_sync(0xffffffffu, (int)fv_is_zero<L>(v), 2, 4);
  const bool w_inf = __shfl_sync(0xffffffffu, (int)fv_is_zero<L>(w), 2, 4);
  if constexpr (kSkip) {
    if (__all_sync(0xffffffffu, v_inf || w_inf)) {
      quad_pick<L>(v, w_inf, v, w);
      return;
    }
  }
  uint32_t g[L], p[L], d[L], a[L], b[L], q[L], r[L], h[L];
  quad_get<L>(g, w, lane ^ 2);
  f_mul<T, true>(p, v, g);                // U1 = X1 ZZ2, S1 = Y1 ZZZ2, U2 = ZZ1 X2, S2 = ZZZ1 Y2
  quad_get<L>(g, p, lane ^ 2);
  quad_pick<L>(a, lane < 2, g, p);
  quad_pick<L>(b, lane < 2, p, g);
  T::sub(d, a, b);                        // lanes 0, 2: P = U2 - U1; lanes 1, 3: R = S2 - S1
  const bool same_x = __shfl_sync(0xffffffffu, (int)fv_is_zero<L>(d), 0, 4);
  const bool same_y = __shfl_sync(0xffffffffu, (int)fv_is_zero<L>(d), 1, 4);
  quad_pick<L>(a, lane < 2, d, v);
  quad_pick<L>(b, lane < 2, d, w);
  f_mul<T, true>(q, a, b);                // PP, R^2, ZZ1 ZZ2, ZZZ1 ZZZ2
  quad_get<L>(b, q, 0);                   // PP
  quad_get<L>(a, d, 0);                   // P
  quad_pick<L>(a, lane == 0, p, a);
  quad_pick<L>(a, lane == 2, q, a);
  f_mul<T, true>(r, a, b);                // Q = U1 PP, PPP, ZZ3, PPP
  quad_get<L>(g, r, 0);                   // Q
  uint32_t x3[L];
  T::sub(x3, q, r);
  T::sub(x3, x3, g);
  T::sub(x3, x3, g);                      // lane 1: X3 = R^2 - PPP - 2 Q
  T::sub(b, g, x3);                       // lane 1: Q - X3
  quad_get<L>(a, p, 1);                   // S1
  quad_get<L>(g, r, 1);                   // PPP
  quad_pick<L>(a, lane == 1, d, a);
  quad_pick<L>(a, lane == 3, q, a);
  quad_pick<L>(b, lane == 1, b, g);
  f_mul<T, true>(h, a, b);                // S1 PPP, R (Q - X3), -, ZZZ3
  quad_pick<L>(a, lane == 0, h, x3);
  quad_get<L>(g, a, lane ^ 1);            // lane 0: X3, lane 1: S1 PPP
  T::sub(b, h, g);                        // lane 1: Y3
  quad_pick<L>(a, lane == 0, g, r);       // lane 2: ZZ3
  quad_pick<L>(a, lane == 1, b, a);
  quad_pick<L>(a, lane == 3, h, a);
  const bool twice = same_x && same_y && !v_inf && !w_inf;
  if (__any_sync(0xffffffffu, twice)) {
    fv_copy<L>(b, v);
    quad_dbl<T>(b);
    quad_pick<L>(a, twice, b, a);
  }
  const bool opposite = same_x && !same_y && !v_inf && !w_inf;
#pragma unroll
  for (int j = 0; j < L; ++j) v[j] = w_inf ? v[j] : v_inf ? w[j] : opposite ? 0u : a[j];
}

// Coordinate `lane` of point i.
template <class T>
__device__ __forceinline__ void quad_load(uint32_t v[T::L], const uint4 *base, uint64_t i) {
  T::load(v, base, 4 * i + (threadIdx.x & 3));
}

template <class T>
__device__ __forceinline__ void quad_store(uint4 *base, uint64_t i, const uint32_t v[T::L]) {
  T::store(base, 4 * i + (threadIdx.x & 3), v);
}

}  // namespace gb300ntt
