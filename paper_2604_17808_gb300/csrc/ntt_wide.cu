// ntt_wide.cu -- host side of the 377- and 753-bit transforms (ntt_wide.cuh):
// field constants, per-(device, field, size) tables, pass launches, C ABI.
//
// The moduli (the smallest primes c 2^32 + 1, c odd, above floor(pi
// 2^(b-2)) for b = 377 and 753; generators 7 and 11, the smallest quadratic
// non-residues) are public constants of this library (fp_wide.cuh).  The host
// derives R mod p and R^2 mod p from them with a small fixed-width arithmetic;
// every root of unity, inverse and table is computed on the device
// (wide_constants_kernel, wide_table_kernel).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <map>
#include <new>
#include <mutex>
#include <tuple>
#include <vector>

#include "../../include/ntt_gb300.h"
#include "ntt_plan.h"
#include "ntt_wide.cuh"

namespace gb300ntt {
namespace {

#define NTT_TRY_W(expr)                \
  do {                                 \
    const ntt_status _s = (expr);      \
    if (_s != NTT_OK) return _s;       \
  } while (0)

// x = 2 x mod p on NL-limb numbers (x < p).
template <int NL>
void host_double_mod(uint32_t x[NL], const uint32_t p[NL]) {
  uint32_t carry = 0;
  for (int j = 0; j < NL; ++j) {
    const uint32_t nc = x[j] >> 31;
    x[j] = (x[j] << 1) | carry;
    carry = nc;
  }
  bool ge = carry != 0;
  if (!ge) {
    ge = true;
    for (int j = NL - 1; j >= 0; --j)
      if (x[j] != p[j]) {
        ge = x[j] > p[j];
        break;
      }
  }
  if (ge) {
    int64_t br = 0;
    for (int j = 0; j < NL; ++j) {
      const int64_t v = (int64_t)x[j] - p[j] + br;
      x[j] = (uint32_t)v;
      br = v >> 32;
    }
  }
}

template <class F>
WideConst<F> make_const() {
  constexpr int L = F::L;
  WideConst<F> c{};
  uint32_t p[L], x[L] = {1};
  for (int j = 0; j < L; ++j) p[j] = F::p(j);
  for (int b = 0; b < 32 * L; ++b) host_double_mod<L>(x, p);   // R mod p, R = 2^(32 L)
  std::memcpy(c.one, x, sizeof c.one);
  for (int b = 0; b < 32 * L; ++b) host_double_mod<L>(x, p);   // R^2 mod p
  std::memcpy(c.r2, x, sizeof c.r2);
  return c;
}

template <class F>
const WideConst<F> &wide_const() {
  static const WideConst<F> c = make_const<F>();
  return c;
}

int limbs_of(int field) { return field == NTT_FIELD_W377 ? 12 : 24; }

struct WidePlan {
  uint32_t log_n = 0, num_passes = 0;
  uint32_t pass_log[kMaxPasses] = {};
  uint4 *dft_tw[2][12] = {};
  uint4 *tw[2][kMaxPasses] = {};
  bool in_place_one = false;     // in-place calls run as one pass, without the scratch
  uint4 *pre_inv = nullptr;      // N^-1: first-pass input factors of an inverse of one pass
  uint4 *scratch = nullptr;
  uint4 *coset_pre = nullptr;    // s^i, i < N: first-pass input factors of the coset forward kind
  uint4 *coset_post = nullptr;   // s^-i, i < N: last-pass output factors of the coset inverse kind
  uint32_t coset_shift[24] = {}; // the s of those tables (32-bit words, standard form)
  bool coset_ready = false;      // the two tables hold the powers of coset_shift
  uint32_t *kbuf = nullptr;      // constants scratch of the table builders
  std::vector<void *> allocs;
};

std::mutex g_wide_mu;
bool g_wide_ready[8] = {};
int g_wide_sms[8] = {};   // multiprocessors of each device
std::map<std::tuple<int, int, uint32_t>, WidePlan *> g_wide_plans;   // (device, field, log_n)

ntt_status cuda_w(cudaError_t e) { return cuda_status(e); }

// A table of the transform size 2^log_n from the constants in kbuf, which hold
// omega_N^(2^b): the powers of omega_M, M = 2^log_m, are those from b = log_n -
// log_m on.
template <class F>
ntt_status gen_table(uint4 *out, uint32_t log_n, uint32_t log_m, int dir, bool use_n_inv, uint32_t log_mp,
                     uint64_t count, int two_d, bool constant, bool split, const uint32_t *kbuf, cudaStream_t st) {
  constexpr int L = F::L;
  const uint32_t *ladder = constant ? nullptr : kbuf + ((dir ? 32 : 0) + log_n - log_m) * L;
  const uint32_t *init = kbuf + (use_n_inv ? 64 : 65) * L;
  uint64_t blocks = (count + 255) / 256;
  if (blocks > 152ull * 32) blocks = 152ull * 32;
  wide_table_kernel<F><<<(unsigned)(blocks ? blocks : 1), 256, 0, st>>>(out, log_mp, ladder, init, count, two_d,
                                                                         split ? 1 : 0);
  return cuda_w(cudaGetLastError());
}

ntt_status alloc_w(WidePlan *w, uint4 **out, uint64_t bytes) {
  void *p = nullptr;
  const cudaError_t e = cudaMalloc(&p, bytes);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return cuda_w(e);
  }
  w->allocs.push_back(p);
  *out = (uint4 *)p;
  return NTT_OK;
}

// Passes of a transform: up to 2^8 points one (2 or 4 elements per thread hold
// them in one CTA), else as few as the largest tile allows, at least two (one
// CTA with a 2^10-point sub-transform is slower than two passes over several).
uint32_t wide_passes(uint32_t log_n, uint32_t tile_log) {
  if (log_n <= 8) return 1;
  return std::max<uint32_t>(2, (log_n + tile_log - 1) / tile_log);
}

template <class F>
ntt_status build_wide(uint32_t log_n, WidePlan *w) {
  constexpr int L = F::L;
  const uint32_t P = wide_passes(log_n, (uint32_t)WideShape<F>::kLog);
  if (P > (uint32_t)kMaxPasses) return NTT_ERR_UNSUPPORTED;
  w->log_n = log_n;
  w->num_passes = P;
  // A vector that fits one tile needs no scratch in place, so that such calls on
  // several streams do not meet in it: one pass (us, in place, one pass against two
  // through the scratch: 377 bits 2^9 19.7 against 13.3 and 2^10 37.1 against
  // 14.4, 753 bits 2^9 57.2 against 35.0).
  w->in_place_one = P > 1 && log_n <= (uint32_t)WideShape<F>::kLog;
  for (uint32_t j = 0; j < P; ++j) w->pass_log[j] = log_n / P + (j < log_n % P ? 1 : 0);
  const uint64_t eb = 4ull * L;   // table entry
  uint32_t *kbuf = nullptr;
  if (cudaMalloc(&kbuf, 66 * 4 * L) != cudaSuccess) return NTT_ERR_OOM;
  w->allocs.push_back(kbuf);
  w->kbuf = kbuf;
  cudaStream_t st = nullptr;
  // once for the size: one thread, 0.3 ms (377 bits) or 4.2 ms (753)
  wide_constants_kernel<F><<<1, 1, 0, st>>>(kbuf, log_n, wide_const<F>());
  NTT_TRY_W(cuda_w(cudaGetLastError()));
  for (uint32_t j = 0; j < P + (w->in_place_one ? 1 : 0); ++j) {
    const uint32_t logs = j < P ? w->pass_log[j] : log_n;
    for (int dir = 0; dir < 2; ++dir) {
      if (w->dft_tw[dir][logs]) continue;
      const uint64_t cnt = logs ? (1ull << (logs - 1)) : 1;
      NTT_TRY_W(alloc_w(w, &w->dft_tw[dir][logs], cnt * 2 * eb));
      NTT_TRY_W(gen_table<F>(w->dft_tw[dir][logs], log_n, logs, dir, false, 0, cnt, 0, false, true, kbuf, st));
    }
  }
  uint32_t log_m = w->pass_log[0];
  for (uint32_t j = 1; j < P; ++j) {
    const uint32_t logs = w->pass_log[j], log_mp = log_m;
    log_m += logs;
    for (int dir = 0; dir < 2; ++dir) {
      NTT_TRY_W(alloc_w(w, &w->tw[dir][j], (1ull << log_m) * eb));
      NTT_TRY_W(gen_table<F>(w->tw[dir][j], log_n, log_m, dir, dir == 1 && j == P - 1, log_mp, 1ull << log_m, 1, false,
                             false, kbuf, st));
    }
  }
  if (P == 1 || w->in_place_one) {   // single-pass inverse: N^-1 as the pass-0 multiplier
    NTT_TRY_W(alloc_w(w, &w->pre_inv, (1ull << log_n) * eb));
    NTT_TRY_W(gen_table<F>(w->pre_inv, log_n, log_n, 0, true, 0, 1ull << log_n, 0, true, false, kbuf, st));
  }
  if (P > 1 && !w->in_place_one) NTT_TRY_W(alloc_w(w, &w->scratch, (1ull << log_n) * eb));
  return cuda_w(cudaDeviceSynchronize());
}

// The coset tables of shift s (L words, 0 < s < p), s^i and s^-i for
// i < N: allocated on the first coset call for this (device, field, size),
// rewritten in place when a call brings another shift (after the device is
// idle: transforms enqueued earlier may still read the old tables).
template <class F>
ntt_status build_wide_coset(WidePlan *w, const uint32_t *shift) {
  constexpr int L = F::L;
  const uint64_t n = 1ull << w->log_n, eb = 4ull * L;
  if (!w->coset_post) {
    const size_t kept = w->allocs.size();
    uint4 *pre = nullptr, *post = nullptr;
    ntt_status s = alloc_w(w, &pre, n * eb);
    if (s == NTT_OK) s = alloc_w(w, &post, n * eb);
    if (s != NTT_OK) {   // forward and inverse stay usable
      for (size_t i = kept; i < w->allocs.size(); ++i) cudaFree(w->allocs[i]);
      w->allocs.resize(kept);
      return s;
    }
    w->coset_pre = pre;
    w->coset_post = post;
  } else {
    NTT_TRY_W(cuda_w(cudaDeviceSynchronize()));
  }
  w->coset_ready = false;   // until the tables below are written
  uint4 *pre = w->coset_pre, *post = w->coset_post;
  cudaStream_t st = nullptr;
  NTT_TRY_W(cuda_w(cudaMemcpy(w->kbuf + 64 * L, shift, 4 * L, cudaMemcpyHostToDevice)));
  wide_coset_constants_kernel<F><<<1, 1, 0, st>>>(w->kbuf, wide_const<F>());
  uint64_t blocks = (n + 255) / 256;
  if (blocks > 152ull * 32) blocks = 152ull * 32;
  wide_table_kernel<F><<<(unsigned)blocks, 256, 0, st>>>(pre, 0, w->kbuf, w->kbuf + 65 * L, n, 0, 0);
  wide_table_kernel<F><<<(unsigned)blocks, 256, 0, st>>>(post, 0, w->kbuf + 32 * L, w->kbuf + 65 * L, n, 0, 0);
  NTT_TRY_W(cuda_w(cudaGetLastError()));
  NTT_TRY_W(cuda_w(cudaDeviceSynchronize()));
  std::memcpy(w->coset_shift, shift, 4 * L);
  w->coset_ready = true;
  return NTT_OK;
}

// Tile of a pass launch, by the rule of the 256-bit passes (pass_shape in
// ntt_plan.cu): as few elements per thread as still fit the GPU at once.
template <class F>
TileShape wide_shape(uint32_t log_n, uint32_t logs, int sms) {
  using W = WideShape<F>;
  const uint64_t slots = (uint64_t)sms * W::kThreads * W::kMinBlocks;
  for (uint32_t pl = 1; pl < 3; ++pl) {
    const uint32_t t = std::max(logs, pl + 5);
    if ((1u << (t - pl)) <= (uint32_t)W::kThreads && (1ull << log_n) >> pl <= slots) return TileShape{logs, t, pl};
  }
  return TileShape{logs, (uint32_t)W::kLog, 3};
}

template <class F, int MODE>
cudaError_t wide_launch(const PassArgs &a, const TileShape &s, cudaStream_t st) {
  const uint64_t g = 1ull << (s.tl - s.logs), tiles = (a.num_sub + g - 1) / g;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)tiles);
  cfg.blockDim = dim3(1u << (s.tl - s.pl));
  cfg.dynamicSmemBytes = (size_t)(4 * F::L) << s.tl;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];   // see pdl_wait
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, wide_pass_kernel<F, MODE>, a, s);
}

template <class F>
cudaError_t wide_pass(int mode, const PassArgs &a, uint32_t log_n, uint32_t logs, int sms, cudaStream_t st) {
  const TileShape s = wide_shape<F>(log_n, logs, sms);
  switch (mode) {
    case kModeInner: return wide_launch<F, kModeInner>(a, s, st);
    case kModeFirst: return wide_launch<F, kModeFirst>(a, s, st);
    default: return wide_launch<F, kModeFirstPre>(a, s, st);
  }
}

template <class F>
cudaError_t wide_set_attrs() {
  constexpr int smem = WideShape<F>::kBytes;
  cudaError_t e = cudaFuncSetAttribute(wide_pass_kernel<F, kModeInner>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(wide_pass_kernel<F, kModeFirst>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(wide_pass_kernel<F, kModeFirstPre>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  return e;
}

// The (device, field, size) tables, built on first use; with a shift
// (L words), also the coset tables of that shift.  The caller holds
// g_wide_mu until its transform is enqueued, so no other call can rewrite
// the coset tables in between.
ntt_status wide_plan(int field, uint32_t log_n, const uint32_t *shift, WidePlan **out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return NTT_ERR_NO_DEVICE;
  if (dev < 0 || dev >= 8) return NTT_ERR_UNSUPPORTED;
  if (!g_wide_ready[dev]) {
    NTT_TRY_W(cuda_w(wide_set_attrs<FieldW377>()));
    NTT_TRY_W(cuda_w(wide_set_attrs<FieldW753>()));
    NTT_TRY_W(cuda_w(cudaDeviceGetAttribute(&g_wide_sms[dev], cudaDevAttrMultiProcessorCount, dev)));
    g_wide_ready[dev] = true;
  }
  auto key = std::make_tuple(dev, field, log_n);
  auto it = g_wide_plans.find(key);
  WidePlan *w = nullptr;
  if (it != g_wide_plans.end()) {
    w = it->second;
  } else {
    w = new (std::nothrow) WidePlan();
    if (!w) return NTT_ERR_OOM;
    const ntt_status s = limbs_of(field) == 12 ? build_wide<FieldW377>(log_n, w) : build_wide<FieldW753>(log_n, w);
    if (s != NTT_OK) {
      for (void *p : w->allocs) cudaFree(p);
      delete w;
      return s;
    }
    g_wide_plans[key] = w;
  }
  if (shift && (!w->coset_ready || std::memcmp(w->coset_shift, shift, 4 * limbs_of(field)) != 0)) {
    // a failure leaves forward and inverse usable and the coset tables
    // marked unwritten (the next coset call writes them again)
    NTT_TRY_W(limbs_of(field) == 12 ? build_wide_coset<FieldW377>(w, shift) : build_wide_coset<FieldW753>(w, shift));
  }
  *out = w;
  return NTT_OK;
}

// 0 < s < p for a shift of 12 or 24 little-endian words.
bool shift_in_range(ntt_field field, const uint32_t *sw) {
  const int nl = limbs_of((int)field);
  uint32_t p[24];
  for (int j = 0; j < nl; ++j) p[j] = nl == 12 ? FieldW377::p(j) : FieldW753::p(j);
  bool zero = true;
  for (int j = 0; j < nl; ++j) zero = zero && sw[j] == 0;
  if (zero) return false;
  for (int j = nl - 1; j >= 0; --j)
    if (sw[j] != p[j]) return sw[j] < p[j];
  return false;   // s == p
}

// One transform; `shift` (L words, checked by the caller) is used by the
// coset kinds only.  The table lock is held until every pass is enqueued.
ntt_status wide_transform(ntt_field field, ntt_kind kind, uint32_t log_n, const uint32_t *shift, const void *d_in,
                          void *d_out, ntt_stream stream) {
  std::lock_guard<std::mutex> lk(g_wide_mu);
  WidePlan *w = nullptr;
  const bool coset = kind == NTT_KIND_COSET || kind == NTT_KIND_COSET_INVERSE;
  const ntt_status s = wide_plan((int)field, log_n, coset ? shift : nullptr, &w);
  if (s != NTT_OK) return s;
  const int NL = limbs_of((int)field);
  int dev = 0;
  NTT_TRY_W(cuda_w(cudaGetDevice(&dev)));   // below 8 (wide_plan)
  const int dir = (kind == NTT_KIND_INVERSE || kind == NTT_KIND_COSET_INVERSE) ? 1 : 0;
  const bool one = d_in == d_out && w->in_place_one;
  const uint32_t P = one ? 1 : w->num_passes;
  uint4 *work = (P > 1 && d_in == d_out) ? w->scratch : (uint4 *)d_out;
  for (uint32_t j = 0; j < P; ++j) {
    const uint32_t logs = one ? log_n : w->pass_log[j];
    PassArgs a{};
    a.dft_tw = w->dft_tw[dir][logs];
    a.num_sub = 1ull << (log_n - logs);
    int mode;
    if (j == 0) {
      a.src = (const uint4 *)d_in;
      a.dst = P == 1 ? (uint4 *)d_out : work;
      a.log_mp = log_n - logs;
      a.num_digits = P - 1;
      uint32_t dshift = 0;
      for (uint32_t d = 1; d < P; ++d) {
        a.digit_log[d - 1] = (uint8_t)w->pass_log[d];
        a.digit_shift[d - 1] = (uint8_t)dshift;
        dshift += w->pass_log[d];
      }
      a.mul = kind == NTT_KIND_COSET ? w->coset_pre : (P == 1 && dir == 1) ? w->pre_inv : nullptr;
      mode = a.mul ? kModeFirstPre : kModeFirst;
    } else {
      uint32_t log_mp = 0;
      for (uint32_t i = 0; i < j; ++i) log_mp += w->pass_log[i];
      a.src = work;
      a.dst = j == P - 1 ? (uint4 *)d_out : work;
      a.log_mp = log_mp;
      a.mul = w->tw[dir][j];
      mode = kModeInner;
    }
    if (j == P - 1 && kind == NTT_KIND_COSET_INVERSE) a.post = w->coset_post;
    a.n_vec = 1ull << log_n;
    a.n_mul = a.mul ? (j == 0 ? 1ull << log_n : 1ull << (a.log_mp + logs)) : 0;
    const cudaError_t e = NL == 12 ? wide_pass<FieldW377>(mode, a, log_n, logs, g_wide_sms[dev], (cudaStream_t)stream)
                                   : wide_pass<FieldW753>(mode, a, log_n, logs, g_wide_sms[dev], (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_status(e);
  }
  return NTT_OK;
}

}  // namespace
}  // namespace gb300ntt

using namespace gb300ntt;

extern "C" {

ntt_status ntt_field_element_bytes(ntt_field field, uint32_t *bytes) {
  if (!bytes) return NTT_ERR_INVALID_ARG;
  switch (field) {
    case NTT_FIELD_BLS12_381_FR:
    case NTT_FIELD_BN254_FR: *bytes = 32; return NTT_OK;
    case NTT_FIELD_W377: *bytes = 48; return NTT_OK;
    case NTT_FIELD_W753: *bytes = 96; return NTT_OK;
    default: return NTT_ERR_INVALID_ARG;
  }
}

ntt_status ntt_wide_transform(ntt_field field, ntt_kind kind, uint32_t log_n, const void *d_in, void *d_out,
                              ntt_stream stream) {
  if (field != NTT_FIELD_W377 && field != NTT_FIELD_W753) return NTT_ERR_INVALID_ARG;
  if (kind != NTT_KIND_FORWARD && kind != NTT_KIND_INVERSE && kind != NTT_KIND_COSET && kind != NTT_KIND_COSET_INVERSE)
    return NTT_ERR_INVALID_ARG;
  if (log_n < 1 || log_n > 24) return NTT_ERR_UNSUPPORTED;
  if (!d_in || !d_out || ((uintptr_t)d_in | (uintptr_t)d_out) % 16) return NTT_ERR_INVALID_ARG;
  uint32_t gen[24] = {field == NTT_FIELD_W377 ? 7u : 11u};   // the default shift: the generator
  return wide_transform(field, kind, log_n, gen, d_in, d_out, stream);
}

ntt_status ntt_wide_transform_shift(ntt_field field, ntt_kind kind, uint32_t log_n, const uint32_t *h_shift,
                                    const void *d_in, void *d_out, ntt_stream stream) {
  if (field != NTT_FIELD_W377 && field != NTT_FIELD_W753) return NTT_ERR_INVALID_ARG;
  if (kind != NTT_KIND_COSET && kind != NTT_KIND_COSET_INVERSE) return NTT_ERR_INVALID_ARG;
  if (log_n < 1 || log_n > 24) return NTT_ERR_UNSUPPORTED;
  if (!d_in || !d_out || ((uintptr_t)d_in | (uintptr_t)d_out) % 16) return NTT_ERR_INVALID_ARG;
  if (!h_shift || !shift_in_range(field, h_shift)) return NTT_ERR_INVALID_ARG;
  return wide_transform(field, kind, log_n, h_shift, d_in, d_out, stream);
}

}  // extern "C"
