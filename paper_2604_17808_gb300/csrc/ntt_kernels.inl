// ntt_kernels.inl -- kernel instantiations and launchers for one field.
//
// Included by the kernels_<field>*.cu files with NTT_FIELD (the field type),
// NTT_NS (a namespace for the field's launchers) and one NTT_PART_* macro,
// so that the kernel families of a field compile in parallel, one nvcc
// process each:
//   NTT_PART_PASS             the pass kernels;
//   NTT_PART_BATCH            the persistent batched kernel;
//   NTT_PART_MATRIX           the matrix-form (tensor-core) pass;
//   NTT_PART_MISC             table generators, element-wise kernels and
//                             the launcher table.
#include "../../include/ntt_gb300.h"
#include "ntt_launch.h"

#include <algorithm>

namespace gb300ntt {
namespace NTT_NS {

// launchers defined by the other parts of this field
cudaError_t prepare_pass();
cudaError_t pass(int mode, const TileShape &s, const PassArgs &a, uint64_t tiles, int sms, cudaStream_t st);
cudaError_t prepare_batch();
cudaError_t batch(const BatchLaunch &b, cudaStream_t st);
cudaError_t prepare_matrix();
cudaError_t matrix_pass(int logs, int mode, const MatrixPassArgs &ma, const CUtensorMap &in_map, uint32_t grid,
                        cudaStream_t st);

namespace {

using F = NTT_FIELD;

__device__ __forceinline__ void fe_from_param(uint32_t r[8], const Fe32 &a) {
#pragma unroll
  for (int j = 0; j < 8; ++j) r[j] = a.w[j];
}

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Launch with programmatic stream serialisation (see pdl_wait):
// consecutive passes overlap their launch latency and CTA scheduling.
template <class K, class... A>
cudaError_t launch_pdl(K kernel, dim3 grid, dim3 block, int smem, cudaStream_t st, const A &...a) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, a...);
}

__device__ __forceinline__ uint32_t ld_acquire_gpu(const uint32_t *p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

}  // namespace

#if defined(NTT_PART_PASS)

namespace {

template <int MODE>
cudaError_t set_pass_attr() {
  cudaError_t e = cudaFuncSetAttribute(ntt_pass_kernel<F, MODE, 128>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kGroupBytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(ntt_pass_kernel<F, MODE, 256>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             2 * kGroupBytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(ntt_pass_kernel<F, MODE, 896>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kGroups * kGroupBytes);
  return e;
}

template <int MODE>
cudaError_t pass_mode(const TileShape &s, const PassArgs &a, uint64_t tiles, int sms, cudaStream_t st) {
  const uint32_t threads = 1u << (s.tl - s.pl);
  const int smem = 32 << s.tl;
  const uint32_t n = (uint32_t)tiles;
  // seven tiles per CTA where that makes the pass one wave that six do not
  constexpr uint64_t kResident = TileBounds<128>::kMinBlocks;
  if (s.tl == 10 && s.pl == 3 && tiles > kResident * sms && tiles <= (uint64_t)kGroups * sms)
    return launch_pdl(ntt_pass_kernel<F, MODE, 896>, (n + kGroups - 1) / kGroups, kGroups * kGroupThreads,
                      kGroups * kGroupBytes, st, a, s, n);
  if (threads <= 128) return launch_pdl(ntt_pass_kernel<F, MODE, 128>, n, threads, smem, st, a, s, n);
  return launch_pdl(ntt_pass_kernel<F, MODE, 256>, n, threads, smem, st, a, s, n);
}

}  // namespace

cudaError_t prepare_pass() {
  cudaError_t e = set_pass_attr<kModeInner>();
  if (e == cudaSuccess) e = set_pass_attr<kModeFirst>();
  if (e == cudaSuccess) e = set_pass_attr<kModeFirstPre>();
  return e;
}

cudaError_t pass(int mode, const TileShape &s, const PassArgs &a, uint64_t tiles, int sms, cudaStream_t st) {
  if (s.pl < 1 || s.pl > 3 || s.tl > 11 || s.logs < 1 || s.logs > s.tl || s.tl - s.pl > 8)
    return cudaErrorInvalidValue;
  switch (mode) {
    case kModeInner: return pass_mode<kModeInner>(s, a, tiles, sms, st);
    case kModeFirst: return pass_mode<kModeFirst>(s, a, tiles, sms, st);
    case kModeFirstPre: return pass_mode<kModeFirstPre>(s, a, tiles, sms, st);
    default: return cudaErrorInvalidValue;
  }
}

#elif defined(NTT_PART_BATCH)

namespace {

// One tile of one segment (a non-inlined function per mode and instance).
template <int MODE, int MAXT>
__device__ __noinline__ void batch_tile_fn(const BatchSeg &sg, uint64_t tile, uint32_t smem) {
  pass_tile<Elem256<F>, MODE, false>(sg.a, TileShape{sg.logs, sg.tl, sg.pl}, tile, smem, threadIdx.x, 0);
}

template <int MAXT>
__device__ __forceinline__ void batch_tile(const BatchSeg &sg, uint64_t tile, uint32_t smem) {
  switch (sg.mode) {
    case kModeInner: batch_tile_fn<kModeInner, MAXT>(sg, tile, smem); break;
    case kModeFirst: batch_tile_fn<kModeFirst, MAXT>(sg, tile, smem); break;
    default: batch_tile_fn<kModeFirstPre, MAXT>(sg, tile, smem); break;
  }
}

// CTAs claim items (one tile of one pass of one job) in increasing order.
// An item of pass j waits until every tile of pass j-1 of its job is done;
// those tiles have smaller item indices, so they are held by CTAs that have
// already started and never wait on later items: no deadlock.  Every wait
// is bounded by b.wait_ns (globaltimer); on timeout the CTA records
// NTT_ERR_TIMEOUT in *b.err and returns, and every CTA stops claiming
// items once *b.err is set.
//
// Two instances, as for the pass kernels: 128 threads and tiles of up to 1024
// elements, 6 CTAs per SM, and 256 threads and 2048 elements, 3 CTAs per SM, for
// lists with a 2^11-point pass.
template <int MAXT>
__global__ void __launch_bounds__(MAXT, TileBounds<MAXT>::kMinBlocks) batch_kernel(const BatchLaunch b) {
  extern __shared__ uint4 smem[];
  __shared__ uint32_t s_item;
  __shared__ int32_t s_seg;
  const uint32_t t = threadIdx.x;
  const uint32_t tile_smem = (uint32_t)__cvta_generic_to_shared(smem);
  for (;;) {
    if (t == 0) {
      uint32_t item = atomicAdd(b.head, 1u);
      if (*(volatile uint32_t *)b.err != 0) item = b.total_items;
      int32_t seg = -1;
      if (item < b.total_items) {
        int lo = 0, hi = (int)b.num_segs - 1;
        while (lo < hi) {
          const int mid = (lo + hi + 1) >> 1;
          if (b.segs[mid].first_item <= item) lo = mid;
          else hi = mid - 1;
        }
        seg = lo;
        const int32_t dep = b.segs[lo].dep_seg;
        if (dep >= 0) {
          const uint32_t need = b.segs[lo].dep_tiles;
          const uint64_t t0 = global_ns();
          while (ld_acquire_gpu(b.done + dep) < need) {
            if (global_ns() - t0 > b.wait_ns) {
              atomicCAS(b.err, 0u, (uint32_t)NTT_ERR_TIMEOUT);
              item = b.total_items;   // stop
              break;
            }
            __nanosleep(128);
          }
        }
      }
      s_item = item;
      s_seg = seg;
    }
    __syncthreads();
    const uint32_t item = s_item;
    if (item >= b.total_items) return;
    const int32_t seg = s_seg;
    const BatchSeg &sg = b.segs[seg];
    batch_tile<MAXT>(sg, item - sg.first_item, tile_smem);
    __syncthreads();
    if (t == 0) {
      __threadfence();
      atomicAdd(b.done + seg, 1u);
    }
  }
}

}  // namespace

cudaError_t batch(const BatchLaunch &b, cudaStream_t st) {
  if (b.tile_log <= 10)
    batch_kernel<128><<<b.sm_count * TileBounds<128>::kMinBlocks, 128, kGroupBytes, st>>>(b);
  else
    batch_kernel<256><<<b.sm_count * TileBounds<256>::kMinBlocks, 256, 2 * kGroupBytes, st>>>(b);
  return cudaGetLastError();
}

cudaError_t prepare_batch() {
  cudaError_t e = cudaFuncSetAttribute(batch_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGroupBytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(batch_kernel<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * kGroupBytes);
  return e;
}

#elif defined(NTT_PART_MATRIX)

namespace {

template <int LOGS, int MODE, bool BARRETT>
cudaError_t set_matrix_attr() {
  return cudaFuncSetAttribute(ntt_matrix_pass_kernel<F, LOGS, MODE, BARRETT>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize, matrix_smem_bytes<LOGS>());
}

template <int LOGS>
cudaError_t set_matrix_attrs() {
  cudaError_t e = set_matrix_attr<LOGS, kModeInner, false>();
  if (e == cudaSuccess) e = set_matrix_attr<LOGS, kModeInner, true>();
  if (e == cudaSuccess) e = set_matrix_attr<LOGS, kModeFirst, false>();
  if (e == cudaSuccess) e = set_matrix_attr<LOGS, kModeFirst, true>();
  return e;
}

template <int LOGS, int MODE>
cudaError_t matrix_mode(const MatrixPassArgs &ma, const CUtensorMap &in_map, uint32_t grid, cudaStream_t st) {
  const int smem = matrix_smem_bytes<LOGS>();
  if (ma.barrett)
    return launch_pdl(ntt_matrix_pass_kernel<F, LOGS, MODE, true>, grid, kMatThreads, smem, st, ma, in_map);
  return launch_pdl(ntt_matrix_pass_kernel<F, LOGS, MODE, false>, grid, kMatThreads, smem, st, ma, in_map);
}

template <int LOGS>
cudaError_t matrix_logs(int mode, const MatrixPassArgs &ma, const CUtensorMap &in_map, uint32_t grid,
                        cudaStream_t st) {
  switch (mode) {
    case kModeInner: return matrix_mode<LOGS, kModeInner>(ma, in_map, grid, st);
    case kModeFirst: return matrix_mode<LOGS, kModeFirst>(ma, in_map, grid, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t matrix_pass(int logs, int mode, const MatrixPassArgs &ma, const CUtensorMap &in_map, uint32_t grid,
                        cudaStream_t st) {
  switch (logs) {
    case 1: return matrix_logs<1>(mode, ma, in_map, grid, st);
    case 2: return matrix_logs<2>(mode, ma, in_map, grid, st);
    case 3: return matrix_logs<3>(mode, ma, in_map, grid, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t prepare_matrix() {
  cudaError_t e = set_matrix_attrs<1>();
  if (e == cudaSuccess) e = set_matrix_attrs<2>();
  if (e == cudaSuccess) e = set_matrix_attrs<3>();
  return e;
}

#elif defined(NTT_PART_MISC)

namespace {

// acc *= base^e using the ladder pw (bits of e below 32).
__device__ __forceinline__ void ladder_mul(uint32_t acc[8], uint64_t e, const Pow2Table &pw) {
  for (int b = 0; b < 32 && (e >> b) != 0; ++b) {
    if ((e >> b) & 1) {
      uint32_t w[8];
      fe_from_param(w, pw.v[b]);
      mont_mul<F>(acc, acc, w);
    }
  }
}

__global__ void gen_2d_kernel(uint4 *out, uint32_t log_s, uint32_t log_mp, const Pow2Table pw,
                              const uint4 *fac, const Fe32 init) {
  const uint64_t total = 1ull << (log_s + log_mp);
  for (uint64_t idx = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t n = idx >> log_mp, q = idx & ((1ull << log_mp) - 1);
    uint32_t acc[8];
    fe_from_param(acc, init);
    if (fac) {
      uint32_t f[8];
      fe_load_global(f, fac, n);
      mont_mul<F>(acc, acc, f);
    }
    ladder_mul(acc, n * q, pw);
    fe_store_global(out, idx, acc);
  }
}

__global__ void gen_1d_kernel(uint4 *out, uint64_t count, const Pow2Table pw, const Fe32 init) {
  for (uint64_t idx = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; idx < count;
       idx += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t acc[8];
    fe_from_param(acc, init);
    ladder_mul(acc, idx, pw);
    fe_store_global(out, idx, acc);
  }
}

// Table of the DFT twiddles: entry i holds base^i as the residues of mul_split,
// A = base^i 2^128 and B = base^i 2^256 mod p.
__global__ void gen_split_kernel(uint4 *out, uint64_t count, const Pow2Table pw, const Fe32 one) {
  const uint32_t r128[8] = {0, 0, 0, 0, 1, 0, 0, 0};
  for (uint64_t idx = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; idx < count;
       idx += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t acc[8], low[8];
    fe_from_param(acc, one);
    ladder_mul(acc, idx, pw);
    mont_mul<F>(low, acc, r128);
    fe_store_global(out, 2 * idx, low);
    fe_store_global(out, 2 * idx + 1, acc);
  }
}

__global__ void mul_vec_kernel(uint4 *out, const uint4 *a, const uint4 *b, uint64_t count) {
  for (uint64_t idx = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; idx < count;
       idx += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t x[8], y[8];
    fe_load_global(x, a, idx);
    fe_load_global(y, b, idx);
    mont_mul<F>(x, x, y);
    fe_store_global(out, idx, x);
  }
}

// Pointwise quotient of a prover on coset evaluations:
//   out[i] = (a[i] b[i] - c[i]) z[i mod len]
// in one pass over the vectors (3 reads, 1 write, two products per element):
// a b + (p - c) goes through one Montgomery reduction, which leaves
// (a b - c) 2^-256, and the multiplier z 2^512 turns that back into standard
// form.
__global__ void quotient_kernel(uint4 *out, const uint4 *a, const uint4 *b, const uint4 *c, const QuotientZ z,
                                uint64_t count) {
  const uint64_t zmask = z.len - 1;
  const uint32_t zero[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  for (uint64_t idx = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; idx < count;
       idx += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t x[8], y[8], w[8];
    fe_load_global(w, c, idx);
    sub_mod<F>(w, zero, w);             // -c
    fe_load_global(x, a, idx);
    fe_load_global(y, b, idx);
    mont_mul_add<F>(x, x, y, w);        // (a b - c) 2^-256
    fe_from_param(w, z.z[idx & zmask]);
    mont_mul<F>(x, x, w);               // (a b - c) z
    fe_store_global(out, idx, x);
  }
}

// out[i] = a[i] * (b[i] * 2^-256)^reps: `reps` dependent Montgomery products
// per element, per-thread carry chains (variant 0) or 8 lanes per element
// with shuffle carries (variant 1).
__global__ void mul_rep_kernel(uint4 *out, const uint4 *a, const uint4 *b, uint64_t count, uint32_t reps) {
  for (uint64_t idx = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; idx < count;
       idx += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t x[8], y[8];
    fe_load_global(x, a, idx);
    fe_load_global(y, b, idx);
    for (uint32_t r = 0; r < reps; ++r) mont_mul<F>(x, x, y);
    fe_store_global(out, idx, x);
  }
}

__global__ void mul_rep_coop_kernel(uint32_t *out, const uint32_t *a, const uint32_t *b, uint64_t count,
                                    uint32_t reps) {
  // 8 lanes per element; the grid covers every element exactly (no early exit
  // of part of a warp: the shuffles need all 32 lanes)
  const uint64_t gid = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  const uint32_t j = threadIdx.x & 7u;
  const uint64_t elem = gid >> 3;
  const bool live = elem < count;
  uint32_t x = live ? a[elem * 8 + j] : 0u;
  const uint32_t y = live ? b[elem * 8 + j] : 0u;
  for (uint32_t r = 0; r < reps; ++r) x = mont_mul_coop<F>(x, y, j);
  if (live) out[elem * 8 + j] = x;
}

cudaError_t prepare() {
  cudaError_t e = prepare_pass();
  if (e == cudaSuccess) e = prepare_matrix();
  if (e == cudaSuccess) e = prepare_batch();
  return e;
}

unsigned grid_for(uint64_t count) {
  uint64_t blocks = (count + 255) / 256;
  if (blocks > 152ull * 64) blocks = 152ull * 64;
  return (unsigned)(blocks ? blocks : 1);
}

cudaError_t gen_2d(uint4 *out, uint32_t log_s, uint32_t log_mp, const Pow2Table &pw, const uint4 *fac,
                   Fe32 init, cudaStream_t st) {
  gen_2d_kernel<<<grid_for(1ull << (log_s + log_mp)), 256, 0, st>>>(out, log_s, log_mp, pw, fac, init);
  return cudaGetLastError();
}

cudaError_t gen_1d(uint4 *out, uint64_t count, const Pow2Table &pw, Fe32 init, cudaStream_t st) {
  gen_1d_kernel<<<grid_for(count), 256, 0, st>>>(out, count, pw, init);
  return cudaGetLastError();
}

cudaError_t gen_split(uint4 *out, uint64_t count, const Pow2Table &pw, Fe32 one, cudaStream_t st) {
  gen_split_kernel<<<grid_for(count), 256, 0, st>>>(out, count, pw, one);
  return cudaGetLastError();
}

cudaError_t mul_vec(uint4 *out, const uint4 *a, const uint4 *b, uint64_t count, cudaStream_t st) {
  mul_vec_kernel<<<grid_for(count), 256, 0, st>>>(out, a, b, count);
  return cudaGetLastError();
}

cudaError_t mul_rep(uint4 *out, const uint4 *a, const uint4 *b, uint64_t count, uint32_t reps, int variant,
                    cudaStream_t st) {
  if (variant == 0) {
    mul_rep_kernel<<<grid_for(count), 256, 0, st>>>(out, a, b, count, reps);
  } else {
    const uint64_t threads = count * 8;
    mul_rep_coop_kernel<<<(unsigned)((threads + 255) / 256), 256, 0, st>>>(
        (uint32_t *)out, (const uint32_t *)a, (const uint32_t *)b, count, reps);
  }
  return cudaGetLastError();
}

cudaError_t quotient(uint4 *out, const uint4 *a, const uint4 *b, const uint4 *c, const QuotientZ &z, uint64_t count,
                     cudaStream_t st) {
  quotient_kernel<<<grid_for(count), 256, 0, st>>>(out, a, b, c, z, count);
  return cudaGetLastError();
}

const FieldLaunchers kLaunchers = {prepare, pass,    gen_2d,      gen_1d,  gen_split,
                                   mul_vec, batch,   mul_rep,     matrix_pass, quotient};

}  // namespace

const FieldLaunchers &launchers() { return kLaunchers; }

#endif

}  // namespace NTT_NS
}  // namespace gb300ntt
