"""Debug builds check tile offsets and twiddle indices, which the pass kernels compute
at run time from the tile shape: every shape of the plans stays quiet and exact,
and an index past the end is reported and its access skipped (asked of the check
itself, with memory behind the end)."""

import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from ntt_synth import uniform_elements

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
KINDS = ("forward", "inverse", "coset", "coset_inverse")


@pytest.mark.parametrize("field", ["bls12_381_fr", "bn254_fr"])
@pytest.mark.parametrize("log_n,split,tile_log", [(2, None, 10), (7, None, 10), (9, [9], 10), (10, None, 10),
                                                  (10, [10], 10), (11, None, 10), (12, [11, 1], 11),
                                                  (14, [1, 3, 10], 11), (19, None, 10), (20, None, 10),
                                                  (21, [5, 8, 8], 10), (21, None, 10)])
def test_shapes_are_quiet_and_exact(field, log_n, split, tile_log):
    from paper_2604_17808_gb300 import _native as N

    dbg = N.load_debug()
    plan, ref = ctypes.c_void_p(), N.ntt_plan_create(field, log_n, coset=True)
    assert dbg.ntt_plan_create(ctypes.byref(plan), N.FIELD[field], log_n, 1) == 0
    try:
        if split:
            arr = (ctypes.c_uint32 * len(split))(*split)
            assert dbg.ntt_plan_set_passes(plan, len(split), arr, tile_log) == 0
        x = torch.from_numpy(uniform_elements(field, 1 << log_n, 4 + log_n).view(np.int64)).cuda()
        for kind in KINDS:
            y, z, w = torch.empty_like(x), torch.empty_like(x), x.clone()
            N.ntt_execute(ref, kind, x, z)
            assert dbg.ntt_execute(plan, N.KIND[kind], x.data_ptr(), y.data_ptr(), None) == 0
            assert dbg.ntt_execute(plan, N.KIND[kind], w.data_ptr(), w.data_ptr(), None) == 0
            torch.cuda.synchronize()
            assert torch.equal(y, z) and torch.equal(w, z), kind
        code = ctypes.c_uint32(99)
        assert dbg.ntt_plan_poll_error(plan, ctypes.byref(code)) == 0 and code.value == 0
    finally:
        dbg.ntt_plan_destroy(plan)
        N.ntt_plan_destroy(ref)


SOURCE = r"""
#define NTT_DEBUG
#include "ntt_pass.cuh"
using namespace gb300ntt;
// One thread; two tiles' shared memory and two tables' entries for one of each.
__global__ void probe(const uint4 *table, uint32_t *err, uint32_t index, int what, uint32_t *out) {
  using El = Elem256<FieldBls12381Fr>;
  extern __shared__ uint4 smem[];
  const uint32_t tile = (uint32_t)__cvta_generic_to_shared(smem);
  const TileShape s = {5, 6, 1};   // 64 elements, sub-transforms of 32 points
  PassArgs a = {};
  a.dft_tw = table;
  a.dbg_err = err;
  uint32_t ones[8], A[8], B[8] = {};
  for (int k = 0; k < 8; ++k) ones[k] = 1, A[k] = 2;
  for (uint32_t i = 0; i < 2 * 64; ++i) El::tile_store(tile, 32 * i, 7, ones);
  if (what == 0) tile_get<El>(a, s, A, tile, index);
  if (what == 1) { tile_put<El>(a, s, tile, index, A); El::tile_load(A, tile, index, 7); }
  if (what == 2) twiddle_get<El>(a, s, A, B, table, index);
  out[0] = A[0];
  out[1] = B[0];
}
extern "C" int run(const void *table, uint32_t *err, uint32_t index, int what, uint32_t *out) {
  probe<<<1, 1, 2 * 64 * 32>>>((const uint4 *)table, err, index, what, out);
  return (int)cudaDeviceSynchronize();
}
"""


def test_checks_fire_past_the_end(tmp_path):
    src, path = tmp_path / "probe.cu", tmp_path / "probe.so"
    src.write_text(SOURCE)
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared", "-Xcompiler",
                    "-fPIC", "-I", os.path.join(ROOT, "paper_2604_17808_gb300", "csrc"), "-o", str(path), str(src)],
                   check=True)
    lib, ptr = ctypes.CDLL(str(path)), ctypes.c_void_p
    table = torch.full((2 * 16 * 16,), 3, dtype=torch.int32, device="cuda")   # 32 entries of 64 bytes, 16 of them the table
    # (what, index): the last one inside, the first one outside; values read back
    for what, inside, outside, seen, skipped in ((0, 63 * 32, 64 * 32, (1, 0), (0, 0)),
                                                 (1, 63 * 32, 64 * 32, (2, 0), (1, 0)),
                                                 (2, 15, 16, (3, 3), (0, 0))):
        for index, values, code in ((inside, seen, 0), (outside, skipped, 8)):
            err = torch.zeros(1, dtype=torch.int32, device="cuda")
            out = torch.zeros(2, dtype=torch.int32, device="cuda")
            torch.cuda.synchronize()
            assert lib.run(ptr(table.data_ptr()), ptr(err.data_ptr()), index, what, ptr(out.data_ptr())) == 0
            assert tuple(out.tolist()) == values and err.item() == code, (what, index)
