"""Which buckets the long trees take, in a call over one window: the limit depends on
how long the average bucket is, of the windows that the call runs over.  The
library's source is compiled with a function that reads a plan's totals: 100,000
entries in the 2048 buckets of one 12-bit window are 49 a bucket and six segments
of eight, longer than a segment, so that the buckets of up to nine segments are
added up by one thread each."""

import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from ntt_synth import uniform_elements

pytestmark = [pytest.mark.gpu, pytest.mark.timeout(900)]

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include "msm.cu"
extern "C" int totals(msm_plan p, uint32_t out[4]) {
  gb300ntt::MsmTotals t;
  if (cudaMemcpy(&t, p->tot, sizeof t, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
  out[0] = t.entries;
  out[1] = t.seg_len;
  out[2] = t.crossing;
  out[3] = t.items[0];
  return 0;
}
"""


def test_limit_follows_the_windows_of_the_call(tmp_path):
    import paper_2604_17808_gb300 as native

    src, path = tmp_path / "probe.cu", tmp_path / "probe.so"
    src.write_text(SOURCE)
    csrc = os.path.join(ROOT, "paper_2604_17808_gb300", "csrc")
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared", "-Xcompiler",
                    "-fPIC", "-I", csrc, "-o", str(path), str(src)], check=True)
    lib = ctypes.CDLL(str(path))
    n, u64, ptr = 100_000, ctypes.c_uint64, ctypes.c_void_p

    def dev(seed):
        return torch.from_numpy(uniform_elements("bn254_fr", n, seed).view(np.int64)).cuda()

    scalars, points = dev(1), torch.empty((n, 8), dtype=torch.int64, device="cuda")
    native.msm_fixed_base("bn254_g1", dev(2), n, points)
    result = torch.empty(8, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    plan = ptr()
    assert lib.msm_plan_create(ctypes.byref(plan), 0, u64(n), 12) == 0
    try:
        assert lib.msm_execute_windows(plan, ptr(scalars.data_ptr()), ptr(points.data_ptr()), u64(n), 3, 4,
                                       ptr(result.data_ptr()), None) == 0
        out = (ctypes.c_uint32 * 4)()
        assert lib.totals(plan, out) == 0
    finally:
        assert lib.msm_plan_destroy(plan) == 0
    entries, seg_len, crossing, items = out
    assert 0.99 * n < entries <= n and seg_len == 8
    assert crossing > 1900 and items < 300, (crossing, items)
    want = native.MsmPlan(n, window_bits=12).execute_windows(scalars, points, 3, 4)
    assert torch.equal(result, want)
