"""Squares and differences of two products over the base fields of the curves
(csrc/fp_square.cuh), against Python integers: operands whose limbs are all zeros
or all ones in every combination that stays below the modulus, which is where the
carry chains end or do not, the ends of the range, and random ones."""
import ctypes
import itertools
import os
import random
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include "ec_xyzz.cuh"
using namespace gb300ntt;
template <class T>
__global__ void probe(const uint32_t *x, uint32_t *square, uint32_t *diff, uint32_t n) {
  constexpr int L = T::L;
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  uint32_t v[4][L], r[L];
  for (int k = 0; k < 4; ++k)
    for (int j = 0; j < L; ++j) v[k][j] = x[(size_t)((i + (uint64_t)k * k * 7) % n) * L + j];
  f_sqr<T, true>(r, v[0]);
  for (int j = 0; j < L; ++j) square[(size_t)i * L + j] = r[j];
  uint32_t p[L];
  for (int j = 0; j < L; ++j) p[j] = T::modulus(j);
  words_add<L>(p, p, v[0]);
  f_sqr<T, true>(r, p);
  for (int j = 0; j < L; ++j) square[(size_t)(n + i) * L + j] = r[j];
  f_mul_sub<T>(r, v[0], v[1], v[2], v[3]);
  for (int j = 0; j < L; ++j) diff[(size_t)i * L + j] = r[j];
}
extern "C" int run(int curve, const uint32_t *x, uint32_t *square, uint32_t *diff, uint32_t n) {
  if (curve == 0) probe<FqBn254><<<(n + 127) / 128, 128>>>(x, square, diff, n);
  else probe<FqBls381><<<(n + 127) / 128, 128>>>(x, square, diff, n);
  return (int)cudaDeviceSynchronize();
}
"""

MODULUS = {
    0: 21888242871839275222246405745257275088696311157297823662689037894645226208583,
    1: int("1a0111ea397fe69a4b1ba7b6434bacd764774b84f38512bf6730d2a0f6b0f6241eabfffeb153ffffb9feffffffffaaab", 16),
}


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    d = tmp_path_factory.mktemp("field_square")
    src, lib = d / "probe.cu", d / "probe.so"
    src.write_text(SOURCE)
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared", "-Xcompiler",
                    "-fPIC", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2604_17808_gb300", "csrc"), "-o", str(lib), str(src)], check=True)
    return ctypes.CDLL(str(lib))


@pytest.mark.parametrize("curve,limbs", [(0, 8), (1, 12)])
def test_squares_and_differences(probe, curve, limbs):
    import torch

    p, rng = MODULUS[curve], random.Random(5 + curve)
    xs = [0, 1, 2, p - 1, p - 2, p >> 1, (p >> 1) + 1]
    top = p >> (32 * (limbs - 1))
    for pattern in itertools.product((0, 0xFFFFFFFF), repeat=limbs - 1):
        low = sum(w << (32 * j) for j, w in enumerate(pattern))
        xs += [low, (top - 1) << (32 * (limbs - 1)) | low]
    xs += [rng.randrange(p) for _ in range(5000)]
    rng.shuffle(xs)
    n = len(xs)
    assert all(0 <= x < p for x in xs)
    raw = b"".join(x.to_bytes(4 * limbs, "little") for x in xs)
    x = torch.frombuffer(bytearray(raw), dtype=torch.int32).cuda()
    square, diff = torch.empty(2 * x.numel(), dtype=torch.int32, device="cuda"), torch.empty_like(x)
    ptr = ctypes.c_void_p
    assert probe.run(curve, ptr(x.data_ptr()), ptr(square.data_ptr()), ptr(diff.data_ptr()), ctypes.c_uint32(n)) == 0
    r_inv = pow(1 << (32 * limbs), -1, p)

    def ints(t):
        b = t.cpu().numpy().tobytes()
        return [int.from_bytes(b[i:i + 4 * limbs], "little") for i in range(0, len(b), 4 * limbs)]

    assert ints(square) == 2 * [v * v * r_inv % p for v in xs]   # of v and of v + p
    assert ints(diff) == [(xs[i] * xs[(i + 7) % n] - xs[(i + 28) % n] * xs[(i + 63) % n]) * r_inv % p for i in range(n)]
