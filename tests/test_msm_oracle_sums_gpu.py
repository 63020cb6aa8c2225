"""Sums with long buckets, equal, opposite and infinite operands, sparse scalars, many
windows in several sweeps, against k G by the oracle's integer arithmetic: nothing
of the expected point comes from the library (its inputs do: points t G, a sample
of them checked against the oracle first)."""

import numpy as np
import pytest
import torch

import oracle as O
from oracle import msm_oracle as mo

pytestmark = pytest.mark.gpu

CURVES = {"bn254_g1": ("bn254_fr", mo.BN254_G1, 4), "bls12_381_g1": ("bls12_381_fr", mo.BLS12_381_G1, 6)}


def _scalars(name, n, r, rng):
    if name == "constant":
        return [r - 1] * n
    if name == "bits":
        return [int(v) for v in rng.randint(0, 2, n)]
    if name == "zeros":
        return [0] * n
    if name == "sparse":
        return [int.from_bytes(rng.bytes(32), "little") % r if i % 100 == 0 else 0 for i in range(n)]
    return [int.from_bytes(rng.bytes(32), "little") % r for _ in range(n)]


def _ts(name, n, r, rng):
    if name == "same":
        return [7] * n
    if name == "cancel":
        return [3 if i % 2 else r - 3 for i in range(n)]
    if name == "few":   # equal, opposite and infinite neighbours
        return [(0, 1, r - 1, 2)[int(v)] for v in rng.randint(0, 4, n)]
    return [int.from_bytes(rng.bytes(32), "little") % r for _ in range(n)]


@pytest.mark.parametrize("curve", list(CURVES))
@pytest.mark.parametrize("scalars,points,n,window,flat", [
    ("constant", "same", 9, 8, False), ("constant", "uniform", 20_000, 8, True), ("constant", "cancel", 60, 0, False),
    ("bits", "uniform", 90_001, 0, False), ("bits", "few", 20_000, 8, False), ("zeros", "uniform", 300, 0, False),
    ("sparse", "uniform", 90_001, 9, True), ("sparse", "uniform", 90_001, 0, False), ("uniform", "few", 5_000, 0, False),
    ("uniform", "uniform", 1, 0, False), ("uniform", "uniform", 1_000, 1, False), ("uniform", "uniform", 300_007, 8, False)])
def test_sum_against_the_oracle(curve, scalars, points, n, window, flat):
    import paper_2604_17808_gb300 as lib

    field, group, limbs = CURVES[curve]
    r = O.get_field(field).modulus
    rng = np.random.RandomState(n + len(scalars))
    ss, ts = _scalars(scalars, n, r, rng), _ts(points, n, r, rng)

    def dev(v):
        return torch.from_numpy(O.ints_to_limbs(v).view(np.int64)).cuda()

    plan = lib.MsmPlan(n, window_bits=window, curve=curve)
    pts = torch.empty((n, 2 * limbs), dtype=torch.int64, device="cuda")
    lib.msm_fixed_base(curve, dev(ts), n, pts)
    sample = [0, n // 2, n - 1]
    got = mo.words_to_points(pts[sample].cpu().numpy().view(np.uint64), limbs)
    assert got == [mo.scalar_mul(group, ts[i], group.generator) for i in sample]
    if flat:
        plan.set_bases(pts)
        res = plan.execute_bases(dev(ss))
    else:
        res = plan.execute(dev(ss), pts)
    want = mo.scalar_mul(group, sum(s * t for s, t in zip(ss, ts)) % r, group.generator)
    assert mo.words_to_points(res.cpu().numpy().view(np.uint64).reshape(1, -1), limbs)[0] == want
