"""Buckets over many segments: the short sums, the radix-4 trees of the long
ones, the four-lane additions with their excluded cases (equal, opposite and
infinite operands meet in them when every scalar and point is the same), and
segment lengths that shrink with sparse scalars.  Exact, against the closed form
(sum s_i t_i) G."""

import numpy as np
import pytest
import torch

import oracle as O
from oracle import msm_oracle as mo

pytestmark = pytest.mark.gpu

FIELD = {"bn254_g1": "bn254_fr", "bls12_381_g1": "bls12_381_fr"}


def _case(name, n, r):
    rng = np.random.RandomState(n)
    ts = [int(v) for v in rng.randint(1, 2**31 - 1, n)]
    if name == "constant":       # one bucket per window, every point the same
        return [r - 1] * n, [7] * n
    if name == "cancel":         # one bucket, sum O
        return [5] * n, [(3 if i % 2 else r - 3) for i in range(n)]
    if name == "sparse":         # one point in a hundred
        return [int(rng.randint(1, 2**30)) * 2**190 % r if i % 100 == 0 else 0 for i in range(n)], ts
    if name == "repeated":       # many equal and opposite neighbours, points at infinity, dense scalars
        return [int(v) * 2**220 % r + int(v) for v in rng.randint(1, 2**31 - 1, n)], [(0, 1, r - 1, 2)[int(v)] for v in
                                                                                     rng.randint(0, 4, n)]
    return [int(v) for v in rng.randint(0, 2, n)], ts   # bits


@pytest.mark.parametrize("curve", ["bn254_g1", "bls12_381_g1"])
@pytest.mark.parametrize("name", ["constant", "cancel", "sparse", "bits", "repeated"])
@pytest.mark.parametrize("n,flat", [(9, False), (60, False), (300, True), (20_000, False), (20_000, True),
                                    (90_001, False), (90_001, True)])
def test_pieces(curve, name, n, flat):
    import paper_2604_17808_gb300 as lib

    r = O.get_field(FIELD[curve]).modulus
    ss, ts = _case(name, n, r)

    def dev(v):
        return torch.from_numpy(O.ints_to_limbs(v).view(np.int64)).cuda()

    plan = lib.MsmPlan(n, window_bits=8, curve=curve)
    pts = torch.empty((n, plan.point_words), dtype=torch.int64, device="cuda")
    lib.msm_fixed_base(curve, dev([t % r for t in ts]), n, pts)
    if flat:
        plan.set_bases(pts)
        got = plan.execute_bases(dev(ss))
    else:
        got = plan.execute(dev(ss), pts)
    one = lib.MsmPlan(1, curve=curve)   # (sum s t) G, from a single point
    g = torch.empty((1, plan.point_words), dtype=torch.int64, device="cuda")
    lib.msm_fixed_base(curve, dev([1]), 1, g)
    want = one.execute(dev([sum(s * t for s, t in zip(ss, ts)) % r]), g)
    assert torch.equal(got, want)
    if curve == "bn254_g1" and n == 9:   # the single product against the oracle
        k = sum(s * t for s, t in zip(ss, ts)) % r
        assert mo.words_to_points(want.cpu().numpy().view(np.uint64))[0] == mo.fixed_base_points([k])[0]
