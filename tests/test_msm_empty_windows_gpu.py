"""Scalars that leave most buckets and windows empty (all zero, all one, 20 bits):
the sum is exact, and the call does not spend the time of the doublings and
additions of the point at infinity."""

import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu

FIELD = {"bn254_g1": "bn254_fr", "bls12_381_g1": "bls12_381_fr"}


def _ms(plan, scalars, points):
    best = 1e9
    plan.execute(scalars, points)
    for _ in range(8):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        plan.execute(scalars, points)
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("curve", ["bn254_g1", "bls12_381_g1"])
def test_empty_windows(curve):
    import numpy as np

    import paper_2604_17808_gb300 as lib

    n, r = 5000, O.get_field(FIELD[curve]).modulus
    rng = np.random.RandomState(3)

    def dev(v):
        return torch.from_numpy(O.ints_to_limbs(v).view(np.int64)).cuda()

    plan = lib.MsmPlan(n, curve=curve)
    ts = [int(v) for v in rng.randint(1, 2**31 - 1, n)]
    points = torch.empty((n, plan.point_words), dtype=torch.int64, device="cuda")
    lib.msm_fixed_base(curve, dev(ts), n, points)
    uniform = [int.from_bytes(rng.bytes(32), "little") % r for _ in range(n)]
    lists = {"zeros": [0] * n, "ones": [1] * n, "20 bits": [int(v) for v in rng.randint(0, 2**20, n)],
             "one point": [0] * (n - 1) + [r - 1]}
    for name, ss in lists.items():
        want = torch.empty((1, plan.point_words), dtype=torch.int64, device="cuda")
        lib.msm_fixed_base(curve, dev([sum(s * t for s, t in zip(ss, ts)) % r]), 1, want)
        assert torch.equal(plan.execute(dev(ss), points), want[0]), name
    full = _ms(plan, dev(uniform), points)
    assert _ms(plan, dev(lists["zeros"]), points) < 0.45 * full
