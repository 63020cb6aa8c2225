"""Calls over many points, all windows and ranges of them, against the closed form
of the signed digits: accumulation threads that take several segments each with
buckets over hundreds of segments, and scatters that take their windows in several
sweeps (more sorted entries than stay in the L2)."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu

FIELD = {"bn254_g1": "bn254_fr", "bls12_381_g1": "bls12_381_fr"}
C = 8


def _digits(s, count):
    out, carry = [], 0
    for k in range(count):
        v = (s >> (C * k) & (2**C - 1)) + carry
        carry = int(v > 2**(C - 1))
        out.append(v - carry * 2**C)
    return out


@pytest.mark.parametrize("curve,n,windows", [("bn254_g1", 1_200_003, None), ("bn254_g1", 1_200_003, (5, 21)),
                                             ("bn254_g1", 800_001, (30, 31)),
                                             ("bls12_381_g1", 600_001, None), ("bls12_381_g1", 600_001, (30, 32))])
def test_many_points(curve, n, windows):
    import paper_2604_17808_gb300 as lib

    r = O.get_field(FIELD[curve]).modulus
    rng = np.random.RandomState(n)
    distinct = [int.from_bytes(rng.bytes(32), "little") % r for _ in range(997)] + [0, 1, r - 1]
    ts = [int(v) for v in rng.randint(1, 2**31 - 1, n)]

    def dev(v):
        return torch.from_numpy(O.ints_to_limbs(v).view(np.int64)).cuda()

    plan = lib.MsmPlan(n, window_bits=C, curve=curve)
    pts = torch.empty((n, plan.point_words), dtype=torch.int64, device="cuda")
    lib.msm_fixed_base(curve, dev(ts), n, pts)
    pick = torch.arange(n, device="cuda") % len(distinct)
    scalars = dev(distinct)[pick].contiguous()
    count = plan.info()["num_windows"]
    kb, ke = windows or (0, count)
    got = [plan.execute_windows(scalars, pts, kb, ke) for _ in range(3)]
    parts = [sum(d << (C * k) for k, d in enumerate(_digits(s, count)) if kb <= k < ke) for s in distinct]
    total = sum(parts[i % len(distinct)] * t for i, t in enumerate(ts)) % r
    one = lib.MsmPlan(1, curve=curve)
    g = torch.empty((1, plan.point_words), dtype=torch.int64, device="cuda")
    lib.msm_fixed_base(curve, dev([1]), 1, g)
    want = one.execute(dev([total]), g)
    assert all(torch.equal(v, want) for v in got)
