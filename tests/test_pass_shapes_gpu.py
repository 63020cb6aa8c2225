"""Every tile shape of the butterfly passes (2, 4 and 8 elements per thread,
sub-transforms from 2 points to 2^11) against the oracle, on vectors that push
the lazy values in [0, 2p) to their ends: all p - 1, p - 1 and 0 in turn, and
uniform ones.  Exact integers, so the tolerance is zero."""

import numpy as np
import pytest
import torch

import oracle
from ntt_synth import uniform_elements

pytestmark = pytest.mark.gpu


def _vectors(field, log_n):
    n = 1 << log_n
    p = oracle.get_field(field).modulus
    top = np.tile(oracle.ints_to_limbs([p - 1]), (n, 1))
    alternating = top.copy()
    alternating[1::2] = 0
    return [top, alternating, uniform_elements(field, n, 7700 + log_n)]


# default splits: 2^1..2^3 inside one thread, 2^7 and 2^10 one pass, 2^17 (9, 8)
# with 4 and 2 elements per thread, 2^19 (10, 9) with 8 and 4, 2^21 (7, 7, 7)
# many waves; explicit splits put a 2^11-point pass and a 2-point one in front
@pytest.mark.parametrize("field", ["bls12_381_fr", "bn254_fr"])
@pytest.mark.parametrize("log_n,split,tile_log", [(1, None, 10), (2, None, 10), (3, None, 10), (7, None, 10),
                                                  (10, None, 10), (17, None, 10), (19, None, 10), (21, None, 10),
                                                  (12, [11, 1], 11), (13, [2, 11], 10), (14, [1, 3, 10], 11)])
def test_shapes_match_the_oracle(field, log_n, split, tile_log):
    from paper_2604_17808_gb300 import _native as N

    plan = N.ntt_plan_create(field, log_n, coset=True)
    try:
        if split:
            N.ntt_plan_set_passes(plan, split, tile_log)
        vectors = _vectors(field, log_n)
        kinds = ("forward", "inverse", "coset", "coset_inverse") if log_n < 19 else ("inverse", "coset")
        for x in vectors if log_n < 19 else vectors[-1:]:
            for kind in kinds:
                d_x = torch.from_numpy(np.ascontiguousarray(x).view(np.int64)).cuda()
                d_y = torch.empty_like(d_x)
                N.ntt_execute(plan, kind, d_x, d_y)
                got = d_y.cpu().numpy().view(np.uint64)
                assert np.array_equal(got, oracle.c_transform(field, kind, x)), (kind,)
    finally:
        N.ntt_plan_destroy(plan)
