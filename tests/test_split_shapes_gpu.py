"""Sub-transforms that the default splits do not have, as explicit splits (2^10 in one
pass, 2^19 as 10 + 9 and the other way, three passes at 2^19), and all four kinds at
2^20 points on the butterfly path, where a pass is one wave of seven tiles to a
CTA.  Against the oracle, exact."""

import numpy as np
import pytest
import torch

import oracle
from ntt_synth import uniform_elements

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("field", ["bls12_381_fr", "bn254_fr"])
@pytest.mark.parametrize("log_n,split", [(10, [10]), (19, [10, 9]), (19, [9, 10]), (19, [7, 6, 6]), (20, None)])
def test_split_against_the_oracle(field, log_n, split):
    from paper_2604_17808_gb300 import _native as N

    plan = N.ntt_plan_create(field, log_n, coset=True)
    try:
        N.ntt_plan_set_passes(plan, split or [10, 10], 10)
        x = uniform_elements(field, 1 << log_n, 8800 + log_n)
        for kind in ("coset", "inverse") if split else ("forward", "inverse", "coset", "coset_inverse"):
            d_x = torch.from_numpy(x.view(np.int64)).cuda()
            d_y = torch.empty_like(d_x)
            N.ntt_execute(plan, kind, d_x, d_y)
            assert np.array_equal(d_y.cpu().numpy().view(np.uint64), oracle.c_transform(field, kind, x)), kind
    finally:
        N.ntt_plan_destroy(plan)
