"""Job lists at every tile shape of the batched kernel: few points (2 and 4
elements per thread), many (8), and lists with a 2^11-point pass (2048-element
tiles).  Every job against the same transform run alone, byte for byte."""

import numpy as np
import pytest
import torch

from ntt_synth import uniform_elements

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("field", ["bls12_381_fr", "bn254_fr"])
@pytest.mark.parametrize("sizes,split11", [((1, 4, 10, 12), False), ((17, 8, 2), False), ((18, 18, 16), False),
                                           ((20, 13), False), ((12, 14, 9), True)])
def test_batch_shapes(field, sizes, split11):
    from paper_2604_17808_gb300 import _native as N

    plans, jobs, alone = [], [], []
    try:
        for i, log_n in enumerate(sizes):
            plan = N.ntt_plan_create(field, log_n, coset=True)
            plans.append(plan)
            if split11 and log_n == 12:
                N.ntt_plan_set_passes(plan, [11, 1], 11)
            for kind in ("forward", "coset_inverse"):
                x = torch.from_numpy(uniform_elements(field, 1 << log_n, 31 * i + log_n).view(np.int64)).cuda()
                y, z = torch.empty_like(x), torch.empty_like(x)
                jobs.append((plan, kind, x, y))
                N.ntt_execute(plan, kind, x, z)
                alone.append(z)
        N.ntt_batch_submit(jobs)
        torch.cuda.synchronize()
        assert N.ntt_batch_poll_error() == 0
        assert all(torch.equal(j[3], z) for j, z in zip(jobs, alone))
        for j in jobs:
            j[3].zero_()
        N.ntt_batch_submit_static(jobs)
        torch.cuda.synchronize()
        assert N.ntt_batch_poll_error() == 0
        assert all(torch.equal(j[3], z) for j, z in zip(jobs, alone))
    finally:
        for p in plans:
            N.ntt_plan_destroy(p)
