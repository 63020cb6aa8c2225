"""Host buffers that the passes read and write themselves (page-locked), ones
that are copied (pageable, misaligned) and mixtures: the same bytes as the
device transform, in h_out and in d_work, at one- and two-pass sizes and at the
tile shapes of the larger transfers."""

import numpy as np
import pytest
import torch

from ntt_synth import uniform_elements

pytestmark = pytest.mark.gpu


def _host(n, how):
    if how == "pageable":
        return torch.empty((n, 4), dtype=torch.int64)
    if how == "misaligned":   # page-locked, 8 bytes past an element boundary
        return torch.empty(4 * n + 4, dtype=torch.int64).pin_memory()[1:4 * n + 1].view(n, 4)
    return torch.empty((n, 4), dtype=torch.int64).pin_memory()


@pytest.mark.parametrize("field,log_n", [("bls12_381_fr", 2), ("bn254_fr", 8), ("bls12_381_fr", 10),
                                         ("bn254_fr", 15), ("bls12_381_fr", 19), ("bn254_fr", 20)])
@pytest.mark.parametrize("src,dst", [("pinned", "pinned"), ("pageable", "pinned"), ("pinned", "misaligned"),
                                     ("misaligned", "pageable"), ("pinned", "same")])
def test_host_buffers(field, log_n, src, dst):
    from paper_2604_17808_gb300 import _native as N

    n = 1 << log_n
    x = torch.from_numpy(uniform_elements(field, n, 90 + log_n).view(np.int64))
    plan = N.ntt_plan_create(field, log_n, coset=True)
    try:
        for kind in ("forward", "coset_inverse"):
            d_x = x.cuda()
            want = torch.empty_like(d_x)
            N.ntt_execute(plan, kind, d_x, want)
            h_in = _host(n, src)
            h_in.copy_(x)
            h_out = h_in if dst == "same" else _host(n, dst)
            work = torch.empty_like(d_x)
            N.ntt_transform_host(plan, kind, h_in, h_out, work)
            assert torch.equal(h_out, want.cpu()) and torch.equal(work, want), kind
    finally:
        N.ntt_plan_destroy(plan)
