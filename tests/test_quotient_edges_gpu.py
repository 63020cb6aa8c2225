"""The pointwise quotient at the edges of its operands: a b + (p - c) enters
one Montgomery reduction, so its carries are largest where a, b and p - c
are.  Exact integers, so the tolerance is zero."""

import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("field", ["bls12_381_fr", "bn254_fr"])
def test_quotient_at_the_edges(field):
    import numpy as np

    from paper_2604_17808_gb300 import _native as N

    p = O.get_field(field).modulus
    edge = [0, 1, 2, p - 1, p - 2, 2**32 - 1, 2**64, 2**192 - 1, (2**255 - 1) % p, (p + 1) // 2]
    rows = [(a, b, c) for a in edge for b in edge for c in edge]
    z = [p - 1, 1, 3, 0]
    dev = [torch.from_numpy(O.ints_to_limbs([r[k] for r in rows]).view(np.int64)).cuda() for k in range(3)]
    out = torch.empty_like(dev[0])
    N.ntt_pointwise_quotient(field, *dev, z, out, len(rows))
    got = O.limbs_to_ints(out.cpu().numpy().view(np.uint64))
    assert got == [(a * b - c) * z[i % 4] % p for i, (a, b, c) in enumerate(rows)]
