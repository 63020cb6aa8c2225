"""The 377- and 753-bit transforms on vectors at the ends of the field (all p -
1; p - 1 and 0 in turn), at sizes of every tile shape, against the Python
oracle.  Exact integers, so the tolerance is zero."""

import numpy as np
import pytest
import torch

from oracle import ntt_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("field,log_n", [("w377", 2), ("w377", 8), ("w377", 10), ("w753", 1), ("w753", 8),
                                         ("w753", 10)])
def test_ends_of_the_field(field, log_n):
    from paper_2604_17808_gb300 import _native as N

    f = O.get_field(field)
    n, words = 1 << log_n, 6 if field == "w377" else 12
    top = [f.modulus - 1] * n
    for x in (top, [v if i % 2 else 0 for i, v in enumerate(top)]):
        raw = b"".join(v.to_bytes(8 * words, "little") for v in x)
        d_x = torch.from_numpy(np.frombuffer(raw, dtype=np.int64).reshape(n, words).copy()).cuda()
        for kind in ("forward", "inverse", "coset", "coset_inverse"):
            d_y = torch.empty_like(d_x)
            N.ntt_wide_transform(field, kind, log_n, d_x, d_y)
            got = d_y.cpu().numpy().tobytes()
            got = [int.from_bytes(got[i:i + 8 * words], "little") for i in range(0, len(got), 8 * words)]
            assert got == O.transform(f, kind, x), kind
