"""The first call of a size builds its tables; the field constants behind them come
from one thread and are computed once for the size, however many passes it has.
At 753 bits they are nearly all of the first call, so that of 2^9 points (two
passes) takes about as long as that of 2^8 (one)."""

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import time
import torch
from paper_2604_17808_gb300 import _native as N
def first(log_n):
    x = torch.ones((1 << log_n, 12), dtype=torch.int64, device="cuda")
    y = torch.empty_like(x)
    torch.cuda.synchronize()
    t = time.perf_counter()
    N.ntt_wide_transform("w753", "forward", log_n, x, y)
    torch.cuda.synchronize()
    return time.perf_counter() - t
first(2)
print(first(8), first(9))
"""


def test_first_call_does_not_grow_with_the_passes():
    r = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, capture_output=True, text=True, timeout=300, check=True)
    one, two = map(float, r.stdout.split())
    assert two < 1.6 * one, (one, two)   # computed once per table it would be 2.0
