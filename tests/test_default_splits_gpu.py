"""The default pass split of a plan: as few passes of at most 2^10 points as
possible, but two where one CTA of 128 threads with 2 elements each would not hold
the transform.  In a process of its own: a tuned size keeps its tuned split in the
process that tuned it."""

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
from paper_2604_17808_gb300 import _native as N
for field in ("bls12_381_fr", "bn254_fr"):
    for log_n in (1, 8, 9, 10, 11, 18, 19, 20, 21, 22):
        plan = N.ntt_plan_create(field, log_n)
        print(N.ntt_plan_describe(plan)["pass_log"])
        N.ntt_plan_destroy(plan)
"""

SPLITS = [[1], [8], [5, 4], [5, 5], [6, 5], [9, 9], [10, 9], [10, 10], [7, 7, 7], [8, 7, 7]]


def test_default_splits():
    env = {k: v for k, v in os.environ.items() if k != "NTT_TUNE_CACHE"}
    r = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, capture_output=True, text=True, timeout=300, check=True,
                       env=env)
    assert [eval(line) for line in r.stdout.splitlines()] == 2 * SPLITS
