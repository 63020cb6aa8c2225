"""In-place transforms of plans that have more than one pass but fit one CTA's
tile (2^9 and 2^10 points): one launch, without the plan's scratch vector, so that
calls on several streams may share a plan.  The single pass against the oracle,
exact, also as an explicit split of one pass."""

import numpy as np
import pytest
import torch

import oracle
from ntt_synth import uniform_elements

pytestmark = pytest.mark.gpu

KINDS = ("forward", "inverse", "coset", "coset_inverse")


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int64)).cuda()


@pytest.mark.parametrize("field", ["bls12_381_fr", "bn254_fr"])
@pytest.mark.parametrize("log_n", [9, 10])
def test_in_place_is_one_launch_and_exact(field, log_n):
    from paper_2604_17808_gb300 import _native as N

    n = 1 << log_n
    p = oracle.get_field(field).modulus
    ends = np.tile(oracle.ints_to_limbs([p - 1, 0]), (n // 2, 1))
    plan = N.ntt_plan_create(field, log_n, coset=True)
    try:
        for shift in (None, 12345):
            if shift:
                N.ntt_plan_set_coset_shift(plan, shift)
            N.ntt_plan_enable_timing(plan, True)
            for x in (uniform_elements(field, n, 900 + log_n), ends):
                for kind in KINDS:
                    buf, out = _dev(x), _dev(x)
                    N.ntt_execute(plan, kind, buf, buf)
                    N.ntt_execute(plan, kind, _dev(x), out)
                    assert torch.equal(buf, out), (kind, shift)
                    if not shift:
                        assert np.array_equal(buf.cpu().numpy().view(np.uint64), oracle.c_transform(field, kind, x)), kind
            N.ntt_plan_read_timing(plan)
            N.ntt_execute(plan, "inverse", buf, buf)
            launches = N.ntt_plan_read_timing(plan)[1]
            assert launches[0] == 1 and sum(launches) == 1
            N.ntt_plan_enable_timing(plan, False)
    finally:
        N.ntt_plan_destroy(plan)


@pytest.mark.parametrize("field", ["bls12_381_fr", "bn254_fr"])
@pytest.mark.parametrize("log_n", [9, 10])
def test_in_place_on_several_streams(field, log_n):
    from paper_2604_17808_gb300 import _native as N

    plan = N.ntt_plan_create(field, log_n, coset=True)
    try:
        streams = [torch.cuda.Stream() for _ in range(4)]
        bufs = [[_dev(uniform_elements(field, 1 << log_n, 97 * s + i)) for i in range(16)] for s in range(4)]
        want = [[torch.empty_like(b) for b in row] for row in bufs]
        for row, wrow in zip(bufs, want):
            for i, (b, w) in enumerate(zip(row, wrow)):
                N.ntt_execute(plan, KINDS[i % 4], b, w, torch.cuda.current_stream())
        torch.cuda.synchronize()
        for i in range(16):
            for stream, row in zip(streams, bufs):
                N.ntt_execute(plan, KINDS[i % 4], row[i], row[i], stream)
        torch.cuda.synchronize()
        assert all(torch.equal(b, w) for row, wrow in zip(bufs, want) for b, w in zip(row, wrow))
    finally:
        N.ntt_plan_destroy(plan)


@pytest.mark.parametrize("field", ["bls12_381_fr", "bn254_fr"])
@pytest.mark.parametrize("log_n", [9, 10])
def test_one_pass_split(field, log_n):
    from paper_2604_17808_gb300 import _native as N

    plan = N.ntt_plan_create(field, log_n, coset=True)
    try:
        N.ntt_plan_set_passes(plan, [log_n], 10)
        x = uniform_elements(field, 1 << log_n, 300 + log_n)
        for kind in KINDS:
            d_x = _dev(x)
            d_y = torch.empty_like(d_x)
            N.ntt_execute(plan, kind, d_x, d_y)
            assert np.array_equal(d_y.cpu().numpy().view(np.uint64), oracle.c_transform(field, kind, x)), kind
    finally:
        N.ntt_plan_destroy(plan)


@pytest.mark.parametrize("field", ["bls12_381_fr", "bn254_fr"])
@pytest.mark.parametrize("log_n", [9, 10])
def test_host_transforms_from_several_threads(field, log_n):
    """Host transforms of one plan from threads with streams of their own, next to
    in-place transforms of device buffers: only one of them at a time may use the
    plan's scratch."""
    import threading

    from paper_2604_17808_gb300 import _native as N

    n, threads, reps = 1 << log_n, 4, 60
    plan = N.ntt_plan_create(field, log_n, coset=True)
    try:
        xs = [uniform_elements(field, n, 40 * t + log_n) for t in range(threads)]
        want = [[oracle.c_transform(field, kind, x) for kind in KINDS] for x in xs]
        wrong = []

        def work(t):
            stream, w = torch.cuda.Stream(), torch.empty((n, 4), dtype=torch.int64, device="cuda")
            h_in = torch.from_numpy(xs[t].view(np.int64)).pin_memory()
            h_out = torch.empty_like(h_in).pin_memory()
            for i in range(reps):
                kind = KINDS[(i + t) % 4]
                if t == 0:
                    with torch.cuda.stream(stream):
                        w.copy_(h_in)
                        N.ntt_execute(plan, kind, w, w, stream)
                        got = w.cpu()
                else:
                    N.ntt_transform_host(plan, kind, h_in, h_out, w, stream)
                    got = h_out
                if not np.array_equal(got.numpy().view(np.uint64), want[t][(i + t) % 4]):
                    wrong.append((t, i))

        pool = [threading.Thread(target=work, args=(t,)) for t in range(threads)]
        for p in pool:
            p.start()
        for p in pool:
            p.join()
        assert not wrong
    finally:
        N.ntt_plan_destroy(plan)
