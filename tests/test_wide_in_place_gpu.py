"""In-place calls of the 377- and 753-bit transforms around the largest size that
fits one tile (2^10 and 2^9 points): the same bytes as out of place, and up to
that size on several streams at once, as one launch that uses no scratch vector."""

import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu

KINDS = ("forward", "inverse", "coset", "coset_inverse")
CASES = [("w377", 8), ("w377", 9), ("w377", 10), ("w377", 11), ("w753", 8), ("w753", 9), ("w753", 10)]


def _vector(field, log_n, seed):
    words, top = (6, 0x1921FB54442D18) if field == "w377" else (12, 0x1921F)
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randint(-2**63, 2**63 - 1, (1 << log_n, words), dtype=torch.int64, device="cuda", generator=g)
    x[:, -1] = torch.randint(0, top, (1 << log_n,), dtype=torch.int64, device="cuda", generator=g)
    return x


@pytest.mark.parametrize("field,log_n", CASES)
def test_in_place_equals_out_of_place(field, log_n):
    from paper_2604_17808_gb300 import _native as N

    for kind in KINDS:
        for shift in (None, 77) if kind.startswith("coset") else (None,):
            x = _vector(field, log_n, 5)
            y = torch.empty_like(x)
            N.ntt_wide_transform(field, kind, log_n, x, y, None, shift)
            N.ntt_wide_transform(field, kind, log_n, x, x, None, shift)
            assert torch.equal(x, y), (kind, shift)


@pytest.mark.parametrize("field,log_n", [c for c in CASES if c[1] <= (10 if c[0] == "w377" else 9)])
def test_one_launch_on_several_streams(field, log_n):
    from paper_2604_17808_gb300 import _native as N

    x = _vector(field, log_n, 6)
    N.ntt_wide_transform(field, "inverse", log_n, x, x)
    torch.cuda.synchronize()
    rt, graph, count = ctypes.CDLL("libcudart.so.13"), ctypes.c_void_p(), ctypes.c_size_t()   # torch's
    stream = torch.cuda.Stream()
    handle = ctypes.c_void_p(stream.cuda_stream)
    assert rt.cudaStreamBeginCapture(handle, 1) == 0
    N.ntt_wide_transform(field, "inverse", log_n, x, x, stream)
    assert rt.cudaStreamEndCapture(handle, ctypes.byref(graph)) == 0
    assert rt.cudaGraphGetNodes(graph, None, ctypes.byref(count)) == 0
    assert rt.cudaGraphDestroy(graph) == 0
    assert count.value == 1
    streams = [torch.cuda.Stream() for _ in range(4)]
    bufs = [[_vector(field, log_n, 100 * s + i) for i in range(8)] for s in range(4)]
    want = [[torch.empty_like(b) for b in row] for row in bufs]
    for row, wrow in zip(bufs, want):
        for b, w in zip(row, wrow):
            N.ntt_wide_transform(field, "forward", log_n, b, w)
    torch.cuda.synchronize()
    for i in range(8):
        for stream, row in zip(streams, bufs):
            N.ntt_wide_transform(field, "forward", log_n, row[i], row[i], stream)
    torch.cuda.synchronize()
    assert all(torch.equal(b, w) for row, wrow in zip(bufs, want) for b, w in zip(row, wrow))
