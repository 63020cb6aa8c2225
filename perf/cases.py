"""The calls this library is used for, as measurable cases.

A case is a dict of plain values; `prepare` makes what a prover's program holds
before the call (vectors on the GPU, a plan), `run` is one pass through the
public entry points.  Sizes are the ones of the benchmark and the tests; the
drawn cases spread over the same ranges.

Every output is a vector of field elements or a curve point: whole numbers, the
same bytes on every run.
"""

from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2604_17808_gb300 as lib
from paper_2604_17808_gb300 import _native as native

# modulus, 64-bit words per element, generator
FIELDS = {
    "bls12_381_fr": (0x73EDA753299D7D483339D80809A1D80553BDA402FFFE5BFEFFFFFFFF00000001, 4, 7),
    "bn254_fr": (0x30644E72E131A029B85045B68181585D2833E84879B9709143E1F593F0000001, 4, 5),
    "w377": (0x1921FB54442D18469898CC51701B839A252049C1114CF98E804177D4C76273644A29410F31C6809BBDF2BD500000001, 6, 7),
    "w753": (0x1921FB54442D18469898CC51701B839A252049C1114CF98E804177D4C76273644A29410F31C6809BBDF2A33679A748636605614DBE4BE286E9FC26ADADAA3848BC90B6AECC4BCFD8DE89885D34C6FDAD617FEB96DE80D6FDBDCD300000001, 12, 11),
}
# scalar field, base-field modulus, generator point, 64-bit words per coordinate
CURVES = {
    "bn254_g1": ("bn254_fr", 0x30644E72E131A029B85045B68181585D97816A916871CA8D3C208C16D87CFD47, (1, 2), 4),
    "bls12_381_g1": (
        "bls12_381_fr",
        0x1A0111EA397FE69A4B1BA7B6434BACD764774B84F38512BF6730D2A0F6B0F6241EABFFFEB153FFFFB9FEFFFFFFFFAAAB,
        (0x17F1D3A73197D7942695638C4FA9AC0FC3688C4F9774B905A14E3A3F171BAC586C55E83FF97A1AEFFB3AF00ADB22C6BB,
         0x08B3F481E3AAA0F1A09E30ED741D8AE4FCF5E095D5D00AF600DB18CB2C04B3EDD03CC744A2888AE40CAA232946C5E7E1), 6),
}
KINDS = ("forward", "inverse", "coset", "coset_inverse")


def listed():
    return [
        # smallest proofs and recursion layers: one small vector, launch latency counts
        {"name": "transform_2e12", "op": "transform", "field": "bls12_381_fr", "kind": "forward", "log_n": 12,
         "path": "auto"},
        # an ordinary circuit: evaluations back to coefficients
        {"name": "inverse_2e17", "op": "transform", "field": "bn254_fr", "kind": "inverse", "log_n": 17,
         "path": "auto"},
        # the benchmark's workload: there and back at 2^20
        {"name": "step_2e20", "op": "step", "field": "bls12_381_fr", "log_n": 20},
        # the largest single vector: a low-degree extension onto a coset
        {"name": "coset_2e24", "op": "transform", "field": "bn254_fr", "kind": "coset", "log_n": 24, "path": "auto"},
        # the tensor-core path, chosen by the caller, back from the coset
        {"name": "matrix_2e22", "op": "transform", "field": "bls12_381_fr", "kind": "coset_inverse", "log_n": 22,
         "path": "matrix"},
        # many polynomials of one proof system in one submission
        {"name": "batch_64", "op": "batch", "field": "bls12_381_fr", "jobs": 64, "min_log": 14, "max_log": 22,
         "pick": 4},
        # a prover's quotient step on a coset four times as long as the domain
        {"name": "quotient_2e18", "op": "quotient", "field": "bn254_fr", "log_n": 18},
        # vectors in pinned host memory, there and back over the bus
        {"name": "host_2e18", "op": "host", "field": "bls12_381_fr", "kind": "forward", "log_n": 18},
        # a commitment to a large ragged vector of points
        {"name": "msm_bn254_4m", "op": "msm", "curve": "bn254_g1", "n": 4_194_301, "scalars": "uniform"},
        # a small ragged one of witness values: mostly bits and short numbers
        {"name": "msm_bls_witness", "op": "msm", "curve": "bls12_381_g1", "n": 49_999, "scalars": "witness"},
        # polynomial commitment with the setup points prepared: inverse transform, then the sum
        {"name": "commit_2e20", "op": "commit", "curve": "bls12_381_g1", "log_n": 20},
        # the wide field
        {"name": "wide_753_2e18", "op": "wide", "field": "w753", "kind": "coset", "log_n": 18},
    ]


def draw(rng: random.Random):
    op = rng.choices(("transform", "step", "batch", "quotient", "host", "msm", "commit", "wide"),
                     (4, 2, 2, 1, 2, 4, 1, 3))[0]
    field = rng.choice(("bls12_381_fr", "bn254_fr"))
    curve = rng.choice(("bn254_g1", "bls12_381_g1"))
    if op == "transform":
        path = rng.choice(("auto", "auto", "matrix"))
        return {"op": op, "field": field, "kind": rng.choice(KINDS),
                "log_n": rng.randint(12 if path == "matrix" else 8, 24), "path": path}
    if op == "step":
        return {"op": op, "field": field, "log_n": rng.randint(8, 23)}
    if op == "batch":
        lo = rng.randint(10, 16)
        return {"op": op, "field": rng.choice((field, "both")), "jobs": rng.randint(2, 48), "min_log": lo,
                "max_log": rng.randint(lo, 21), "pick": rng.randrange(1000)}
    if op == "quotient":
        return {"op": op, "field": field, "log_n": rng.randint(9, 20)}
    if op == "host":
        return {"op": op, "field": field, "kind": rng.choice(KINDS), "log_n": rng.randint(10, 21)}
    if op == "msm":
        # the larger curve at most at the cost of the largest listed one
        top = 1 << (22 if curve == "bn254_g1" else 20)
        return {"op": op, "curve": curve, "n": int(math.exp(rng.uniform(math.log(500), math.log(top)))) | 1,
                "scalars": rng.choice(("uniform", "witness"))}
    if op == "commit":
        return {"op": op, "curve": curve, "log_n": rng.randint(10, 20)}
    wide = rng.choice(("w377", "w753"))
    return {"op": op, "field": wide, "kind": rng.choice(KINDS), "log_n": rng.randint(8, 20 if wide == "w377" else 19)}


# ------------------------------------------------------------------ inputs


def _elements(field, n, seed):
    """n elements below the modulus, uniform but for its last 2^-50th or less: [n, words] int64 on the GPU."""
    p, words, _ = FIELDS[field]
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randint(-2**63, 2**63 - 1, (n, words), dtype=torch.int64, device="cuda", generator=g)
    x[:, -1] = torch.randint(0, p >> (64 * (words - 1)), (n,), dtype=torch.int64, device="cuda", generator=g)
    return x


def _scalars(case, field, n, seed):
    x = _elements(field, n, seed)
    if case.get("scalars") == "witness":
        # half bits, a quarter 16-bit numbers, a quarter full field elements
        g = torch.Generator(device="cuda").manual_seed(seed + 77)
        sort = torch.randint(0, 4, (n,), device="cuda", generator=g)
        small = sort < 3
        x[small, 1:] = 0
        x[:, 0] = torch.where(sort < 2, x[:, 0] & 1, torch.where(sort == 2, x[:, 0] & 0xFFFF, x[:, 0]))
    return x


def _points(curve, n, seed):
    """n points t G with uniform t, affine: [n, 2 words]; and the t."""
    field, _, _, words = CURVES[curve]
    t = _elements(field, n, seed)
    pts = torch.empty((n, 2 * words), dtype=torch.int64, device="cuda")
    lib.msm_fixed_base(curve, t, n, pts, torch.cuda.current_stream())
    return pts, t


def _plan(field, log_n, kind="forward", path="auto"):
    return lib.Plan(field, log_n, coset=kind.startswith("coset"), path=None if path == "auto" else path)


def _batch_jobs(case):
    """(field, log_n, kind) of every job; the same for every seed of the inputs."""
    rng = random.Random(case["pick"])
    fields = ("bls12_381_fr", "bn254_fr") if case["field"] == "both" else (case["field"],)
    return [(rng.choice(fields), rng.randint(case["min_log"], case["max_log"]), rng.choice(("forward", "inverse")))
            for _ in range(case["jobs"])]


def _quotient_z(field, log_n):
    """1 / (x^n - 1) on the coset of 4 n points: its four values."""
    p, _, gen = FIELDS[field]
    s_n = pow(gen, 1 << log_n, p)
    w4 = pow(gen, (p - 1) // 4, p)
    return [pow(s_n * pow(w4, j, p) - 1, -1, p) for j in range(4)]


def prepare(case, seed):
    op = case["op"]
    stream = torch.cuda.current_stream()
    if op in ("transform", "step"):
        n = 1 << case["log_n"]
        x = _elements(case["field"], n, seed)
        plan = _plan(case["field"], case["log_n"], case.get("kind", "forward"), case.get("path", "auto"))
        return {"case": case, "plan": plan, "x": x, "y": torch.empty_like(x), "z": torch.empty_like(x)}
    if op == "batch":
        plans, jobs, outs = {}, [], []
        for i, (field, log_n, kind) in enumerate(_batch_jobs(case)):
            if (field, log_n) not in plans:
                plans[field, log_n] = _plan(field, log_n)
            x = _elements(field, 1 << log_n, seed * 64 + i)
            outs.append(torch.empty_like(x))
            jobs.append((plans[field, log_n].handle, kind, x, outs[-1]))
        return {"case": case, "plans": plans, "jobs": jobs, "outs": outs}
    if op == "quotient":
        m = 4 << case["log_n"]
        plan = _plan(case["field"], case["log_n"] + 2, "coset")
        x = [_elements(case["field"], m, 3 * seed + j) for j in range(3)]
        return {"case": case, "plan": plan, "x": x, "y": [torch.empty_like(v) for v in x],
                "z": _quotient_z(case["field"], case["log_n"]), "q": torch.empty_like(x[0])}
    if op == "host":
        x = _elements(case["field"], 1 << case["log_n"], seed)
        return {"case": case, "plan": _plan(case["field"], case["log_n"], case["kind"]), "x": x.cpu().pin_memory(),
                "y": torch.empty(x.shape, dtype=torch.int64).pin_memory(), "work": x}
    if op == "msm":
        points, _ = _points(case["curve"], case["n"], seed + 1)
        scalars = _scalars(case, CURVES[case["curve"]][0], case["n"], seed)
        return {"case": case, "plan": lib.MsmPlan(case["n"], curve=case["curve"]), "s": scalars, "p": points}
    if op == "commit":
        n = 1 << case["log_n"]
        field = CURVES[case["curve"]][0]
        points, _ = _points(case["curve"], n, seed + 1)
        msm = lib.MsmPlan(n, curve=case["curve"])
        msm.set_bases(points, stream=stream)
        x = _elements(field, n, seed)
        return {"case": case, "msm": msm, "plan": _plan(field, case["log_n"]), "x": x, "y": torch.empty_like(x)}
    x = _elements(case["field"], 1 << case["log_n"], seed)
    return {"case": case, "x": x, "y": torch.empty_like(x)}


def run(state):
    case = state["case"]
    op = case["op"]
    stream = torch.cuda.current_stream()
    if op == "transform":
        return state["plan"].run(case["kind"], state["x"], state["y"], stream)
    if op == "step":
        state["plan"].forward(state["x"], state["y"], stream)
        state["plan"].inverse(state["y"], state["z"], stream)
        return state["y"], state["z"]
    if op == "batch":
        lib.ntt_batch_submit(state["jobs"], stream)
        return state["outs"]
    if op == "quotient":
        plan, y = state["plan"], state["y"]
        for a, b in zip(state["x"], y):
            plan.coset_forward(a, b, stream)
        lib.ntt_pointwise_quotient(case["field"], y[0], y[1], y[2], state["z"], state["q"], state["q"].shape[0], stream)
        return plan.coset_inverse(state["q"], state["q"], stream)
    if op == "host":
        lib.ntt_transform_host(state["plan"].handle, case["kind"], state["x"], state["y"], state["work"], stream)
        return state["y"]
    if op == "msm":
        return state["plan"].execute(state["s"], state["p"], stream=stream)
    if op == "commit":
        state["plan"].inverse(state["x"], state["y"], stream)
        return state["y"], state["msm"].execute_bases(state["y"], stream=stream)
    native.ntt_wide_transform(case["field"], case["kind"], case["log_n"], state["x"], state["y"], stream)
    return state["y"]


# -------------------------------------------------------------------- work


def _transform_work(words, log_n, kind="forward"):
    """Each element in and out once; N/2 log N butterflies and one factor per
    element, a Montgomery product of L 32-bit limbs being 2 L^2 multiply-adds."""
    n, limbs = 1 << log_n, 2 * words
    products = n // 2 * log_n + (0 if kind == "forward" else n)
    return 2 * n * 8 * words, 2 * 2 * limbs * limbs * products


def _msm_work(curve, n, points_read=True):
    """Scalars and points once; 10 products per point and window of about log2 n - 3 bits."""
    field, _, _, words = CURVES[curve]
    limbs = 2 * words
    window = max(4, int(math.log2(n)) - 3)
    count = -(-(FIELDS[field][0].bit_length() + 1) // window)
    return n * (32 + (16 * words if points_read else 0)), 2 * 2 * limbs * limbs * 10 * n * count


def work(case):
    op = case["op"]
    if op in ("transform", "host", "wide"):
        b, f = _transform_work(FIELDS[case["field"]][1], case["log_n"], case["kind"])
    elif op == "step":
        b, f = (2 * v for v in _transform_work(4, case["log_n"]))
    elif op == "batch":
        parts = [_transform_work(4, log_n, kind) for _, log_n, kind in _batch_jobs(case)]
        b, f = sum(v[0] for v in parts), sum(v[1] for v in parts)
    elif op == "quotient":
        # three transforms in, the pointwise step, one transform back: 3 vectors read, 1 written
        _, f = _transform_work(4, case["log_n"] + 2, "coset")
        m = 4 << case["log_n"]
        b, f = 4 * 32 * m, 4 * f + 2 * 320 * m
    elif op == "msm":
        b, f = _msm_work(case["curve"], case["n"])
    else:
        b, f = _transform_work(4, case["log_n"], "inverse")
        b2, f2 = _msm_work(case["curve"], 1 << case["log_n"])
        b, f = b + b2, f + f2
    return {"bytes": b, "flops": f}


# ---------------------------------------------- the same by Python integers


def _ints(x):
    a = x.cpu().numpy()
    raw, size = np.ascontiguousarray(a).tobytes(), a.shape[1] * 8
    return [int.from_bytes(raw[i:i + size], "little") for i in range(0, len(raw), size)]


def _limbs(values, words):
    raw = b"".join(v.to_bytes(8 * words, "little") for v in values)
    return np.frombuffer(raw, dtype=np.int64).reshape(-1, words).copy()


def _dft(x, w, p):
    """sum_n x_n w^(k n) by halving."""
    n = len(x)
    if n == 1:
        return x
    even, odd = _dft(x[0::2], w * w % p, p), _dft(x[1::2], w * w % p, p)
    top, low, t = [0] * (n // 2), [0] * (n // 2), 1
    for k in range(n // 2):
        v = t * odd[k]
        top[k], low[k] = (even[k] + v) % p, (even[k] - v) % p
        t = t * w % p
    return top + low


def _transform(field, kind, x):
    p, _, gen = FIELDS[field]
    n = len(x)
    w = pow(gen, (p - 1) // n, p)
    if kind in ("forward", "coset"):
        if kind == "coset":
            x = [v * pow(gen, i, p) % p for i, v in enumerate(x)]
        return _dft(x, w, p)
    n_inv, s = pow(n, -1, p), pow(gen, -1, p) if kind == "coset_inverse" else 1
    return [v * n_inv * pow(s, i, p) % p for i, v in enumerate(_dft(x, pow(w, -1, p), p))]


def _multiple(curve, k):
    """k G, affine, by doubling and adding."""
    _, q, g, _ = CURVES[curve]

    def add(a, b):
        if a is None or b is None:
            return a or b
        if a[0] == b[0]:
            if (a[1] + b[1]) % q == 0:
                return None
            m = 3 * a[0] * a[0] * pow(2 * a[1], -1, q) % q
        else:
            m = (b[1] - a[1]) * pow(b[0] - a[0], -1, q) % q
        x = (m * m - a[0] - b[0]) % q
        return x, (m * (a[0] - x) - a[1]) % q

    acc = None
    for bit in bin(k)[2:]:
        acc = add(acc, acc)
        if bit == "1":
            acc = add(acc, g)
    return acc or (0, 0)


def _sum_point(curve, scalars, ts):
    """sum s (t G) = (sum s t) G."""
    field, _, _, words = CURVES[curve]
    r = FIELDS[field][0]
    return _limbs(_multiple(curve, sum(s * t for s, t in zip(scalars, ts)) % r), words).reshape(-1)


def exact(case, seed):
    op = case["op"]
    if op in ("transform", "step", "host", "wide"):
        if case["log_n"] > 17:
            return None
        field = case["field"]
        x = _ints(_elements(field, 1 << case["log_n"], seed))
        words = FIELDS[field][1]
        if op == "step":
            return _limbs(_transform(field, "forward", x), words), _limbs(x, words)
        return _limbs(_transform(field, case["kind"], x), words)
    if op == "msm" and case["n"] <= 1 << 20:
        field = CURVES[case["curve"]][0]
        return _sum_point(case["curve"], _ints(_scalars(case, field, case["n"], seed)),
                          _ints(_elements(field, case["n"], seed + 1)))
    if op == "commit" and case["log_n"] <= 16:
        field, n = CURVES[case["curve"]][0], 1 << case["log_n"]
        coeffs = _transform(field, "inverse", _ints(_elements(field, n, seed)))
        return _limbs(coeffs, 4), _sum_point(case["curve"], coeffs, _ints(_elements(field, n, seed + 1)))
    return None
