"""Workloads of the library as its users call it, for timing and comparison.

Every case goes through the public Python entry points and covers one of:

    modp      Low(A A^T) mod p, device buffers (``aat_modp``)
    gemm      X Y^T mod p (``aat_gemm_modp``)
    quat      quaternion M M^H mod p (``aah_quat_modp``)
    host      Low(A A^T) mod p from and to pinned host memory
    aah       Low(A A^H) over C (``aah_complex``)
    aatc      Low(A A^T) over C by Algorithm 1 (``aat_complex``)
    batch     many uneven products in one plan (``Plan``)

Results are written into buffers that the caller keeps, as a program that
calls the library repeatedly does.  The F_p calls ask for a zero strict upper
triangle (``AAT_ZERO_UPPER``), so that every entry of every output is defined.
"""
from __future__ import annotations

import math
import random

import torch

import paper_2101_01025_gb300 as aat

M31 = 2**31 - 1
#: The primes of the workloads: two digits with pair sums, two digits without,
#: three digits, four digits; both kinds of Y and a = 1 (p = 3 mod 8).
PRIMES = (65521, 131071, 1000003, 2147483587, M31)


def listed():
    return [
        # one small product of a larger program: launch and host latency
        {"name": "modp_96x160", "kind": "modp", "n": 96, "k": 160, "p": 65521},
        # the smallest workload of the method's own experiments, one level of
        # the recursion with the 2 x 2 skew-orthogonal Y
        {"name": "modp_512_level1", "kind": "modp", "n": 512, "k": 512, "p": 131071, "levels": 1},
        # an ordinary odd-sized product over a word-size prime
        {"name": "modp_1001x3001", "kind": "modp", "n": 1001, "k": 3001, "p": M31},
        # large products over 16- and 17-bit primes
        {"name": "modp_8192_p65521", "kind": "modp", "n": 8192, "k": 8192, "p": 65521},
        {"name": "modp_16384x4096_p131071", "kind": "modp", "n": 16384, "k": 4096, "p": 131071},
        # the headline size over the largest Mersenne prime below 2^31,
        # balanced residues
        {"name": "modp_16384", "kind": "modp", "n": 16384, "k": 16384, "p": M31,
         "balanced": True},
        # a general product of ragged sizes
        {"name": "gemm_2500x4001x3003", "kind": "gemm", "m": 2500, "n": 4001, "k": 3003, "p": M31},
        # quaternion matrices (five general products and a symmetric one)
        {"name": "quat_2048x1500", "kind": "quat", "n": 2048, "k": 1500, "p": 65521},
        # data that starts and ends in host memory
        {"name": "host_6000x5000", "kind": "host", "n": 6000, "k": 5000, "p": M31},
        # complex products, FP32 accuracy class and the two-piece class
        {"name": "aah_8192_fp32", "kind": "aah", "n": 8192, "k": 8192, "prec": "fp32"},
        {"name": "aatc_3000x5001_bf16x3", "kind": "aatc", "n": 3000, "k": 5001, "prec": "bf16x3"},
        # 256 F_p and 64 complex products of uneven sizes in one plan
        {"name": "batch_256_64", "kind": "batch", "fp": 256, "cplx": 64, "p": 65521,
         "n_hi": 2048, "k_hi": 4096, "sizes": 5},
    ]


def _log_int(rng, lo, hi):
    return int(min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def draw(rng):
    kind = rng.choice(["modp", "modp", "modp", "gemm", "quat", "host", "aah", "aatc", "batch"])
    if kind == "modp":
        c = {"kind": kind, "n": _log_int(rng, 64, 16384), "k": _log_int(rng, 64, 16384),
             "p": rng.choice(PRIMES), "balanced": rng.random() < 0.5}
        if c["n"] <= 4096 and rng.random() < 0.3:
            c["levels"] = rng.choice([0, 1, 2])
        return c
    if kind == "gemm":
        return {"kind": kind, "m": _log_int(rng, 64, 8192), "n": _log_int(rng, 64, 8192),
                "k": _log_int(rng, 64, 8192), "p": rng.choice(PRIMES)}
    if kind == "quat":
        return {"kind": kind, "n": _log_int(rng, 64, 4096), "k": _log_int(rng, 64, 4096),
                "p": rng.choice(PRIMES)}
    if kind == "host":
        return {"kind": kind, "n": _log_int(rng, 64, 8192), "k": _log_int(rng, 64, 8192),
                "p": rng.choice(PRIMES)}
    if kind in ("aah", "aatc"):
        return {"kind": kind, "n": _log_int(rng, 64, 8192), "k": _log_int(rng, 64, 8192),
                "prec": rng.choice(["fp32", "bf16x3"])}
    return {"kind": kind, "fp": rng.choice([16, 64, 256]), "cplx": rng.choice([8, 24, 64]),
            "p": rng.choice(PRIMES), "n_hi": rng.choice([512, 1024, 2048]),
            "k_hi": rng.choice([1024, 2048, 4096]), "sizes": rng.randrange(1 << 30)}


# ------------------------------------------------------------------ inputs

_PREC = {"fp32": aat.AAT_C_FP32, "bf16x3": aat.AAT_C_BF16X3}


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _residues(g, shape, p, balanced=False):
    x = torch.randint(0, p, shape, dtype=torch.int32, device="cuda", generator=g)
    if balanced:
        x = torch.where(x > p // 2, x - p, x)
    return x


def _normal(g, shape):
    return torch.randn(shape, dtype=torch.complex64, device="cuda", generator=g)


def _zeros(n, dtype=torch.int32):
    return torch.zeros((n, n), dtype=dtype, device="cuda")


def _batch_sizes(case):
    """(n, k) per problem, log-uniform: F_p problems first, then complex."""
    rng = random.Random(case["sizes"])
    return [(_log_int(rng, 64, case["n_hi"]), _log_int(rng, 64, case["k_hi"]))
            for _ in range(case["fp"] + case["cplx"])]


def _flat_results(case, cplx=torch.complex64):
    """The batch's zeroed results: one buffer for the F_p problems and one for
    the complex ones, each result in them at a multiple of 256 bytes."""
    sizes = [n for n, _ in _batch_sizes(case)]
    bufs, views = [], []
    for ns, dtype in ((sizes[:case["fp"]], torch.int32), (sizes[case["fp"]:], cplx)):
        room = [(n * n + 63) // 64 * 64 for n in ns]
        buf = torch.zeros(sum(room), dtype=dtype, device="cuda")
        off = 0
        for n, r in zip(ns, room):
            views.append(buf[off:off + n * n].view(n, n))
            off += r
        bufs.append(buf)
    return bufs, views


def _inputs(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "modp":
        return [_residues(g, (case["n"], case["k"]), case["p"], case.get("balanced", False))]
    if kind == "gemm":
        return [_residues(g, (case["m"], case["k"]), case["p"]),
                _residues(g, (case["n"], case["k"]), case["p"])]
    if kind == "quat":
        return [_residues(g, (case["n"], case["k"]), case["p"]) for _ in range(4)]
    if kind == "host":
        return [_residues(g, (case["n"], case["k"]), case["p"])]
    if kind in ("aah", "aatc"):
        return [_normal(g, (case["n"], case["k"]))]
    return [_residues(g, s, case["p"]) if i < case["fp"] else _normal(g, s)
            for i, s in enumerate(_batch_sizes(case))]


def prepare(case, seed):
    kind = case["kind"]
    x = _inputs(case, seed)
    st = {"case": case, "x": x}
    if kind == "modp":
        st["c"] = _zeros(case["n"])
    elif kind == "gemm":
        st["c"] = torch.zeros((case["m"], case["n"]), dtype=torch.int32, device="cuda")
    elif kind == "quat":
        st["c"] = tuple(_zeros(case["n"]) for _ in range(4))
    elif kind == "host":
        a = torch.empty(x[0].shape, dtype=torch.int32, pin_memory=True)
        a.copy_(x[0])
        st["x"] = [a]
        st["c"] = torch.zeros((case["n"], case["n"]), dtype=torch.int32, pin_memory=True)
    elif kind in ("aah", "aatc"):
        st["c"] = _zeros(case["n"], torch.complex64)
    else:
        # the plan writes lower triangles only
        st["c"], views = _flat_results(case)
        st["plan"] = aat.Plan([("modp", a, c, case["p"], 0) if i < case["fp"]
                               else ("aah", a, c, 0, aat.AAT_C_FP32)
                               for i, (a, c) in enumerate(zip(x, views))])
    return st


def run(state):
    case, x, c = state["case"], state["x"], state["c"]
    kind = case["kind"]
    if kind == "modp":
        return aat.aat_modp(x[0], case["p"], C=c, flags=aat.AAT_ZERO_UPPER,
                            levels=case.get("levels"))
    if kind == "gemm":
        return aat.aat_gemm_modp(x[0], x[1], case["p"], C=c)
    if kind == "quat":
        return aat.aah_quat_modp(*x, case["p"], H=c, flags=aat.AAT_ZERO_UPPER)
    if kind == "host":
        return aat.aat_modp_host(x[0], case["p"], C=c, flags=aat.AAT_ZERO_UPPER)
    if kind == "aah":
        return aat.aah_complex(x[0], C=c, flags=_PREC[case["prec"]])
    if kind == "aatc":
        # the recursion uses the strict upper triangle as scratch
        return aat.aat_complex(x[0], C=c, flags=_PREC[case["prec"]]).tril_()
    state["plan"].execute()
    return c


# -------------------------------------------------------------- compulsory work

def _low(n, k, elem, mac):
    """Low(A A^*), n x k: A once, the n x n result once; n (n + 1) / 2 entries."""
    return elem * (n * k + n * n), mac * (n * (n + 1) // 2) * k


def work(case):
    kind = case["kind"]
    if kind in ("modp", "host"):
        b, f = _low(case["n"], case["k"], 4, 2)
    elif kind == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        b, f = 4 * (m * k + n * k + m * n), 2 * m * n * k
    elif kind == "quat":
        n, k = case["n"], case["k"]
        b, f = 16 * (n * k + n * n), 5 * 2 * n * n * k + n * (n + 1) * k
    elif kind in ("aah", "aatc"):
        # two real products: one of n^2 k, one symmetric, multiply-adds
        n, k = case["n"], case["k"]
        b, f = 8 * n * k + 4 * n * (n + 1), 2 * n * n * k + n * (n + 1) * k
    else:
        b = f = 0
        for i, (n, k) in enumerate(_batch_sizes(case)):
            if i < case["fp"]:
                b += 4 * n * k + 2 * n * (n + 1)
                f += n * (n + 1) * k
            else:
                b += 8 * n * k + 4 * n * (n + 1)
                f += 2 * n * n * k + n * (n + 1) * k
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------ 64-bit values

def _mul_mod(x, y, p):
    """x y^T mod p, int64 in [0, p): FP64 products of 16-bit halves, whose
    sums stay below 2^53 (|x| < p < 2^31, at most 2^20 terms)."""
    def halves(t):
        lo = torch.remainder(t, 65536)
        return lo.double(), torch.div(t - lo, 65536, rounding_mode="floor").double()

    def dot(a, b):
        return torch.remainder((a @ b.T).to(torch.int64), p)

    if p < 1 << 17:
        return dot(x.double(), y.double())
    (xl, xh), (yl, yh) = halves(x.to(torch.int64)), halves(y.to(torch.int64))
    mid = dot(xl, yh) + dot(xh, yl)
    return torch.remainder(dot(xh, yh) * ((1 << 32) % p) + torch.remainder(mid, p) * 65536
                           + dot(xl, yl), p)


def _quat_mod(a, b, c, d, p):
    """Hamilton product of M = a + b i + c j + d k with its conjugate transpose."""
    def m(x, y):
        return _mul_mod(x, y, p)
    h1 = m(a, a) + m(b, b) + m(c, c) + m(d, d)
    h2 = m(b, a) - m(a, b) + m(d, c) - m(c, d)
    h3 = m(c, a) - m(a, c) + m(b, d) - m(d, b)
    h4 = m(d, a) - m(a, d) + m(c, b) - m(b, c)
    return tuple(torch.remainder(h, p).tril() for h in (h1, h2, h3, h4))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("modp", "host") and (
            case["n"] ** 2 * case["k"] * (1 if case["p"] < 1 << 17 else 4) > 8e12):
        return None  # over 15 seconds of FP64 products
    x = _inputs(case, seed)
    if kind == "modp":
        return _mul_mod(x[0], x[0], case["p"]).tril()
    if kind == "gemm":
        return _mul_mod(x[0], x[1], case["p"])
    if kind == "quat":
        return _quat_mod(*x, case["p"])
    if kind == "host":
        return _mul_mod(x[0], x[0], case["p"]).tril().cpu()
    if kind == "aah":
        z = x[0].to(torch.complex128)
        return (z @ z.conj().T).tril()
    if kind == "aatc":
        z = x[0].to(torch.complex128)
        return (z @ z.T).tril()
    bufs, views = _flat_results(case, torch.complex128)
    for i, (t, c) in enumerate(zip(x, views)):
        if i < case["fp"]:
            c.copy_(_mul_mod(t, t, case["p"]).tril())
        else:
            z = t.to(torch.complex128)
            c.copy_((z @ z.conj().T).tril())
    return bufs
