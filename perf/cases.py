"""Timed cases: what programs built on the library ask of it, through its
public entry points.

Positions and widths are those of the repository's own workloads
(paper_2507_06579_gb300/workloads.py, sweep.py, bench.py): single membership
queries, ranges from 10^3 to 10^9 wide between 5 and 2^44, the 2^24-blocks of
the pi_E(x) sweep with and without classes and over the primes alone, the
batch of uneven intervals, and a burst of serving requests.  The seed moves
the ranges (or draws the queries), so other seeds are other inputs of the same
cost.  Every output is a whole number: flags, classes, counts.

A program keeps one context for its lifetime, and tunes it once when it runs
large batches; so do these cases (one plain and one tuned context a process).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2507_06579_gb300 as E
from paper_2507_06579_gb300 import sweep, workloads

D_LIMIT = E.EIS_D_LIMIT
BLOCK = 1 << 24  # the sweep's block of d

_contexts = {}


def _context(tuned):
    """The process's context; tuned: with the per-decade settings timed once,
    as a program does at start-up."""
    if tuned not in _contexts:
        ctx = E.Context(0)
        if tuned:
            ctx.autotune_decades(10**6, 10**12)
        _contexts[tuned] = ctx
    return _contexts[tuned]


def listed():
    return [
        # the smallest calls: is this d in E?  A program that asks one d at a
        # time, d of the serving configuration's range (below 10^12) ...
        {"name": "queries below 1e12", "kind": "queries", "hi": 10**12, "n": 32},
        # ... and at the top of the supported range
        {"name": "queries below 2^44", "kind": "queries", "hi": D_LIMIT, "n": 16},
        # the small configuration: every candidate of a range of width 10^6 at
        # the low end, one byte each, into host memory
        {"name": "codes 1e6", "kind": "codes", "lo": 5, "width": 10**6},
        # an ordinary range call: a ragged window near 10^11, both bitmaps into
        # device tensors
        {"name": "classify 1e7 at 1e11", "kind": "classify", "lo": 10**11, "width": 10**7 + 3003,
         "tuned": False},
        # a Table 1 interval: length 10^8 below 10^10
        {"name": "classify 1e8 at 1e10", "kind": "classify", "lo": 99 * 10**8, "width": 10**8,
         "tuned": True},
        # the benchmark's window, length 10^9 below 10^11, in a tuned context
        {"name": "classify 1e9 at 1e11", "kind": "classify", "lo": 10**11 - 10**9, "width": 10**9,
         "tuned": True},
        # a range at the top of the supported d (the corrected quotient)
        {"name": "classify 2e6 below 2^44", "kind": "classify", "lo": D_LIMIT - 3 * 10**6,
         "width": 2 * 10**6 + 17, "tuned": False},
        # the class of eps_d in F_4* for every d of a window
        {"name": "classes 1e7 at 1e10", "kind": "log", "lo": 10**10, "width": 10**7},
        # a plan kept and launched again: [5, 10^9] as the sweep's blocks
        {"name": "plan of blocks to 1e9", "kind": "plan", "lo": 5, "blocks": 60},
        # the sweep's own step: one batch of blocks with the class counts
        {"name": "sweep 16 blocks at 9e10", "kind": "sweep", "lo": 9 * 10**10, "blocks": 16,
         "primes": False, "classes": True},
        # the serving loop when 2000 requests of the serving mix (90% range
        # counts, 10% membership queries) arrive at once
        {"name": "burst of 2000 requests", "kind": "serve", "n": 2000},
        # the batch of uneven intervals, counted in one call
        {"name": "batch of 4096 intervals", "kind": "batch", "n": 4096, "len_max": 10**7},
    ]


def _log(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def _width(rng, lo, least, most, seconds):
    """A width between least and most whose walk from lo takes at most about
    `seconds` (a tenth of the d are walked, about 0.07 sqrt(d) steps each, at
    2.5e12 steps a second)."""
    cap = seconds * 2.5e12 / (0.1 * 0.07 * math.sqrt(lo))
    return _log(rng, least, max(least + 1, min(most, cap)))


def draw(rng):
    kind = rng.choice(["queries", "codes", "classify", "classify", "log", "plan", "sweep", "batch",
                       "serve"])
    if kind == "queries":
        return {"kind": kind, "hi": _log(rng, 10**9, D_LIMIT), "n": rng.randint(8, 48)}
    if kind == "plan":
        return {"kind": kind, "lo": _log(rng, 5, 10**10), "blocks": rng.randint(2, 60)}
    if kind == "sweep":
        lo = _log(rng, 10**8, 10**11)
        return {"kind": kind, "lo": lo, "blocks": rng.randint(2, 16), "primes": rng.random() < 0.3,
                "classes": rng.random() < 0.5}
    if kind == "serve":
        return {"kind": kind, "n": _log(rng, 50, 4000)}
    if kind == "batch":
        return {"kind": kind, "n": _log(rng, 64, 4096), "len_max": _log(rng, 10**4, 10**7)}
    lo = _log(rng, 10**6, 16 * 10**12)
    if kind == "codes":
        return {"kind": kind, "lo": lo, "width": _width(rng, lo, 10**3, 10**8, 0.3)}
    if kind == "log":
        return {"kind": kind, "lo": lo, "width": _width(rng, lo, 10**4, 10**8, 0.3)}
    tuned = rng.random() < 0.5
    return {"kind": kind, "lo": lo, "width": _width(rng, lo, 10**3, 10**9, 0.5), "tuned": tuned}


def _in_D(d):
    """d square-free (d == 5 mod 8), by trial division with odd p."""
    p = np.arange(3, math.isqrt(d) + 1, 2, dtype=np.int64)
    return not bool(np.any(d % (p * p) == 0))


def _moved(case, seed):
    """[lo, hi) of the case, its place moved by the seed by at most a tenth of
    its width (never above 2^44)."""
    lo, width = case["lo"], case["width"]
    r = np.random.default_rng(seed)
    step = max(8, width // 10)
    lo = lo + int(r.integers(0, step))
    lo = max(0, min(lo, D_LIMIT - width))
    return lo, lo + width


def prepare(case, seed):
    kind = case["kind"]
    r = np.random.default_rng(seed)
    state = {"kind": kind, "ctx": _context(bool(case.get("tuned", kind == "batch")))}
    if kind == "queries":
        ds = []
        while len(ds) < case["n"]:
            d = int(r.integers(1, case["hi"] // 8)) * 8 + 5
            if d < case["hi"] and _in_D(d):
                ds.append(d)
        state["ds"] = ds
    elif kind == "plan":
        lo = case["lo"] + int(r.integers(0, BLOCK))
        blocks = [(lo + i * BLOCK, lo + (i + 1) * BLOCK) for i in range(case["blocks"])]
        state["plan"] = state["ctx"].plan_create([a for a, _ in blocks], [b for _, b in blocks])
    elif kind == "sweep":
        lo = case["lo"] + int(r.integers(0, BLOCK))
        state["chunk"] = [(lo + i * BLOCK, lo + (i + 1) * BLOCK) for i in range(case["blocks"])]
        state["count"] = sweep.gpu_counter(state["ctx"], case["primes"], case["classes"])
    elif kind == "serve":
        stream = workloads.serving_stream(case["n"], 1e4, seed=seed)
        state["server"] = E.Server(state["ctx"])
        state["requests"] = ([0.0] * len(stream),
                             [E.EIS_REQ_MEMBER if k == "member" else E.EIS_REQ_COUNT
                              for _, k, _, _ in stream],
                             [a for _, _, a, _ in stream], [b for _, _, _, b in stream])
    elif kind == "batch":
        state["lo"], state["hi"] = workloads.batched_intervals(
            n=case["n"], seed=seed, len_range=(1e3, float(case["len_max"])))
    else:
        state["lo"], state["hi"] = _moved(case, seed)
        if kind == "classify":
            n, _ = E.num_candidates(state["lo"], state["hi"])
            state["flags"] = torch.empty((n + 31) // 32, dtype=torch.int32, device="cuda")
            state["sqfree"] = torch.empty_like(state["flags"])
    return state


def run(state):
    ctx, kind = state["ctx"], state["kind"]
    if kind == "queries":
        return np.array([ctx.is_eisenstein(d) for d in state["ds"]])
    if kind == "codes":
        return list(ctx.classify_range_u8(state["lo"], state["hi"]))
    if kind == "classify":
        return list(ctx.classify_range(state["lo"], state["hi"], state["flags"], state["sqfree"]))
    if kind == "log":
        return ctx.classify_range_log(state["lo"], state["hi"])
    if kind == "plan":
        state["plan"].launch()
        return [state["plan"].counts(), state["plan"].counts_D()]
    if kind == "sweep":
        rows = state["count"](state["chunk"])
        # (#D, #E) per block, then the class counts per block
        return [np.array([row[:2] for row in rows]), np.array([row[2] for row in rows if len(row) > 2])]
    if kind == "serve":
        got = state["server"].replay(*state["requests"])
        return [got["results"], got["status"]]
    return ctx.count_batch(state["lo"], state["hi"])


def work(case):
    """Bytes of one pass: the ends of every range (or the queried d) in, the
    flags, classes and counts out.  (The rest is integer work of which no
    least number is known.)"""
    kind = case["kind"]
    if kind == "queries":
        return {"bytes": 9 * case["n"], "flops": 0}
    if kind == "plan":
        return {"bytes": 32 * case["blocks"], "flops": 0}
    if kind == "sweep":
        return {"bytes": (32 + 24 * case["classes"]) * case["blocks"], "flops": 0}
    if kind in ("batch", "serve"):
        return {"bytes": 24 * case["n"], "flops": 0}
    n = case["width"] / 8
    return {"bytes": 16 + (n / 4 if kind == "classify" else n), "flops": 0}


def exact(case, seed):
    """codes of a short range at the low end by walking the continued fraction
    of (1 + sqrt d)/2 over whole periods in 64-bit integers: the generator of
    the unit as (x, y) with x + y omega mod 2, omega^2 = omega + 1."""
    if case["kind"] != "codes" or case["lo"] + case["width"] > 2 * 10**6:
        return None
    lo, hi = _moved(case, seed)
    d = np.arange(lo + (13 - lo % 8) % 8, hi, 8, dtype=np.int64)
    codes = np.ones(len(d), dtype=np.uint8)
    for k in range(3, math.isqrt(hi) + 1, 2):
        codes[d % (k * k) == 0] = 0
    live = np.flatnonzero(codes)
    dd = d[live]
    s = np.sqrt(dd.astype(np.float64)).astype(np.int64)
    s -= s * s > dd
    s += (s + 1) * (s + 1) <= dd
    P, Q = np.ones_like(dd), np.full_like(dd, 2)
    x, y = np.ones_like(dd), np.zeros_like(dd)
    while len(live):
        P = (P + s) // Q * Q - P
        # times (P + sqrt d)/2 = (P - 1)/2 + omega; Q/2 is odd
        u = (P - 1) // 2 % 2
        x, y = (u * x + y) % 2, (x + u * y + y) % 2
        Q = (dd - P * P) // Q
        end = Q == 2
        codes[live[end & (x == 1) & (y == 0)]] = 2
        live, dd, s, P, Q, x, y = (v[~end] for v in (live, dd, s, P, Q, x, y))
    return [codes, int((codes == 2).sum())]
