"""Performance cases: the calls a user of the library makes, over the sizes and
magnitudes they are made at.

A case is a dict of plain values; ``kind`` names the entry point:

* ``range``: ``Context.verify_range`` over ``n`` even numbers from about
  ``lo``.  ``out`` is what the caller asks for: "hist" the merged histogram
  (a unit of the journaled command line, ``run.py``), "rows" per-segment
  records and histogram rows, "pmin" the p_min array in device memory;
* ``batch``: ``Context.verify_batch`` over ``count`` ranges, lengths
  log-uniform in [2^lmin, 2^lmax] even n, starts uniform in [smin, smax];
* ``queries``: ``Context.query`` (``count`` 1) or ``Context.query_batch``
  on uniform even n below ``top``;
* ``partitions``: ``Context.partitions`` of ``n`` even numbers from about ``lo``;
* ``sieve``: ``Context.sieve_segment`` of ``bits`` odd numbers from about ``lo``
  into device memory.

The seed moves a case's first number (or draws its ranges and queries); its
sizes are the case's own.
"""
import math
import random

import numpy as np
import torch

from paper_2603_02621_gb300 import gb, workloads

P1, P2 = 1 << 15, 1 << 20


def listed():
    return [
        # one p_min(n) asked for by itself: launches and latency alone
        dict(name="query_one", kind="queries", count=1, top=4 * 10**18),
        # a batch of single-number queries, as a server's query lane collects them
        dict(name="queries_4096", kind="queries", count=4096, top=4 * 10**18),
        # the shortest range a server is asked for, at an ordinary offset
        dict(name="range_64k_at_1e15", kind="range", lo=10**15, n=1 << 16, seg=1 << 24, p1=P1, p2=P2, out="hist"),
        # every p_min below 10^7, kept per n (the smallest exhaustive table)
        dict(name="pmin_to_1e7", kind="range", lo=4, n=4999999, seg=1 << 24, p1=1 << 16, p2=0, out="pmin"),
        # [4, 10^10] with per-segment outputs
        dict(name="range_to_1e10", kind="range", lo=4, n=4999999999, seg=1 << 24, p1=P1, p2=P2, out="rows"),
        # the headline: every even n to 10^12
        dict(name="range_to_1e12", kind="range", lo=4, n=499999999999, seg=1 << 27, p1=P1, p2=P2, out="hist"),
        # one journaled unit of a long verification in the middle of the range
        dict(name="unit_at_1e15", kind="range", lo=10**15, n=1 << 32, seg=1 << 27, p1=P1, p2=P2, out="hist"),
        # a 10^11-wide window at the frontier of published verifications
        dict(name="window_at_4e18", kind="range", lo=4 * 10**18 - 2 * 10**11, n=5 * 10**10, seg=1 << 27, p1=P1, p2=P2,
             out="hist"),
        # thousands of uneven ranges in one call
        dict(name="batch_4096", kind="batch", count=4096, lmin=10, lmax=26, smin=10**9, smax=10**15, base=32 * 10**6),
        # what a serving lane admits at once: ranges of 2^16 .. 2^30 n up to 4e18
        dict(name="batch_serving", kind="batch", count=24, lmin=16, lmax=30, smin=10**9, smax=4 * 10**18,
             base=2 * 10**9 + 10**6),
        # a prime bitset for the caller's own use; an odd length
        dict(name="sieve_window", kind="sieve", lo=10**13 + 1, bits=(1 << 30) + 12345),
        # partition counts of a run of numbers near 10^9
        dict(name="partitions_1e9", kind="partitions", lo=10**9, n=2000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["range", "range", "range", "range", "batch", "batch", "queries", "partitions", "sieve"])
    if kind == "range":
        out = rng.choice(["hist", "hist", "rows", "pmin"])
        lo = 4 if rng.random() < 0.25 else _log(rng, 10**4, 39 * 10**17) // 2 * 2
        top = 1 << (26 if out == "pmin" else 34)
        n = _log(rng, 1000, top)
        seg = rng.choice([1 << 20, 1 << 24, 1 << 27]) if n > 1 << 20 else 1 << 24
        if out == "rows":
            seg = max(seg, 1 << 24)
        return dict(kind="range", lo=lo, n=n, seg=seg, p1=rng.choice([1 << 13, P1, 1 << 16]),
                    p2=P2 if rng.random() < 0.8 else 0, out=out)
    if kind == "batch":
        lmax = rng.randint(14, 26)
        top = _log(rng, 10**10, 4 * 10**18)
        count = _log(rng, 1, 4096) if top < 10**16 else _log(rng, 1, 32)
        return dict(kind="batch", count=count, lmin=10, lmax=lmax, smin=10**9, smax=top, base=math.isqrt(top) + 10**5)
    if kind == "queries":
        return dict(kind="queries", count=_log(rng, 1, 8192), top=_log(rng, 10**6, 9 * 10**18))
    if kind == "partitions":
        return dict(kind="partitions", lo=_log(rng, 10**4, 4 * 10**9) // 2 * 2, n=_log(rng, 1, 3000))
    return dict(kind="sieve", lo=_log(rng, 10**3, 10**15) | 1, bits=_log(rng, 10**4, 1 << 31))


def _start(case, rng):
    """The case's first number: its lo, moved by the seed by at most a few
    millionths of where it lies (from 4 on by at most 2000)."""
    return case["lo"] + 2 * rng.randrange(1, 1000 + case["lo"] // 10**7)


def _ranges(case, seed):
    return workloads.batched_ranges(case["count"], seed=seed + 1, log2_min=case["lmin"], log2_max=case["lmax"],
                                    start_min=case["smin"], start_max=case["smax"])


def _numbers(case, seed):
    rng = random.Random(seed)
    return [rng.randrange(4, case["top"]) // 2 * 2 for _ in range(case["count"])]


def prepare(case, seed):
    kind = case["kind"]
    rng = random.Random(seed)
    stream = torch.cuda.current_stream().cuda_stream
    st = dict(case=case)
    if kind == "range":
        lo = _start(case, rng)
        hi = lo + 2 * case["n"]
        base = max(1 << 16, math.isqrt(hi + 2 * P2) + 4096)
        st.update(lo=lo, hi=hi, ctx=gb.Context(device=0, base_limit=base, seg_len=case["seg"], p1=case["p1"],
                                               p2=case["p2"], stream=stream))
        final = max(case["p1"], case["p2"])
        st["hist_len"] = st["ctx"].prime_pi(final)
        if case["out"] == "pmin":
            st["pmin"] = torch.zeros(case["n"], dtype=torch.int32, device="cuda")
    elif kind == "batch":
        # records (six 64-bit words each) and histogram rows stay in device memory
        st.update(ranges=_ranges(case, seed),
                  records=torch.zeros((case["count"], 6), dtype=torch.int64, device="cuda"),
                  hist=torch.zeros((case["count"], 3512), dtype=torch.int64, device="cuda"),
                  ctx=gb.Context(device=0, base_limit=case["base"], p1=P1, p2=P2, stream=stream))
    elif kind == "queries":
        ns = _numbers(case, seed)
        st.update(ns=ns[0] if len(ns) == 1 else np.array(ns, dtype=np.uint64),
                  ctx=gb.Context(device=0, base_limit=1 << 20, p1=P1, p2=P2, stream=stream))
    elif kind == "partitions":
        lo = _start(case, rng)
        hi = lo + 2 * case["n"]
        st.update(lo=lo, hi=hi, ctx=gb.Context(device=0, base_limit=1 << 17, stream=stream))
    else:
        lo = _start(case, rng)
        base = max(1 << 16, math.isqrt(lo + 2 * case["bits"]) + 4096)
        st.update(lo=lo, q=torch.zeros((case["bits"] + 63) // 64, dtype=torch.int64, device="cuda"),
                  ctx=gb.Context(device=0, base_limit=base, stream=stream))
    return st


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind == "range":
        if case["out"] == "rows":
            r = ctx.verify_range(state["lo"], state["hi"], segs=True, seg_hist_stride=3512, allow_erange=True)
            r["segs"] = np.array([list(seg.values()) for seg in r["segs"]], dtype=np.int64)
            r["seg_hist"] = r["seg_hist"].view(np.int64)
            return r
        if case["out"] == "pmin":
            r = ctx.verify_range(state["lo"], state["hi"], pmin=state["pmin"], hist_cap=state["hist_len"])
            r["pmin"] = state["pmin"]
        else:
            r = ctx.verify_range(state["lo"], state["hi"], hist_cap=state["hist_len"])
        r["hist"] = r["hist"].view(np.int64)
        return r
    if kind == "batch":
        r = ctx.verify_batch(state["ranges"], results=state["records"], hist=state["hist"], hist_stride=3512,
                             allow_erange=True)
        return dict(rc=r["rc"], records=state["records"], hist=state["hist"])
    if kind == "queries":
        return ctx.query(state["ns"]) if case["count"] == 1 else ctx.query_batch(state["ns"])
    if kind == "partitions":
        return ctx.partitions(state["lo"], state["hi"])
    return dict(count=ctx.sieve_segment(state["lo"], case["bits"], state["q"]), bits=state["q"])


def _sieve_ops(bits, top):
    """Strikes of a sieve of `bits` odd numbers below `top`: one per odd
    multiple m p, m coprime to 15, of the primes from 47 to sqrt(top)
    (Mertens: sum 1/p = ln ln sqrt(top) - ln ln 47), and one and per 32-bit
    word for the primes below."""
    r = max(48.0, math.sqrt(top))
    return bits * (8 / 15) * (math.log(math.log(r)) - math.log(math.log(47.0))) + bits / 32


def _cover_ops(n, top):
    """An or per 32 even numbers and prime until a word of them is full: about
    2.4 ln(top) primes (31 words' worth of survivors at rate 2 / ln(top))."""
    return n / 32 * 2.4 * math.log(top)


def work(case):
    """Bytes that come in or go out; integer operations for `flops` (the whole
    path is integer work): strikes of the sieve and word ors of the cover."""
    kind = case["kind"]
    if kind == "range":
        n, top = case["n"], case["lo"] + 2 * case["n"]
        out = 4 * n if case["out"] == "pmin" else 8 * 3512 * (-(-n // case["seg"]) if case["out"] == "rows" else 1)
        return dict(bytes=out, flops=_sieve_ops(n, top) + _cover_ops(n, top))
    if kind == "batch":
        mean = (2.0**case["lmax"] - 2.0**case["lmin"]) / (math.log(2.0) * (case["lmax"] - case["lmin"]))
        n = case["count"] * mean
        return dict(bytes=case["count"] * (16 + 48 + 8 * 3512),
                    flops=_sieve_ops(n, case["smax"]) + _cover_ops(n, case["smax"]))
    if kind == "queries":
        # a pre-sieve of some hundred partners, then about 8 strong tests of
        # 1.5 log2(n) modular products (some 20 integer operations each)
        return dict(bytes=12 * case["count"], flops=case["count"] * (1000 + 8 * 1.5 * math.log2(case["top"]) * 20))
    if kind == "partitions":
        n, top = case["n"], case["lo"] + 2 * case["n"]
        # every pair i <= m / 2 of each n, 32 to an and and a population count
        return dict(bytes=4 * n, flops=_sieve_ops(top / 2, top) + n * (top / 4 / 32) * 2)
    return dict(bytes=case["bits"] / 8, flops=_sieve_ops(case["bits"], case["lo"] + 2 * case["bits"]))


_BASES = (2, 3, 5, 7, 11, 13, 17, 19, 23, 29, 31, 37)


def _is_prime(q):
    if q < 2:
        return False
    for b in _BASES:
        if q % b == 0:
            return q == b
    d, s = q - 1, 0
    while d % 2 == 0:
        d, s = d // 2, s + 1
    for b in _BASES:
        y = pow(b, d, q)
        if y in (1, q - 1):
            continue
        for _ in range(s - 1):
            y = y * y % q
            if y == q - 1:
                break
        else:
            return False
    return True


def _primes_to(limit):
    keep = np.ones(limit + 1, dtype=bool)
    keep[:2] = False
    for p in range(2, math.isqrt(limit) + 1):
        if keep[p]:
            keep[p * p::p] = False
    return np.flatnonzero(keep)


def exact(case, seed):
    """The values by their definitions, where that takes a few seconds."""
    if case["kind"] == "queries" and case["count"] <= 4096:
        primes = [int(p) for p in _primes_to(P1)]
        got = [next((p for p in primes if p < n and _is_prime(n - p)), 0) for n in _numbers(case, seed)]
        return got[0] if case["count"] == 1 else np.array(got, dtype=np.uint32)
    if case["kind"] == "partitions" and case["lo"] < 10**7:
        lo = _start(case, random.Random(seed))
        keep = np.zeros(lo + 2 * case["n"] + 1, dtype=bool)
        keep[_primes_to(lo + 2 * case["n"])] = True
        return np.array([np.count_nonzero(keep[:n // 2 + 1] & keep[n:n - n // 2 - 1:-1])
                         for n in range(lo, lo + 2 * case["n"], 2)], dtype=np.uint32)
    if case["kind"] == "sieve" and case["lo"] < 10**13 and case["bits"] <= 1 << 27:
        lo, bits = _start(case, random.Random(seed)), case["bits"]
        last = lo + 2 * (bits - 1)
        keep = np.ones((bits + 63) // 64 * 64, dtype=bool)
        keep[bits:] = False
        for p in _primes_to(math.isqrt(last))[1:]:
            first = max(int(p) * int(p), -(-lo // int(p)) * int(p))
            if first % 2 == 0:
                first += int(p)
            keep[(first - lo) // 2:bits:int(p)] = False
        words = torch.from_numpy(np.packbits(keep, bitorder="little").view(np.int64).copy())
        return dict(count=int(np.count_nonzero(keep)), bits=words)
    return None
