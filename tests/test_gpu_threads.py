"""Contexts sharing base primes, one host thread each, with calls of very
different sizes at the same time: a launch depends on its own call alone (the
limit of a kernel's dynamic shared memory is a property of the kernel on the
device, which the calls of all threads meet)."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def gbm():
    from paper_2603_02621_gb300 import gb
    gb.load()
    return gb


def _calls(gbm, kind, large):
    """(call, its result) pairs' makers of one size: every launcher whose shared
    memory depends on the call."""
    n = 2 * 10**8 if large else 1000
    lo = 10**12
    if kind == "range":
        return lambda g: g.verify_range(lo, lo + 2 * n, hist_cap=4096)
    if kind == "batch":
        ranges = [(lo, lo + 2 * n), (lo + 2 * n, lo + 4 * n)]
        return lambda g: g.verify_batch(ranges, hist_stride=3512)
    if kind == "pmin":
        buf = torch.zeros(10**6 if large else 1000, dtype=torch.int32, device="cuda")
        P = 1 << 16 if large else 227
        return lambda g: [g.verify_range(10**9, 10**9 + 2 * buf.numel(), P, pmin=buf, hist_cap=8192, allow_erange=True),
                          buf.cpu().numpy()]
    bits = 1 << 27 if large else 1000
    q = torch.zeros(bits // 64 + 1, dtype=torch.int64, device="cuda")
    return lambda g: [g.sieve_segment(10**9 + 1, bits, q), q.cpu().numpy()]


def _same(a, b):
    if isinstance(a, dict):
        return a.keys() == b.keys() and all(_same(a[k], b[k]) for k in a)
    if isinstance(a, list):
        return len(a) == len(b) and all(_same(x, y) for x, y in zip(a, b))
    return np.array_equal(a, b)


@pytest.mark.parametrize("kind", ["range", "batch", "pmin", "sieve"])
def test_small_and_large_calls_at_once(gbm, kind):
    with gbm.Context(device=0, base_limit=1 << 21, p1=1 << 15, p2=0) as parent:
        size = [False] * 4 + [True]
        streams = [torch.cuda.Stream() for _ in size]
        ctxs = [parent.share(s.cuda_stream) for s in streams]
        calls = [_calls(gbm, kind, large) for large in size]
        want = [f(g) for f, g in zip(calls, ctxs)]
        stop, errors, done = threading.Event(), [], [0] * len(size)

        def loop(i, most):
            try:
                with torch.cuda.stream(streams[i]):
                    while done[i] < most and not stop.is_set():
                        if not _same(calls[i](ctxs[i]), want[i]):
                            raise AssertionError(f"call {done[i]} of thread {i} gave another result")
                        done[i] += 1
            except Exception as e:                  # handed to the test's own thread
                errors.append(e)
            stop.set()                              # the small calls go on for as long as the large ones

        threads = [threading.Thread(target=loop, args=(i, 1500 if large else 10**6)) for i, large in enumerate(size)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        for g in ctxs:
            g.close()
    assert not errors, errors
    assert min(done) > 0 and done[-1] == 1500
