"""Short ranges and windows: the first pass's halo alone, the retry pass on
demand, the slices' primes by global atomics, tiles shorter than the default."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

N9781 = 3325581707333960528        # its p_min, 9781, is above 2^13


@pytest.fixture(scope="module")
def gbm():
    from paper_2603_02621_gb300 import gb
    gb.load()
    return gb


def _values(r):
    return [r[k] for k in ("n_checked", "unresolved", "max_pmin", "max_pmin_n", "hist_len")]


@pytest.mark.parametrize("before,n", [(0, 1), (5, 6), (700, 1500), (4000, 70000)])
def test_retry_on_demand(gbm, oracle, before, n):
    """A short range whose first pass (P1 = 2^13) leaves one n open: the retry
    pass gives what one pass to 2^15 gives, in every output."""
    lo = N9781 - 2 * before
    hi = lo + 2 * n
    H = 3512
    with gbm.Context(device=0, base_limit=2 * 10**9, seg_len=1 << 20, p1=1 << 13, p2=1 << 20) as g:
        got = g.verify_range(lo, hi, hist_cap=90000, segs=True, seg_hist_stride=H)
        dev = torch.zeros(n, dtype=torch.int32, device="cuda")
        got_pm = g.verify_range(lo, hi, pmin=dev)
        host = np.zeros(n, dtype=np.uint32)
        g.verify_range(lo, hi, pmin=host)
        again = g.verify_range(N9781 + 2, N9781 + 2002)           # nothing left open: no stale retry
        want = g.verify_range(lo, hi, 1 << 15, hist_cap=90000, segs=True, seg_hist_stride=H)
        q = g.query_batch(np.arange(lo, hi, 2, dtype=np.uint64))
        assert again["unresolved"] == 0 and again["max_pmin"] < 8192
    assert got["max_pmin"] == 9781 and got["max_pmin_n"] == N9781 and got["unresolved"] == 0
    assert _values(got) == _values(want) == _values(got_pm)
    np.testing.assert_array_equal(got["hist"], want["hist"])
    np.testing.assert_array_equal(got["seg_hist"], want["seg_hist"])
    assert got["segs"] == want["segs"]
    np.testing.assert_array_equal(host, q)
    np.testing.assert_array_equal(dev.cpu().numpy().view(np.uint32), q)


@pytest.mark.parametrize("A", [1, 10**12 - 999, 10**13 + 1])
@pytest.mark.parametrize("nbits", [1, 8191, 8192, 8193, (1 << 18) - 1, (1 << 18) + 1, 3 * (1 << 18) + 77, (1 << 22) + 5])
def test_short_windows_vs_oracle(gbm, oracle, A, nbits):
    with gbm.Context(device=0, base_limit=1 << 22) as g:
        q = torch.full(((nbits + 63) // 64,), -1, dtype=torch.int64, device="cuda")
        pc = g.sieve_segment(A, nbits, q)
    bits = np.unpackbits(q.cpu().numpy().view(np.uint8), bitorder="little")
    ref = oracle.odd_bits(A, nbits)
    np.testing.assert_array_equal(bits[:nbits], ref)
    assert not bits[nbits:].any() and pc == int(ref.sum())


@pytest.mark.parametrize("slices", [24, 25, 26])
@pytest.mark.parametrize("tail", [0, 1, 12345])
def test_slices_and_atomics_agree(gbm, monkeypatch, slices, tail):
    """Window lengths around the switch between the slices and the atomics: the
    bits of the longer window's start equal the shorter one's, and both equal
    the sieve without slices."""
    A, nbits = 10**14 + 1, slices * (7 << 18) + tail

    def sieve():
        with gbm.Context(device=0, base_limit=1 << 24) as g:
            q = torch.zeros(((nbits + 63) // 64,), dtype=torch.int64, device="cuda")
            return g.sieve_segment(A, nbits, q), q.cpu()

    pa, qa = sieve()
    monkeypatch.setenv("GB_MID_LOG2", "0")
    pb, qb = sieve()
    assert pa == pb and torch.equal(qa, qb)


@pytest.mark.parametrize("cap", [100, 3512, 100000])
@pytest.mark.parametrize("n", [1000, 1 << 23])
def test_histogram_into_device_memory(gbm, cap, n):
    """The merged histogram into a device buffer of the caller: shorter than the
    histogram's used part, longer, and longer than any prime index."""
    import ctypes
    lo = 10**12
    with gbm.Context(device=0, base_limit=1 << 21, seg_len=1 << 20, p1=1 << 15, p2=1 << 20) as g:
        want = g.verify_range(lo, lo + 2 * n, hist_cap=cap, allow_erange=True)
        dev = torch.full((cap,), -1, dtype=torch.int64, device="cuda")
        r = gbm.gb_range_result()
        r.hist = ctypes.cast(dev.data_ptr(), ctypes.POINTER(ctypes.c_uint64))
        r.hist_cap = cap
        rc = gbm.load().gb_verify_range(g.handle, lo, lo + 2 * n, 0, ctypes.byref(r))
    assert rc == want["rc"]
    np.testing.assert_array_equal(dev.cpu().numpy().view(np.uint64), want["hist"])
