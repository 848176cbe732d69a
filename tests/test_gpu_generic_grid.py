"""The generic cover of a range far shorter than its segment: as many CTAs as
the range needs, whatever the segment's length."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def gbm():
    from paper_2603_02621_gb300 import gb
    gb.load()
    return gb


@pytest.mark.parametrize("n", [1, 1000, 70000])
def test_cover_time_does_not_grow_with_the_segment(gbm, oracle, n):
    lo = 10**12
    ms = {}
    for seg in (1 << 17, 1 << 30):
        buf = torch.zeros(n, dtype=torch.int32, device="cuda")
        with gbm.Context(device=0, base_limit=1 << 21, seg_len=seg, p1=1 << 15, p2=0) as g:
            times = []
            for _ in range(10):
                gbm.gb_profile_enable(g.handle, gbm.GB_PROFILE_EVENTS)
                g.verify_range(lo, lo + 2 * n, pmin=buf)
                times.append(gbm.gb_profile_read(g.handle)["cover"]["ms"])
            ms[seg] = min(times)
        np.testing.assert_array_equal(buf.cpu().numpy().view(np.uint32), oracle.pmin_range(lo, lo + 2 * n, 1 << 15))
    # (the same kernel on the same words: a factor of two is far outside its noise)
    assert ms[1 << 30] < 2 * ms[1 << 17], ms


def test_last_segment_mostly_empty(gbm, oracle):
    """Several segments, the last one with a few n of its many chunks."""
    seg, n = 1 << 17, 2 * (1 << 17) + 5
    lo = 10**9
    buf = torch.zeros(n, dtype=torch.int32, device="cuda")
    H = len(oracle.primes_upto(1 << 15))
    with gbm.Context(device=0, base_limit=1 << 17, seg_len=seg, p1=1 << 15, p2=0) as g:
        r = g.verify_range(lo, lo + 2 * n, pmin=buf, segs=True, seg_hist_stride=H)
    summ, hist = oracle.verify_segments(lo, lo + 2 * n, seg, 1 << 15, H)
    assert [[s["n_checked"], s["unresolved"], s["max_pmin"], s["max_pmin_n"]] for s in r["segs"]] == summ.tolist()
    np.testing.assert_array_equal(r["seg_hist"], hist)
    np.testing.assert_array_equal(buf.cpu().numpy().view(np.uint32), oracle.pmin_range(lo, lo + 2 * n, 1 << 15))
