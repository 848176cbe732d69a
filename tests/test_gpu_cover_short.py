"""The block cover of short chunks: segments of a few words (a warp per class),
chunks of a few warps, ranges whose largest p_min lies in the blocks because no
probed n was covered -- values against the generic cover, and their time against
longer chunks of the same n."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def gbm():
    from paper_2603_02621_gb300 import gb
    gb.load()
    return gb


@pytest.mark.parametrize("P1", [227, 1024, 1 << 15])
@pytest.mark.parametrize("lo", [4, 10**12, 10**15 + 2])
@pytest.mark.parametrize("seg", [1 << 11, 1 << 12, 1 << 13, 9 << 10, 1 << 14, 1 << 15, 46 << 10])
def test_short_segments(gbm, lo, seg, P1):
    n = 5 * seg + 77
    out = []
    with gbm.Context(device=0, base_limit=1 << 26, seg_len=seg - seg % 2048, p1=P1, p2=0) as g:
        for prefix in (0, 1):
            g.set_config(cover_prefix=prefix)
            out.append(g.verify_range(lo, lo + 2 * n, segs=True, seg_hist_stride=3600, hist_cap=3600))
        g.set_config(cover_prefix=0)
        b = g.verify_batch([(s["lo"], s["hi"]) for s in out[0]["segs"]], hist_stride=3600)
    assert out[0]["segs"] == out[1]["segs"] == b["records"]
    np.testing.assert_array_equal(out[0]["seg_hist"], out[1]["seg_hist"])
    np.testing.assert_array_equal(out[0]["seg_hist"], b["hist"])
    np.testing.assert_array_equal(out[0]["hist"], out[1]["hist"])


def _cover_ms(gbm, lo, n, **cfg):
    with gbm.Context(device=0, base_limit=1 << 26, p2=0, **cfg) as g:
        ms = []
        for _ in range(12):
            gbm.gb_profile_enable(g.handle, gbm.GB_PROFILE_EVENTS)
            g.verify_range(lo, lo + 2 * n)
            ms.append(gbm.gb_profile_read(g.handle)["cover"]["ms"])
        return min(ms)


def test_maximum_in_the_blocks_is_no_slow_path(gbm):
    """10^4 n of which one class has none that the probing covers (bound 1024),
    against a bound where it covers some of every class.  Counting the words
    over from global memory took 15 times as long, once more from the merged
    words 3 times."""
    a = _cover_ms(gbm, 10**15, 10**4, p1=1024)
    b = _cover_ms(gbm, 10**15, 10**4, p1=2048)
    assert a < 6 * b, (a, b)


def test_short_segments_time(gbm):
    """The same n in segments of 2^11 and of 2^16: 13 times as long with CTAs of
    16 warps for 64 words, 3 times with one warp per class."""
    a = _cover_ms(gbm, 10**12, 1 << 24, p1=1 << 15, seg_len=1 << 11)
    b = _cover_ms(gbm, 10**12, 1 << 24, p1=1 << 15, seg_len=1 << 16)
    assert a < 6 * b, (a, b)


@pytest.mark.parametrize("lo,n,P1", [(10**18, 1 << 22, 1600), (10**15, 10**6, 1024), (10**12, 3 * 10**6, 709)])
def test_maximum_in_the_blocks_is_the_same_every_time(gbm, lo, n, P1):
    """Chunks finish in any order, and whether one has to look its maximum up
    depends on it; the segments' maxima do not."""
    with gbm.Context(device=0, base_limit=2 * 10**9 if lo > 10**16 else 1 << 26, seg_len=1 << 20, p1=P1, p2=0) as g:
        g.set_config(cover_prefix=1)
        want = g.verify_range(lo, lo + 2 * n, segs=True, hist_cap=300)
        g.set_config(cover_prefix=0)
        for _ in range(40):
            got = g.verify_range(lo, lo + 2 * n, segs=True, hist_cap=300)
            assert got["segs"] == want["segs"]
            np.testing.assert_array_equal(got["hist"], want["hist"])


def test_batches_of_short_ranges_time(gbm):
    """1000 ranges of 1000 n: their cover in CTAs of 16 warps, the classes one
    after the other, took 4.4 times as long as the generic cover of one of them,
    in CTAs of 4 warps as long."""
    ranges = [(10**9 + 40000 * i, 10**9 + 40000 * i + 2000) for i in range(1000)]
    ms = []
    with gbm.Context(device=0, base_limit=1 << 20, p1=1 << 15, p2=0) as g:
        for _ in range(12):
            gbm.gb_profile_enable(g.handle, gbm.GB_PROFILE_EVENTS)
            g.verify_batch(ranges)
            ms.append(gbm.gb_profile_read(g.handle)["cover"]["ms"])
    one = _cover_ms(gbm, 10**9, 1000, p1=1 << 15, cover_prefix=1)
    assert min(ms) < 2.2 * one, (min(ms), one)
