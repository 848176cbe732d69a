"""The block cover's classes mod 3: chunks, streams and tails of every phase,
against the generic cover (which takes the n as they come) and the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

WORDS = 3 * (3 * 512 - 1)          # coverage words of a one-round chunk


@pytest.fixture(scope="module")
def gbm():
    from paper_2603_02621_gb300 import gb
    gb.load()
    return gb


def _same(g, lo, n, P1, H):
    out = []
    for prefix in (0, 1):                       # block cover, generic cover
        g.set_config(cover_prefix=prefix)
        r = g.verify_range(lo, lo + 2 * n, P1, segs=True, seg_hist_stride=H, hist_cap=H)
        out.append(r)
    a, b = out
    assert a["segs"] == b["segs"]
    np.testing.assert_array_equal(a["seg_hist"], b["seg_hist"])
    np.testing.assert_array_equal(a["hist"], b["hist"])
    for k in ("unresolved", "max_pmin", "max_pmin_n", "hist_len"):
        assert a[k] == b[k], k
    return a


@pytest.mark.parametrize("P1", [227, 293, 1 << 13])
@pytest.mark.parametrize("lo", [4, 6, 8, 10, 10**12, 10**12 + 2, 10**12 + 4])
def test_short_ranges(gbm, oracle, lo, P1):
    """Every residue of the first n, lengths around words and streams; n = 4 and
    n = 6, whose partners are no member of a class."""
    H = len(oracle.primes_upto(P1))
    with gbm.Context(device=0, base_limit=1 << 21, seg_len=1 << 20, p1=P1, p2=0) as g:
        for n in (1, 2, 3, 31, 32, 33, 63, 64, 65, 95, 96, 97, 128, 160, 1000, 32 * 96 * 3, 32 * 96 * 3 + 5):
            r = _same(g, lo, n, P1, H)
            if n <= 1000:
                summ, hist = oracle.verify_segments(lo, lo + 2 * n, 1 << 20, P1, H)
                s = r["segs"][0]
                assert [s["n_checked"], s["unresolved"], s["max_pmin"], s["max_pmin_n"]] == summ[0].tolist(), n
                np.testing.assert_array_equal(r["seg_hist"][0], hist[0])


@pytest.mark.parametrize("lo", [4, 10**9 + 2, 10**15, 4 * 10**18 - 10**11])
@pytest.mark.parametrize("words", [WORDS - 1, WORDS, WORDS + 1, WORDS + 2, 2 * WORDS + 1, 40 * WORDS + 7])
def test_chunk_tails(gbm, oracle, lo, words):
    """The last chunk one word short, whole, or a word or two over, with a
    ragged last word."""
    P1 = 1 << 15
    H = len(oracle.primes_upto(P1))
    with gbm.Context(device=0, base_limit=2 * 10**9 + 10**6 if lo > 10**16 else 1 << 25, seg_len=1 << 26, p1=P1,
                     p2=0) as g:
        for n in (32 * words, 32 * words - 13):
            _same(g, lo, n, P1, H)


@pytest.mark.parametrize("seg", [2048, 6144, 1 << 20])
def test_many_segments_and_batches(gbm, oracle, seg):
    """Segments shorter than a chunk, and the batched form of the same ranges."""
    P1 = 1 << 13
    H = len(oracle.primes_upto(P1))
    lo, n = 10**11, 3 * seg * 32 + 77
    with gbm.Context(device=0, base_limit=1 << 20, seg_len=seg, p1=P1, p2=0) as g:
        r = _same(g, lo, n, P1, H)
        g.set_config(cover_prefix=0)
        ranges = [(s["lo"], s["hi"]) for s in r["segs"]]
        b = g.verify_batch(ranges, P1, hist_stride=H)
        assert b["records"] == r["segs"]
        np.testing.assert_array_equal(b["hist"], r["seg_hist"])
