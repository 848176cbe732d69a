"""gb_verify_range_noalloc where the first pass leaves more n open than its
retry list holds (a small P1): the results are still gb_verify_range's and the
oracle's, and nothing is allocated."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

H = 3512
P2 = 1 << 20


@pytest.mark.parametrize("lo", [10**9, 10**12, 10**15])
@pytest.mark.parametrize("n", [1, 63, 1000, 100003])
def test_more_open_n_than_words(oracle, lo, n):
    from paper_2603_02621_gb300 import gb
    hi = lo + 2 * n
    kw = dict(hist_cap=H, seg_hist_stride=H)
    with gb.Context(device=0, base_limit=1 << 26, seg_len=1 << 20, p1=227, p2=P2) as g:
        before = gb.gb_alloc_stats()
        got = g.verify_range_noalloc(lo, hi, **kw)
        assert gb.gb_alloc_stats() == before
        ref = g.verify_range(lo, hi, **kw)
    summ, hist = oracle.verify_segments(lo, hi, n, P2, H)
    assert [got["n_checked"], got["unresolved"], got["max_pmin"], got["max_pmin_n"]] == summ[0].tolist()
    np.testing.assert_array_equal(got["hist"], hist[0])
    for key in ("unresolved", "max_pmin", "max_pmin_n", "hist_len", "n_segments", "p_final", "segs"):
        assert got[key] == ref[key], key
    np.testing.assert_array_equal(got["hist"], ref["hist"])
    np.testing.assert_array_equal(got["seg_hist"], ref["seg_hist"])
