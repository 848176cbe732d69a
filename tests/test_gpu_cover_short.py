"""The block cover of short chunks: ranges whose largest p_min lies in the
blocks because no probed n was covered."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def gbm():
    from paper_2603_02621_gb300 import gb
    gb.load()
    return gb


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
