"""The block cover with a bound so small that it cuts the blocks short: values
against the generic cover, and the steps it takes against what the blocks and the
n they leave open come to."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def gbm():
    from paper_2603_02621_gb300 import gb
    gb.load()
    return gb


# the bounds around the switches of the schedule: 48 odd primes, room for a block
# more in one class, in two, in all, and the last bounds it looks at
@pytest.mark.parametrize("P1", [227, 229, 269, 311, 337, 389, 439, 523, 617, 709, 857, 937, 941, 947])
@pytest.mark.parametrize("lo,n", [(4, 10**6 + 77), (10**12, 10**6 + 77), (10**15 + 2, 70001)])
def test_small_bounds(gbm, lo, n, P1):
    out = []
    with gbm.Context(device=0, base_limit=1 << 26, seg_len=1 << 20, p1=P1, p2=0) as g:
        for prefix in (0, 1):
            g.set_config(cover_prefix=prefix)
            out.append(g.verify_range(lo, lo + 2 * n, segs=True, seg_hist_stride=200, hist_cap=200))
    a, b = out
    assert a["segs"] == b["segs"]
    np.testing.assert_array_equal(a["seg_hist"], b["seg_hist"])
    np.testing.assert_array_equal(a["hist"], b["hist"])


@pytest.mark.parametrize("P1", [300, 512])
def test_steps(gbm, oracle, P1):
    """The n that the n's own useful primes up to the bound's last whole blocks
    leave open are the only ones probed."""
    lo, n = 10**12, 10**6
    odd = oracle.primes_upto(P1)[1:]
    pm = oracle.pmin_range(lo, lo + 2 * n, P1)
    with gbm.Context(device=0, base_limit=1 << 21, seg_len=1 << 20, p1=P1, p2=0) as g:
        gbm.gb_profile_enable(g.handle, True)
        g.verify_range(lo, lo + 2 * n)
        steps = gbm.gb_profile_work(g.handle)["cover_iterations"]
    v = (lo // 2 + np.arange(n)) * 2 % 3
    words, open_n = -(-n // 32), 0
    block_steps = 0
    for c in range(3):
        # 24 useful primes, and whole blocks of 16 with room below the bound (the n
        # divisible by 3: as many as the prefix's primes)
        useful = [p for p in odd if p % 3 != c]
        prefix = 48 if P1 == 300 else 80
        cap = prefix if c == 0 else prefix // 2 + 8
        blocks = max(0, min(-(-(cap - 24) // 16), (len(useful) - 24) // 16))
        last = useful[24 + 16 * blocks - 1]
        x = pm[v == c]
        open_n += int(np.count_nonzero((x == 0) | (x > last)))
        block_steps += (words / 3 + 96 * 17) * 24       # (three words per lane and warp, ends included)
        for b in range(blocks):
            left = int(np.count_nonzero((x == 0) | (x > useful[24 + 16 * b - 1])))
            block_steps += 16 * min(left, words / 3 + 1)
    rounds = 2 if len(odd) - 40 > 32 else 1             # of 32 primes to an open n's end, at most
    assert steps <= block_steps + 32 * rounds * open_n, (steps, block_steps, open_n)
