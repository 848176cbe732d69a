"""One warp per query: p_min past the first window of candidates, batches
around the launch's switch from one warp per CTA to four, small n at the
window's ends, host and device arrays."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

P2 = 1 << 20


@pytest.fixture(scope="module")
def qctx():
    from paper_2603_02621_gb300 import gb
    with gb.Context(device=0, base_limit=1 << 20, p1=1 << 15, p2=P2) as g:
        yield g


@pytest.mark.parametrize("n,p", [(514252927964, 2473), (1000001860632968, 3517), (3999999803335070632, 4643)])
def test_p_min_past_the_first_window(qctx, oracle, n, p):
    assert oracle.pmin_single(n, P2) == p
    assert qctx.query(n) == p
    # the bound just below p_min finds nothing, the bound at it does
    assert qctx.query_batch([n], p - 1).tolist() == [0] and qctx.query_batch([n], p).tolist() == [p]


@pytest.mark.parametrize("lo", [4, 2040, 4086, 2048**2 - 64, 2**32 - 40])
def test_window_ends_and_untested_partners(qctx, oracle, lo):
    ns = np.arange(lo - lo % 2, lo - lo % 2 + 80, 2, dtype=np.uint64)
    want = np.array([oracle.pmin_single(int(n), P2) for n in ns], dtype=np.uint32)
    np.testing.assert_array_equal(qctx.query_batch(ns), want)


@pytest.mark.parametrize("count", [1, 3, 607, 608, 609, 1217, (1 << 16) + 1])
def test_batch_sizes(qctx, oracle, count):
    rng = np.random.default_rng(count)
    ns = rng.integers(2, 2 * 10**18, size=count, dtype=np.uint64) * np.uint64(2)
    got = qctx.query_batch(ns)
    pick = rng.integers(0, count, size=min(count, 40))
    for i in pick:
        assert int(got[i]) == oracle.pmin_single(int(ns[i]), P2), int(ns[i])
    # from and to device memory
    dev = torch.from_numpy(ns.view(np.int64)).cuda()
    np.testing.assert_array_equal(qctx.query_batch(dev), got)
    out = torch.zeros(count, dtype=torch.int32, device="cuda")
    qctx.query_batch(dev, out=out)
    np.testing.assert_array_equal(out.cpu().numpy().view(np.uint32), got)
    out.zero_()
    qctx.query_batch(ns, out=out)
    np.testing.assert_array_equal(out.cpu().numpy().view(np.uint32), got)
