"""The slab sieve of long windows against tiles and slices (another CTA size
takes those): lengths at and past whole rounds of slabs, windows where the last
sieving primes' squares lie inside, and one from below zero."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SLAB = 13 << 17


@pytest.fixture(scope="module")
def gbm():
    from paper_2603_02621_gb300 import gb
    gb.load()
    return gb


def _sieve(gbm, A, nbits, **cfg):
    q = torch.full(((nbits + 63) // 64,), -1, dtype=torch.int64, device="cuda")
    with gbm.Context(device=0, base_limit=1 << 26, **cfg) as g:
        gbm.gb_profile_enable(g.handle, True)
        n = g.sieve_segment(A, nbits, q)
        w = gbm.gb_profile_work(g.handle)
        gbm.gb_profile_enable(g.handle, False)
        m = g.sieve_segment(A, nbits, q)            # without the counters
    assert n == m
    return n, q, w["sieve_strikes"] + w["large_strikes"]


@pytest.mark.parametrize("A", [1, (1 << 33) + 5, (1 << 37) + 1, 5 * 10**11 + 3, 10**12 - 10**9 + 1, 10**15 + 7])
@pytest.mark.parametrize("rounds,more", [(8, 0), (8, 1), (8, -64 + (1 << 18)), (9, 12345)])
def test_slabs_equal_tiles_and_slices(gbm, A, rounds, more):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nbits = rounds * sms * SLAB + more
    na, qa, wa = _sieve(gbm, A, nbits)
    nb, qb, wb = _sieve(gbm, A, nbits, cta_threads=128)
    assert na == nb and wa == wb
    assert torch.equal(qa, qb)


def test_slabs_from_below_zero(gbm):
    A, nbits = -(1 << 22) + 1, (1 << 35) + 12345
    na, qa, _ = _sieve(gbm, A, nbits)
    nb, qb, _ = _sieve(gbm, A, nbits, cta_threads=128)
    assert na == nb and torch.equal(qa, qb)
    assert not qa[: (1 << 21) // 64].any()            # the odd numbers below 0
