"""The merged words of the partition counts' residues: allocated once for a call
of many stretches, and done without where they cannot be had."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture()
def gbm():
    from paper_2603_02621_gb300 import gb
    gb.load()
    yield gb
    gb.gb_fault_set(None)


@pytest.mark.parametrize("which", [4, 5])
def test_without_memory_for_the_residues(gbm, oracle, which):
    """The prime bits, their reversal and the counts are a call's first three
    allocations, the merged words the next two: without them the plain kernel
    counts, and the next call has them."""
    lo, count = 10**8, 200
    want = [oracle.partitions(lo + 2 * j) for j in (0, 77, count - 1)]
    with gbm.Context(device=0, base_limit=1 << 17) as g:
        gbm.gb_fault_set(f"alloc@{which}")
        a = g.partitions(lo, lo + 2 * count)
        gbm.gb_fault_set(None)
        before = gbm.gb_alloc_stats()["count"]
        b = g.partitions(lo, lo + 2 * count)
        assert gbm.gb_alloc_stats()["count"] == before + 2
    np.testing.assert_array_equal(a, b)
    assert [int(a[j]) for j in (0, 77, count - 1)] == want


def test_one_allocation_for_all_stretches(gbm, oracle):
    lo, count = 1 << 20, 1 << 22
    with gbm.Context(device=0, base_limit=1 << 17) as g:
        before = gbm.gb_alloc_stats()["count"]
        got = g.partitions(lo, lo + 2 * count)
        assert gbm.gb_alloc_stats()["count"] <= before + 6     # (one more: the slices' residue table)
    for j in (0, 8191, 8192, 100003, count // 2 + 1, count - 1):
        assert int(got[j]) == oracle.partitions(lo + 2 * j), j


@pytest.mark.parametrize("lo", [1 << 20, (1 << 20) + 2, 1 << 21, 3 * (1 << 20) - 4])
def test_short_sums(gbm, oracle, lo):
    """Stretches of an eighth of the way and of 2^17 n: the n at and around their
    ends, and others."""
    count = 400000
    with gbm.Context(device=0, base_limit=1 << 17) as g:
        got = g.partitions(lo, lo + 2 * count)
        ends, a = [], lo
        while a < lo + 2 * count:
            ends += [a - 2, a, a + 2]
            a += max(a // 64 // 2 * 2, min(a // 8 // 2 * 2, 1 << 18))
        for n in ends[1:]:
            assert int(got[(n - lo) // 2]) == oracle.partitions(n), n
        rng = np.random.default_rng(lo)
        for j in rng.integers(0, count, size=50):
            assert int(got[j]) == oracle.partitions(lo + 2 * int(j)), j


def test_long_calls_of_short_sums(gbm):
    """Where the sums are short a call is its launches: few of them for 2*10^5 n."""
    lo, count = 1 << 20, 200000
    with gbm.Context(device=0, base_limit=1 << 17) as g:
        out = torch.zeros(count, dtype=torch.int32, device="cuda")
        gbm.gb_profile_enable(g.handle, True)
        g.partitions(lo, lo + 2 * count, out=out)
        # a sieve and a reversal, then three launches a stretch: four stretches
        assert gbm.gb_profile_kernels(g.handle) <= 2 + 2 + 3 * 4
