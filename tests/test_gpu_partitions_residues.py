"""Partition counts by residues mod 15 against the plain kernel (short calls
take it) and the oracle: counts around blocks of 480, several stretches of one
call, lengths that leave the streams' words any remainder."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pctx():
    from paper_2603_02621_gb300 import gb
    with gb.Context(device=0, base_limit=1 << 17) as g:
        yield g


def _plain(g, lo, hi):
    # fewer than 96 n a call: the plain kernel
    return np.concatenate([g.partitions(a, min(hi, a + 2 * 90)) for a in range(lo, hi, 2 * 90)])


@pytest.mark.parametrize("lo", [(1 << 20) - 200, 1 << 20, (1 << 20) + 2, 3000002, 16777214, 10**8])
@pytest.mark.parametrize("count", [96, 97, 479, 480, 481, 1000])
def test_residues_equal_plain(pctx, oracle, lo, count):
    got = pctx.partitions(lo, lo + 2 * count)
    np.testing.assert_array_equal(got, _plain(pctx, lo, lo + 2 * count))
    for j in (0, 1, count // 2, count - 1):
        if lo < 10**7:
            assert int(got[j]) == oracle.partitions(lo + 2 * j), j


def test_many_stretches(pctx):
    lo, hi = (1 << 20) - 4000, (1 << 20) + 120000
    np.testing.assert_array_equal(pctx.partitions(lo, hi), _plain(pctx, lo, hi))


def test_largest_n(pctx):
    hi = 1 << 34
    a = pctx.partitions(hi - 2 * 96, hi)
    b = pctx.partitions(hi - 2 * 96, hi - 2 * 90)
    c = pctx.partitions(hi - 2 * 4, hi)
    np.testing.assert_array_equal(a[:6], b)
    np.testing.assert_array_equal(a[-4:], c)
