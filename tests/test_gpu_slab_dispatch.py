"""Which windows go through slabs, seen by the launches: below 10^12 slabs strike
every sieving prime, tiles leave those from the split on to the slices.  And
slabs against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SLAB = 13 << 17
A = 5 * 10**11 + 3


@pytest.fixture(scope="module")
def gbm():
    from paper_2603_02621_gb300 import gb
    gb.load()
    return gb


def _long():
    return 8 * torch.cuda.get_device_properties(0).multi_processor_count * SLAB


def _slices(gbm, g, A, nbits, q):
    """Launches of the primes from the split on for one window."""
    gbm.gb_profile_enable(g.handle, gbm.GB_PROFILE_EVENTS)
    g.sieve_segment(A, nbits, q)
    n = gbm.gb_profile_read(g.handle)["large"]["launches"]
    gbm.gb_profile_enable(g.handle, False)
    return n


@pytest.mark.parametrize("cfg,slabs", [(dict(), True), (dict(tile_bits=1 << 18, cta_threads=256), True),
                                       (dict(bucket_split=1 << 13), True), (dict(bucket_split=1 << 14), False),
                                       (dict(tile_bits=1 << 17), False), (dict(cta_threads=128), False)])
def test_default_tiling_given_in_words(gbm, cfg, slabs):
    """The split that results counts, not whether it was given."""
    nbits = _long()
    q = torch.zeros(nbits // 64, dtype=torch.int64, device="cuda")
    with gbm.Context(device=0, base_limit=1 << 20, **cfg) as g:
        assert (_slices(gbm, g, A, nbits, q) == 0) == slabs
        assert _slices(gbm, g, A, nbits - 64, q) > 0         # a slab short of eight rounds


def _against_oracle(oracle, q, A, nbits, at):
    for off in at:
        n = min(1 << 17, nbits - off)
        words = q[off // 64: (off + n + 63) // 64].cpu().numpy()
        bits = np.unpackbits(words.view(np.uint8), bitorder="little")[:n]
        np.testing.assert_array_equal(bits, oracle.odd_bits(A + 2 * off, n), err_msg=str(off))


@pytest.mark.parametrize("A,rounds", [(1, 10), (1, 0), ((1 << 37) + 1, 8), (A, 9), (10**15 + 7, 8)])
def test_slabs_against_the_oracle(gbm, oracle, A, rounds):
    """Windows at the start, around ends of slabs and of rounds, and at the end.
    (From 1 on, ten rounds reach past 2^32, where slabs begin; rounds 0 stands for
    2^35 numbers, whose sieving primes reach 2^18, so that the launches show it.)"""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nbits = rounds * sms * SLAB + 12345 if rounds else (1 << 35) + 12345
    assert A + 2 * (nbits - 1) >= 1 << 32 and nbits >= _long()
    q = torch.full(((nbits + 63) // 64,), -1, dtype=torch.int64, device="cuda")
    with gbm.Context(device=0, base_limit=1 << 26) as g:
        large = _slices(gbm, g, A, nbits, q)
        if 1 << 36 <= A + 2 * nbits < 1 << 40:
            assert large == 0
    n_rounds = -(-nbits // (SLAB * sms))                     # equal slabs, a multiple of 4096
    slab = min(SLAB, (nbits // (n_rounds * sms) + 4096) // 4096 * 4096)
    ends = [slab, 2 * slab, sms * slab, (n_rounds - 1) * sms * slab]
    at = [0] + [min(max(e - (1 << 16), 0), nbits - 64) // 64 * 64 for e in ends] + [(nbits - (1 << 16)) // 64 * 64]
    _against_oracle(oracle, q, A, nbits, at)
    last = q[nbits // 64:].cpu().numpy().view(np.uint8)
    assert not np.unpackbits(last, bitorder="little")[nbits % 64:].any()


def test_tuned_on_short_windows(gbm, monkeypatch, tmp_path):
    """Tile settings that the autotuner found on a batch, or on windows without
    slabs, leave long windows on their slabs; the same settings given by the
    caller do not, nor do those found on a long window."""
    path = tmp_path / "tune.txt"
    monkeypatch.setenv("GB_TUNE_CACHE", str(path))
    nbits = _long()
    q = torch.zeros(nbits // 64, dtype=torch.int64, device="cuda")
    short = [(10**9, 10**9 + 2000), (10**9 + 4000, 10**9 + 4600)]
    with gbm.Context(device=0, base_limit=1 << 20, p1=1 << 13, p2=0) as g:
        for mode, sample, slabs in ((gbm.GB_TUNE_BATCH, short, True), (gbm.GB_TUNE_PLAIN, short, True),
                                    (gbm.GB_TUNE_PLAIN, [(A - 1, A - 1 + 2 * nbits)], False)):
            g.set_config(tile_bits=1 << 18, bucket_split=0, cta_threads=256, p1=1 << 13, cover_prefix=0, seg_len=1 << 24)
            path.write_text("")
            g.autotune(sample, mode, reps=1)
            # what a search may come up with
            key = path.read_text().split("\t")[0]
            gbm.gb_tune_cache_store(str(path), key, dict(tile_bits=1 << 16, bucket_split=1 << 14, p1=1 << 13,
                                                         cover_prefix=144, seg_len=1 << 24, cta_threads=128), 1.0)
            g.set_config(tile_bits=1 << 18, bucket_split=0, cta_threads=256, p1=1 << 13, cover_prefix=0, seg_len=1 << 24)
            cfg, ms = g.autotune(sample, mode, reps=1)
            assert ms == 1.0 and cfg["tile_bits"] == 1 << 16
            assert (_slices(gbm, g, A, nbits, q) == 0) == slabs, mode
            g.set_config(seg_len=1 << 22)                     # not a tile setting
            assert (_slices(gbm, g, A, nbits, q) == 0) == slabs, mode
            with g.share() as h:
                assert (_slices(gbm, h, A, nbits, q) == 0) == slabs, mode
            g.set_config(cta_threads=512)
            assert _slices(gbm, g, A, nbits, q) > 0
            # a search that keeps the caller's tile settings leaves them the caller's
            gbm.gb_tune_cache_store(str(path), key, dict(tile_bits=1 << 16, bucket_split=1 << 14, p1=1 << 12,
                                                         cover_prefix=144, seg_len=1 << 24, cta_threads=512), 1.0)
            g.set_config(p1=1 << 13)
            g.autotune(sample, mode, reps=1)
            assert g.config()["p1"] == 1 << 12 and _slices(gbm, g, A, nbits, q) > 0
