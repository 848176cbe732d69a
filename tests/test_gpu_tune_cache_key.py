"""Autotune cache lines of earlier kernels (whose keys name none) are not used."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_lines_of_other_kernels_are_not_used(monkeypatch, tmp_path):
    from paper_2603_02621_gb300 import gb
    path = tmp_path / "tune.txt"
    monkeypatch.setenv("GB_TUNE_CACHE", str(path))
    ranges = [(10**9, 10**9 + 2000), (10**9 + 4000, 10**9 + 4600)]
    with gb.Context(device=0, base_limit=1 << 20, seg_len=1 << 20, p1=1 << 13, p2=0) as g:
        g.autotune(ranges, gb.GB_TUNE_BATCH, reps=1)
        key = path.read_text().split("\t")[0]
        base, kernels = key.rsplit("|", 1)
        assert base.count("|") == 7 and kernels[0] == "k" and int(kernels[1:]) >= 2
        stale = dict(tile_bits=1 << 16, bucket_split=1 << 14, p1=1 << 12, cover_prefix=48, seg_len=1 << 20, cta_threads=512)
        for other in (base, base + "|k1", f"{base}|k{int(kernels[1:]) + 1}"):
            path.write_text("")
            gb.gb_tune_cache_store(str(path), other, stale, 1e-9)
            g.set_config(tile_bits=1 << 18, bucket_split=0, cta_threads=256, p1=1 << 13, cover_prefix=0)
            cfg, ms = g.autotune(ranges, gb.GB_TUNE_BATCH, reps=1)
            assert ms > 1e-6, other                              # searched, not looked up
            assert path.read_text().splitlines()[-1].startswith(key + "\t")
