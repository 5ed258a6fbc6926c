"""The autotuner's cache where the library's own choice is the fastest: the
line of zeros that says so is read back as that choice, on CPU, and written
by a tuning run, on the GPU."""
import pytest
import torch

import workloads
from tests.test_tune_cache import cache_key, sample

pfac = pytest.importorskip("paper_1704_02272_gb300")


@pytest.mark.skipif(torch.cuda.is_available(), reason="the cache key names the GPU; this test keys it for none")
@pytest.mark.parametrize("sigma,n,lo,hi", [(256, 1000, 4, 32), (4, 300, 3, 24), (52, 100, 20, 20)])
def test_own_choice_is_read_back(tmp_path, sigma, n, lo, hi):
    with pfac.Table(workloads.tiny_case(9, sigma, n, lo, hi, 0).patterns, sigma, host_only=True) as t:
        text, seg = sample()
        own, key, path = (pfac.plan(t), pfac.kernel(t)), cache_key(t, text.numel(), 1), tmp_path / "tune.txt"
        path.write_text(f"{key} 1 {own[0]['prefix_depth']} 1 1 1 1 16 1 32 1 0.7\n")
        r = pfac.autotune(t, text, seg, cache_path=str(path), stream=0)
        assert r["from_cache"] == 1 and r["variant"] == 1 and pfac.kernel(t) == "queued"
        path.write_text(path.read_text() + f"{key} 0 0 0 0 0 0 0 0 0 0 0.25\n")
        r = pfac.autotune(t, text, seg, cache_path=str(path), stream=0)  # the last line wins
        assert r["from_cache"] == 1 and r["variant"] == 0 and r["scan_ms"] == 0.25
        assert (pfac.plan(t), pfac.kernel(t)) == own


@pytest.mark.skipif(torch.cuda.is_available(), reason="the cache key names the GPU; this test keys it for none")
@pytest.mark.parametrize("line", ["0 2 0 0 0 0 0 0 0 0 0.5", "0 0 0 0 0 0 0 1 0 0 0.5", "0 0 0 0 0 0 24 0 0 0 0.5"])
def test_lines_of_some_zeros_are_ignored(tmp_path, line):
    with pfac.Table(workloads.tiny_case(9, 256, 1000, 4, 32, 0).patterns, 256, host_only=True) as t:
        text, seg = sample()
        default, path = pfac.plan(t), tmp_path / "tune.txt"
        path.write_text(f"{cache_key(t, text.numel(), 1)} {line}\n")
        with pytest.raises(pfac.PfacError):  # tuning needs a GPU
            pfac.autotune(t, text, seg, cache_path=str(path), stream=0)
        assert pfac.plan(t) == default


@pytest.mark.gpu
@pytest.mark.parametrize("sigma,n,lo,hi", [(256, 1000, 4, 32), (20, 3000, 4, 30), (4, 300, 3, 24)])
def test_every_choice_is_cached(tmp_path, sigma, n, lo, hi):
    w = workloads.tiny_case(91, sigma, n, lo, hi, 2 << 20)
    text = torch.from_numpy(w.text).cuda()
    seg = pfac.single_segment(text.numel(), "cuda")
    path = str(tmp_path / "tune.txt")
    with pfac.Table(w.patterns, sigma) as t, pfac.Table(w.patterns, sigma) as u:
        r = pfac.autotune(t, text, seg, cache_path=path)
        assert r["from_cache"] == 0 and r["default_ms"] > 0 and r["scan_ms"] > 0
        s = pfac.autotune(u, text, seg, cache_path=path)
        assert s["from_cache"] == 1
        same = ("variant", "prefix_depth", "bitmap_copies", "scan_kernel", "records_per_slice", "resolver")
        assert {k: s[k] for k in same} == {k: r[k] for k in same}
        assert pfac.plan(u) == pfac.plan(t) and pfac.kernel(u) == pfac.kernel(t)
