"""A workspace sized without options is large enough for the same input with
options that only choose how it is scanned (no GPU)."""
import pytest

import workloads

pfac = pytest.importorskip("paper_1704_02272_gb300")


@pytest.mark.parametrize("sigma,n,lo,hi", [(256, 1000, 4, 32), (256, 20000, 2, 40), (52, 100, 20, 20),
                                           (20, 3000, 4, 30), (4, 3000, 8, 40), (4, 300, 3, 24), (2, 50, 6, 20)])
@pytest.mark.parametrize("n_bytes,segments", [(100, 1), (70_001, 3), (5 << 20, 1), (300 << 20, 400_000)])
def test_options_that_choose_the_scan(sigma, n, lo, hi, n_bytes, segments):
    w = workloads.tiny_case(3, sigma, n, lo, hi, 64)
    with pfac.Table(w.patterns, sigma, host_only=True) as t:
        room = pfac.workspace_bytes(t, n_bytes, segments)
        depth = pfac.plan(t)["prefix_depth"]
        for opt in ({"scan_kernel": 1}, {"variant": 1}, {"prefix_depth": depth}, {"bitmap_copies": 1},
                    {"gram_filter": 1}, {"warps_per_cta": 16}, {"ctas_per_sm": 1}, {"resolver": 1},
                    {"records_per_slice": 32}):
            assert pfac.workspace_bytes(t, n_bytes, segments, **opt) <= room, opt
        # and for fewer bytes and segments, as chunks of it are matched
        for b, s in ((n_bytes // 2, segments), (n_bytes, 1), (1, 1)):
            assert pfac.workspace_bytes(t, b, s) <= room, (b, s)
