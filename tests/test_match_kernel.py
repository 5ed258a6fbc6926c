"""The kernel a call runs, as the library reports it (no GPU): the window and
dense scan kernels take the calls that leave every choice to the library, any
choice the plan's own kernel."""
import pytest

import workloads

pfac = pytest.importorskip("paper_1704_02272_gb300")


def table(sigma, n, lo, hi, **kw):
    return pfac.Table(workloads.tiny_case(9, sigma, n, lo, hi, 0).patterns, sigma, host_only=True, **kw)


@pytest.mark.parametrize("kw", [{}, {"layout": pfac.LAYOUT_DENSE}], ids=["compressed", "uncompressed"])
@pytest.mark.parametrize("sigma,n,lo,hi,plan_kernel", [(256, 1000, 4, 32, "register"), (52, 100, 20, 20, "queued"),
                                                       (20, 3000, 5, 30, "queued"), (4, 3000, 8, 40, "queued")])
def test_window_kernel(sigma, n, lo, hi, plan_kernel, kw):
    with table(sigma, n, lo, hi, **kw) as t:
        assert pfac.kernel(t) == pfac.kernel(t, 1000) == pfac.kernel(t, starts_end=5, position_base=3) == "window"
        for opt in ({"variant": 1}, {"resolver": 1}, {"records_per_slice": 32}, {"bitmap_copies": 1},
                    {"prefix_depth": pfac.plan(t)["prefix_depth"]}):
            assert pfac.kernel(t, 1, **opt) == plan_kernel, opt
        assert pfac.kernel(t, 1, scan_kernel=1) == "queued"


def test_dense_scan_kernel():
    with table(4, 300, 3, 24) as t:
        assert pfac.kernel(t) == "dense" and pfac.kernel(t, 2) == "queued"
        assert pfac.kernel(t, 1, scan_kernel=2) == "register"


def test_other_kernels():
    with table(2, 50, 6, 20) as t:  # one-bit symbols: no window filter
        assert pfac.kernel(t) == "queued"
    with table(256, 200, 4, 12, suffix_merge=True) as t:
        assert pfac.kernel(t) == "queued"
    with table(256, 200, 4, 12, layout=pfac.LAYOUT_DENSE) as t:
        assert pfac.kernel(t, 1, scan_kernel=3) == "serial"
    with table(52, 100, 20, 20) as t, pytest.raises(pfac.PfacError):
        pfac.kernel(t, 1, variant=7)
