"""Host side of the window filter (no GPU): table files written before it
existed load as tables without one, files with it keep it, and its fields are
checked on load."""
import struct

import pytest

import workloads
from tests.test_table_io import EFORMAT, HEADER, fnv1a_words

pfac = pytest.importorskip("paper_1704_02272_gb300")

FIELDS = 40  # the filter's pointer and eight 32-bit fields, last in the table's description


def saved(tmp_path, sigma=52, n=100, lo=20, hi=20):
    w = workloads.tiny_case(5, sigma, n, lo, hi, 64)
    with pfac.Table(w.patterns, sigma, host_only=True) as t:
        t.save(tmp_path / "t.pfac")
        info, plan = t.info(), pfac.plan(t)
        ws = pfac.workspace_bytes(t, 1 << 20, 1)
    return (tmp_path / "t.pfac").read_bytes(), info, plan, ws


def rewrite(path, src, drop=False, at=None, new=b""):
    dt, _, mb = struct.unpack_from("<III", src, 16)
    d = bytearray(src)
    if at is not None:
        d[HEADER + dt - FIELDS + at:HEADER + dt - FIELDS + at + len(new)] = new
    if drop:
        del d[HEADER + dt - FIELDS:HEADER + dt]
        struct.pack_into("<I", d, 16, dt - FIELDS)
        struct.pack_into("<I", d, 24, mb - FIELDS)
    struct.pack_into("<Q", d, 40, fnv1a_words(bytes(d[HEADER:])))
    path.write_bytes(bytes(d))
    return path


def test_older_files_load_without_the_filter(tmp_path):
    src, info, plan, _ = saved(tmp_path)
    old = rewrite(tmp_path / "old.pfac", src, drop=True)
    with pfac.Table.load(old, host_only=True) as t:
        assert t.info() == info and pfac.plan(t) == plan
        assert pfac.workspace_bytes(t, 1 << 20, 1) == pfac.workspace_bytes(t, 1 << 20, 1, scan_kernel=1)


def test_files_keep_the_filter(tmp_path):
    src, info, plan, ws = saved(tmp_path)
    with pfac.Table.load(rewrite(tmp_path / "new.pfac", src), host_only=True) as t:
        assert t.info() == info and pfac.plan(t) == plan
        assert pfac.workspace_bytes(t, 1 << 20, 1) == ws


# offsets among the fields: pointer 0, words 8, copies 12, stride 16, bits 20,
# symbols hashed 24, symbols read 28, packed 32, short 36
@pytest.mark.parametrize("at,new", [(0, struct.pack("<Q", 1 << 40)), (8, struct.pack("<I", 1 << 20)),
                                    (8, struct.pack("<I", 33)), (12, struct.pack("<I", 6)),
                                    (16, struct.pack("<I", 3)), (20, struct.pack("<I", 0)),
                                    (24, struct.pack("<I", 0)), (28, struct.pack("<I", 17)),
                                    (32, struct.pack("<I", 1))])
def test_damaged_filters_are_refused(tmp_path, at, new):
    src = saved(tmp_path)[0]
    bad = rewrite(tmp_path / "bad.pfac", src, at=at, new=new)
    with pytest.raises(pfac.PfacError) as e:
        pfac.Table.load(bad, host_only=True)
    assert e.value.status == EFORMAT
