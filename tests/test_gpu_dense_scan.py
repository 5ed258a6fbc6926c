"""GPU parity of the dense scan kernel (2-bit symbols, one segment, several
expected matches per slice): text lengths around its pieces, slices and
chunks, inputs that are 16-byte but not 32-byte aligned, bytes outside the
alphabet, start ranges, prefix entries in shared memory and through L2, every
record format, and texts whose starts all stay pending so that its entry
buffer overflows.  The oracle's whole list is the reference."""
import numpy as np
import pytest
import torch

import workloads
from tests.gpu_util import assert_same, keys_np, oracle_keys, to_device

pytestmark = pytest.mark.gpu

pfac = pytest.importorskip("paper_1704_02272_gb300")

# name: (sigma, patterns, shortest, longest)
SETS = {"four": (4, 300, 3, 24), "four-many": (4, 12000, 4, 40), "three": (3, 80, 3, 18),
        "four-deep": (4, 1500, 5, 60), "singles": (4, 6, 1, 3)}
SIZES = (1, 15, 16, 17, 31, 33, 63, 500, 511, 512, 513, 1023, 1024, 1025, 1039, 1040, 1041, 3000, 90_001)


def make(name, n_bytes, text_sigma=None, plants=None):
    sigma, n, lo, hi = SETS[name]
    return workloads.tiny_case(8800 + len(name), sigma, n, lo, hi, n_bytes, text_sigma=text_sigma,
                               n_plants=n_bytes // 200 if plants is None else plants)


def check(t, w, what, shift=0):
    text, seg = to_device(w)
    if shift:
        moved = torch.empty(text.numel() + shift + 64, dtype=torch.uint8, device=text.device)
        moved = moved[shift:shift + text.numel()]
        moved.copy_(text)
        text = moved
    keys = pfac.match(t, text, seg, capacity=max(1024, 4 * text.numel()))
    torch.cuda.synchronize()
    assert_same(keys_np(keys), oracle_keys(w), what)


@pytest.mark.parametrize("name", sorted(SETS))
def test_sizes_and_alignment(name):
    base = make(name, 64)
    with pfac.Table(base.patterns, base.sigma) as t:
        assert pfac.plan(t)["records_per_slice"] == 512
        for n_bytes in SIZES + (700_003,):
            w = make(name, n_bytes)
            assert w.patterns == base.patterns
            check(t, w, f"{name} {n_bytes}")
            check(t, w, f"{name} {n_bytes} at 16 bytes", shift=16)


@pytest.mark.parametrize("name", ["four", "three", "four-deep"])
def test_bytes_outside_the_alphabet(name):
    w = make(name, 300_007, plants=2000)
    rs = np.random.RandomState(4)
    at = rs.randint(0, w.n_bytes, size=900)
    w.text[at] = rs.randint(w.sigma, 256, size=at.size)
    with pfac.Table(w.patterns, w.sigma) as t:
        check(t, w, name)


@pytest.mark.parametrize("kw", [{}, {"wide_records": True}, {"layout": pfac.LAYOUT_DENSE}],
                         ids=["packed", "wide", "dense"])
def test_record_formats_start_ranges_and_segments(kw):
    w = make("four-deep", 200_000, plants=1500)
    ref = oracle_keys(w)
    text, seg = to_device(w)
    with pfac.Table(w.patterns, 4, **kw) as t:
        for end in (1, 33, 511, 513, 1024, 1025, 100_001, 199_999, 200_000):
            keys = keys_np(pfac.match(t, text, seg, capacity=1 << 20, starts_end=end, position_base=777))
            want = ref[ref < (np.uint64(end) << np.uint64(24))] + (np.uint64(777) << np.uint64(24))
            assert_same(keys, want, f"starts below {end}")
        for opt in ({"scan_kernel": 1}, {"records_per_slice": 32}):
            assert_same(keys_np(pfac.match(t, text, seg, capacity=1 << 20, **opt)), ref, str(opt))
        many = workloads.Workload("segments", 4, w.patterns, w.text,
                                  np.array([0, 7, 90_000, 200_000], dtype=np.uint64))
        check(t, many, "segments")


def test_every_start_pending():
    # a text of one symbol, over patterns that it keeps walking into
    rs = np.random.RandomState(6)
    pats = [bytes(n) for n in (20, 31, 40)] + workloads.uniform_patterns(rs, 300, 4, 3, 12)
    pats = list(dict.fromkeys(pats))
    for n_bytes in (2_000, 400_003):
        w = workloads.Workload("zeros", 4, pats, np.zeros(n_bytes, np.uint8),
                               workloads.single_segment(n_bytes))
        with pfac.Table(pats, 4) as t:
            check(t, w, f"zeros {n_bytes}")
            foreign = workloads.Workload("foreign", 4, pats, np.full(n_bytes, 9, np.uint8),
                                         workloads.single_segment(n_bytes))
            check(t, foreign, f"foreign {n_bytes}")


def test_host_buffers_in_chunks():
    w = make("four", 300_000)
    text = torch.from_numpy(w.text).pin_memory()
    seg = torch.from_numpy(w.seg_offsets.astype(np.int64))
    ref = oracle_keys(w)
    out = torch.zeros(ref.size + 16, dtype=torch.int64).pin_memory()
    with pfac.Table(w.patterns, w.sigma) as t:
        n = pfac.match_host(t, text, seg, out, chunk_bytes=70_000)
    assert_same(out[:n].numpy().view(np.uint64), ref, "host")
