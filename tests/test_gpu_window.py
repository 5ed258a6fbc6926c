"""GPU parity of the window kernel, which takes the calls that leave every
scan choice to the library: pattern sets that lead to each stride, window
form and bit count, at text lengths around its 16-byte pieces, slices and
1,024-byte chunks, below and above the size where the filter moves to shared
memory, on inputs that are 16-byte but not 32-byte aligned, with bytes outside
the alphabet, segments, start ranges, and texts that overflow its entry buffer
or the slices' records.  The oracle's whole list is the reference."""
import numpy as np
import pytest
import torch

import workloads
from tests.gpu_util import assert_same, keys_np, oracle_keys, to_device

pytestmark = pytest.mark.gpu

pfac = pytest.importorskip("paper_1704_02272_gb300")

# name: (sigma, patterns, shortest, longest)
SETS = {
    "bytes-short": (256, 2500, 2, 30),       # patterns that end inside a window
    "bytes-4": (256, 1000, 4, 32),           # stride 2
    "bytes-20": (256, 300, 20, 24),          # long strides over raw bytes
    "bytes-many": (256, 60000, 5, 12),       # several bits per window
    "bytes-9": (200, 400, 9, 14),            # alphabet below its 8-bit range
    "letters": (52, 100, 20, 20),
    "text-64": (64, 3000, 4, 40),
    "protein": (20, 8000, 4, 30),            # five symbols hashed
    "sixteen": (16, 300, 7, 12),
    "five": (5, 150, 10, 20),
    "dna": (4, 3000, 8, 40),                 # 2-bit windows, stride 1
    "dna-long": (4, 200, 24, 60),            # 2-bit windows, long strides
    "three": (3, 100, 12, 30),
}


def make(name, n_bytes, n_segments=1, text_sigma=None, plants=None):
    sigma, n, lo, hi = SETS[name]
    return workloads.tiny_case(7700 + len(name), sigma, n, lo, hi, n_bytes, n_segments=n_segments,
                               n_plants=plants if plants is not None else 20 + n_bytes // 500,
                               text_sigma=text_sigma)


def check(t, w, what, shift=0):
    text, seg = to_device(w)
    if shift:
        room = torch.empty(text.numel() + shift + 64, dtype=torch.uint8, device=text.device)
        moved = room[shift:shift + text.numel()]
        moved.copy_(text)
        text = moved
    keys = pfac.match(t, text, seg)
    torch.cuda.synchronize()
    assert_same(keys_np(keys), oracle_keys(w), what)


@pytest.mark.parametrize("name", sorted(SETS))
def test_sizes_and_alignment(name):
    sigma, n, lo, hi = SETS[name]
    base = make(name, 64)
    with pfac.Table(base.patterns, sigma) as t:
        for n_bytes in (1, 15, 16, 17, 31, 33, 511, 512, 513, 1023, 1024, 1025, 1039, 1040, 1041,
                        2048, 70_001, 1_000_003):
            w = make(name, n_bytes)
            assert w.patterns == base.patterns
            check(t, w, f"{name} {n_bytes}")
            check(t, w, f"{name} {n_bytes} at 16 bytes", shift=16)


@pytest.mark.parametrize("name", sorted(SETS))
def test_shared_memory_filter(name):
    # more slices than the small form takes; segments; unaligned by 16
    sigma = SETS[name][0]
    w = make(name, 5_000_011, n_segments=3000, plants=4000)
    with pfac.Table(w.patterns, sigma) as t:
        check(t, w, name)
        check(t, w, f"{name} at 16 bytes", shift=16)
        one = make(name, 4_194_304 + 16, plants=4000)
        check(t, one, f"{name} one segment")


@pytest.mark.parametrize("name", ["bytes-9", "letters", "protein", "sixteen", "five", "dna",
                                  "dna-long", "three"])
@pytest.mark.parametrize("n_bytes", [40_001, 3_000_001])
def test_bytes_outside_the_alphabet(name, n_bytes):
    sigma = SETS[name][0]
    w = make(name, n_bytes, n_segments=50, plants=3000)
    rs = np.random.RandomState(3)
    at = rs.randint(0, n_bytes, size=n_bytes // 300)
    w.text[at] = rs.randint(sigma, 256, size=at.size)
    with pfac.Table(w.patterns, sigma) as t:
        check(t, w, name)


def test_short_patterns_before_foreign_bytes():
    # patterns shorter than a window, each followed by a byte outside the
    # alphabet or by a segment's end
    rs = np.random.RandomState(5)
    for sigma in (5, 20, 60, 100):
        pats = workloads.uniform_patterns(rs, 30, sigma, 3, 9)
        text = np.full(200_000, 255, dtype=np.uint8)
        cuts, p = [0], 0
        for i in range(12_000):
            q = pats[i % len(pats)]
            text[p:p + len(q)] = np.frombuffer(q, dtype=np.uint8)
            p += len(q)
            if i % 3 == 0:
                cuts.append(p)
            if i % 3 == 1:
                p += 1
        text = text[:p].copy()
        w = workloads.Workload("foreign", sigma, pats, text,
                               np.array(cuts + [p], dtype=np.uint64))
        with pfac.Table(pats, sigma) as t:
            check(t, w, f"sigma {sigma}")


@pytest.mark.parametrize("name", ["bytes-4", "letters", "dna-long", "protein"])
def test_start_ranges_and_offsets(name):
    sigma = SETS[name][0]
    w = make(name, 300_000, n_segments=9, plants=2000)
    ref = oracle_keys(w)
    text, seg = to_device(w)
    with pfac.Table(w.patterns, sigma) as t:
        for end in (1, 16, 511, 513, 1024, 100_000, 299_999, 300_000):
            keys = keys_np(pfac.match(t, text, seg, starts_end=end, position_base=12345))
            want = ref[ref < (np.uint64(end) << np.uint64(24))] + (np.uint64(12345) << np.uint64(24))
            assert_same(keys, want, f"{name} starts below {end}")


def test_entry_buffer_and_records_overflow():
    # every position of the text starts a match: more candidates than the
    # entry buffer holds and more matches than a slice's records
    pats = [b"\x01" * 9, b"\x01" * 12, b"\x02\x01\x01\x01\x01\x01\x01\x01\x01\x03"]
    rs = np.random.RandomState(8)
    pats += workloads.uniform_patterns(rs, 200, 256, 9, 20)
    text = np.full(6_000_017, 1, dtype=np.uint8)
    text[3_000_000:3_500_000] = rs.randint(0, 256, size=500_000, dtype=np.uint8)
    w = workloads.Workload("runs", 256, pats, text, workloads.single_segment(text.size))
    with pfac.Table(pats, 256) as t:
        check(t, w, "runs")
        w2 = workloads.Workload("runs", 256, pats, text[:90_000].copy(),
                                np.array([0, 4, 40_000, 40_005, 90_000], dtype=np.uint64))
        check(t, w2, "runs, small")


def test_dense_layout_and_other_plans_agree():
    for name in ("bytes-4", "letters", "dna", "protein"):
        sigma = SETS[name][0]
        w = make(name, 3_000_007, n_segments=400, plants=5000)
        text, seg = to_device(w)
        ref = oracle_keys(w)
        for layout in (pfac.LAYOUT_COMPRESSED, pfac.LAYOUT_DENSE):
            with pfac.Table(w.patterns, sigma, layout=layout) as t:
                for opt in ({}, {"scan_kernel": 1}, {"resolver": 1}, {"records_per_slice": 32}):
                    assert_same(keys_np(pfac.match(t, text, seg, **opt)), ref, f"{name} {opt}")


def test_graph_replay_on_changed_text():
    w = make("letters", 2_000_001, plants=800)
    v = workloads.tiny_case(99, 52, 1, 20, 20, 2_000_001)
    text, seg = to_device(w)
    with pfac.Table(w.patterns, 52) as t:
        out = torch.zeros(4096, dtype=torch.int64, device=text.device)
        cnt = torch.zeros(1, dtype=torch.int64, device=text.device)
        st = torch.full((1,), 9, dtype=torch.int32, device=text.device)
        ws = torch.empty(pfac.workspace_bytes(t, text.numel(), 1), dtype=torch.uint8, device=text.device)
        pfac.match_async(t, text, seg, out, cnt, st, ws)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            pfac.match_async(t, text, seg, out, cnt, st, ws)
        for data in (v.text, w.text):
            text.copy_(torch.from_numpy(data))
            g.replay()
            torch.cuda.synchronize()
            x = workloads.Workload("g", 52, w.patterns, data, w.seg_offsets)
            assert int(st.item()) == 0
            assert_same(keys_np(out[:int(cnt.item())]), oracle_keys(x), "replay")


@pytest.mark.parametrize("n_bytes", [30_011, 3_000_017])
def test_crowded_filters(n_bytes):
    # sets so large that most words of the filter hold bits and many windows
    # pass: the entry buffer's parts fill up
    for sigma, n, lo, hi in ((17, 200_000, 6, 8), (64, 260_000, 4, 5)):
        w = workloads.tiny_case(7900 + sigma, sigma, n, lo, hi, n_bytes, n_segments=7,
                                n_plants=20 + n_bytes // 500)
        with pfac.Table(w.patterns, sigma) as t:
            check(t, w, f"{sigma} symbols, {n} patterns, {n_bytes} bytes")
