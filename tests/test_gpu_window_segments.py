"""GPU parity of the window kernel where its entry buffer is full and the text
has many segments: walks inside the scan take their segment ends from what the
launch before wrote, so neither what the workspace held nor another call on the
GPU changes a result.  The oracle's whole list is the reference."""
import numpy as np
import pytest
import torch

import workloads
from tests.gpu_util import assert_same, keys_np, oracle_keys, to_device

pytestmark = pytest.mark.gpu

pfac = pytest.importorskip("paper_1704_02272_gb300")


class Call:
    """One asynchronous call's buffers."""

    def __init__(self, t, w, ref, stream=None):
        self.t, self.ref, self.stream = t, ref, stream
        self.text, self.seg = to_device(w)
        dev = self.text.device
        self.out = torch.zeros(ref.size + 16, dtype=torch.int64, device=dev)
        self.cnt = torch.zeros(1, dtype=torch.int64, device=dev)
        self.st = torch.full((1,), 9, dtype=torch.int32, device=dev)
        self.ws = torch.empty(pfac.workspace_bytes(t, w.n_bytes, self.seg.numel() - 1),
                              dtype=torch.uint8, device=dev)

    def run(self):
        pfac.match_async(self.t, self.text, self.seg, self.out, self.cnt, self.st, self.ws,
                         stream=self.stream)

    def check(self, what):
        assert int(self.st.item()) == 0, what
        n = int(self.cnt.item())
        assert_same(keys_np(self.out[:min(n, self.out.numel())]), self.ref, what)
        assert n == self.ref.size, what


def runs(n_bytes, mean_len, seed):
    """Every position starts a match that a segment's end can cut short."""
    rs = np.random.RandomState(seed)
    pats = [b"\x01" * 9, b"\x01" * 12] + workloads.uniform_patterns(rs, 200, 256, 9, 20)
    text = np.full(n_bytes, 1, dtype=np.uint8)
    lens = rs.randint(0, 2 * mean_len + 1, size=n_bytes // mean_len + 8)
    ends = np.cumsum(lens)
    seg = np.concatenate([[0], ends[ends < n_bytes], [n_bytes]]).astype(np.uint64)
    return workloads.Workload("runs", 256, pats, text, seg)


# below and above the size where the filter moves to shared memory; offsets so
# many that they are read in order, and so few that they are searched
@pytest.mark.parametrize("n_bytes", [200_003, 3_500_017])
@pytest.mark.parametrize("mean_len", [15, 700, 60_000])
def test_full_entry_buffer_over_a_used_workspace(n_bytes, mean_len):
    w = runs(n_bytes, mean_len, 5)
    other = runs(n_bytes, 3 * mean_len, 6)
    with pfac.Table(w.patterns, 256) as t:
        c = Call(t, w, oracle_keys(w))
        oth = torch.from_numpy(other.seg_offsets.astype(np.int64)).to(c.text.device)
        for fill in (0x00, 0x01, 0xFF, None):
            if fill is not None:
                c.ws.fill_(fill)
            elif oth.numel() <= c.seg.numel():  # another call's indices
                pfac.match_async(t, c.text, oth, c.out, c.cnt, c.st, c.ws)
            c.run()
            torch.cuda.synchronize()
            c.check(f"workspace filled with {fill}")


def test_calls_on_two_streams():
    # 50,000 signatures: more starts pass the filter than the buffer holds, on
    # printable text many more
    w = workloads.config3(n_bytes=6 << 20, n_patterns=50000)
    rs = np.random.RandomState(2)
    v = workloads.Workload("printable", 256, w.patterns, 0x20 + rs.randint(0, 95, size=w.n_bytes).astype(np.uint8),
                           w.seg_offsets)
    with pfac.Table(w.patterns, 256) as t:
        ref = [oracle_keys(w), oracle_keys(v)]
        calls = [Call(t, x, r, torch.cuda.Stream()) for x, r in ((w, ref[0]), (v, ref[1])) for _ in range(2)]
        torch.cuda.synchronize()
        for _ in range(4):
            for c in calls:
                with torch.cuda.stream(c.stream):
                    c.ws.fill_(0xFF)
                    c.out.zero_()
                    c.run()
            torch.cuda.synchronize()
            for i, c in enumerate(calls):
                c.check(f"call {i}")
