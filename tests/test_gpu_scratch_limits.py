"""Inputs and requests at the edge of a fixed scratch size: what fits a plan
with 32 records a slice and no entry or queue buffer is taken, whatever the
library would choose with more room, and gives the oracle's keys."""
import numpy as np
import pytest
import torch

import workloads
from tests.gpu_util import assert_same, keys_np, oracle_keys, to_device

pytestmark = pytest.mark.gpu

pfac = pytest.importorskip("paper_1704_02272_gb300")

SCRATCH = 32 << 20


def up(x):
    return (x + 255) & ~255


def scratch_of(slices, segments):
    """The least scratch a call needs: a header, per slice the counts, the
    offset, the overflow list and 32 records, the sums of chunks of 1,024
    slices, and with several segments an index per slice."""
    return (256 + up(4 * slices) + 2 * up(8 * slices) + up(16 * ((slices + 1023) // 1024)) + up(4 * slices) +
            up(256 * slices) + (up(4 * slices) if segments > 1 else 0))


@pytest.mark.parametrize("segments", [1, 2])
def test_noalloc_takes_what_its_array_holds(segments):
    slices = max(s for s in range(100_000, 130_000) if scratch_of(s, segments) <= SCRATCH)
    n = slices * 512
    rs = np.random.RandomState(1)
    pats = workloads.uniform_patterns(rs, 40, 52, 20, 20)
    text = rs.randint(0, 52, size=n).astype(np.uint8)
    seg = np.array([0, n] if segments == 1 else [0, n // 2 + 3, n], dtype=np.uint64)
    for at in rs.randint(0, n - 20, size=500):
        text[at:at + 20] = np.frombuffer(pats[at % 40], dtype=np.uint8)
    w = workloads.Workload("edge", 52, pats, text, seg)
    ref = oracle_keys(w)
    text_d, seg_d = to_device(w)
    with pfac.Table(pats, 52) as t:
        out = torch.zeros(ref.size + 16, dtype=torch.int64, device="cuda")
        cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
        st = torch.full((1,), 9, dtype=torch.int32, device="cuda")
        pfac.match_noalloc(t, text_d, seg_d, out, cnt, st)
        torch.cuda.synchronize()
        assert int(st.item()) == 0
        assert_same(keys_np(out[:int(cnt.item())]), ref, "edge")


@pytest.mark.parametrize("kind", ["letters", "dense"])
def test_server_takes_what_its_pool_holds(kind):
    rs = np.random.RandomState(2)
    n = 4 << 20
    if kind == "letters":
        w = workloads.tiny_case(71, 52, 100, 20, 20, n, n_plants=2000)
        records = 32
    else:
        w = workloads.tiny_case(72, 4, 300, 3, 24, n)
        records = 512
    ref = oracle_keys(w)
    slices = n // 512
    # input, offsets, scratch, count and status, and the first output buffer
    room = n + 256 + scratch_of(slices, 1) + (records - 32) * 8 * slices + 256 + n
    text = torch.from_numpy(w.text).pin_memory()
    seg = torch.from_numpy(w.seg_offsets.astype(np.int64)).pin_memory()
    with pfac.Table(w.patterns, w.sigma) as t:
        with pfac.Server(t, n_slots=2, device_bytes=room, max_request_bytes=n) as s:
            ids = [s.submit(text, seg) for _ in range(3)]
            for i in ids:
                r = s.wait(i, timeout=60)
                assert r["status"] == 0
                assert_same(np.asarray(r["keys"]).view(np.uint64), ref, f"request {i}")
                s.release(i)
