"""GPU parity of the dense scan kernel at the input's last whole 16-byte
piece: occurrences whose first symbols end right there and go on in the
remainder, whose symbols the kernel has not loaded, also where the input is a
chunk of a longer text.  The oracle's whole list is the reference."""
import numpy as np
import pytest
import torch

import workloads
from tests.gpu_util import assert_same, keys_np, oracle_keys, to_device

pytestmark = pytest.mark.gpu

pfac = pytest.importorskip("paper_1704_02272_gb300")


def going_on(pats, k, longest):
    """Patterns of k + 1 to `longest` symbols that no other pattern is a prefix
    of, and whose first k symbols no pattern continues with a 0."""
    every = set(pats)
    heads = {p[:k + 1] for p in pats}
    return [p for p in pats if k < len(p) <= longest and p[k] != 0 and p[:k] + b"\0" not in heads and
            not any(p[:i] in every for i in range(1, k + 1))]


def patterns(n, lo, hi):
    return workloads.uniform_patterns(np.random.RandomState(41), n, 4, lo, hi)


@pytest.mark.parametrize("kw", [{}, {"wide_records": True}, {"layout": pfac.LAYOUT_DENSE}],
                         ids=["packed", "wide", "dense"])
def test_occurrences_into_the_remainder(kw):
    pats = patterns(600, 3, 24)
    rs = np.random.RandomState(17)
    with pfac.Table(pats, 4, **kw) as t:
        p = pfac.plan(t)
        k = p["prefix_depth"]
        assert p["records_per_slice"] == 512
        tried = 0
        for whole in (16, 496, 512, 1008, 1024, 1040, 30_000):
            for rest in range(16):
                for q in going_on(pats, k, k + rest)[:4] + going_on(pats, k, k + rest)[-4:]:
                    if whole < k:
                        continue
                    text = rs.randint(0, 4, size=whole + rest).astype(np.uint8)
                    text[whole - k:whole - k + len(q)] = np.frombuffer(q, dtype=np.uint8)
                    w = workloads.Workload("tail", 4, pats, text, workloads.single_segment(text.size))
                    d, seg = to_device(w)
                    keys = pfac.match(t, d, seg, capacity=8 * text.size)
                    assert_same(keys_np(keys), oracle_keys(w), f"{whole} + {rest}, {len(q)} symbols")
                    tried += 1
        assert tried > 200


def test_occurrences_over_a_chunk_border():
    pats = patterns(400, 3, 14)  # halos below 16 bytes
    rs = np.random.RandomState(18)
    with pfac.Table(pats, 4) as t:
        p = pfac.plan(t)
        k, chunk = p["prefix_depth"], 1024
        assert p["records_per_slice"] == 512
        cross = going_on(pats, k, 14)
        assert cross
        text = rs.randint(0, 4, size=chunk * (len(cross) + 1) + 5).astype(np.uint8)
        for i, q in enumerate(cross):
            at = chunk * (i + 1) - k
            text[at:at + len(q)] = np.frombuffer(q, dtype=np.uint8)
        w = workloads.Workload("chunks", 4, pats, text, workloads.single_segment(text.size))
        ref = oracle_keys(w)
        out = torch.zeros(ref.size + 16, dtype=torch.int64).pin_memory()
        n = pfac.match_host(t, torch.from_numpy(text).pin_memory(),
                            torch.from_numpy(w.seg_offsets.astype(np.int64)), out, chunk_bytes=chunk)
    assert_same(out[:min(n, out.numel())].numpy().view(np.uint64), ref, "chunks")
