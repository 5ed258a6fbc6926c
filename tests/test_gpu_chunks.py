"""GPU parity where the key-count scan changes the units of its chunks (8, 16
or 32 a chunk in small calls, more in large ones), for the window, queued and
dense scan kernels, over texts with empty, sparse and full slices.  The
oracle's whole list is the reference."""
import numpy as np
import pytest
import torch

import workloads
from tests.gpu_util import assert_same, keys_np, oracle_keys, to_device

pytestmark = pytest.mark.gpu

pfac = pytest.importorskip("paper_1704_02272_gb300")

# slices: one chunk and its neighbours; the most of 8, 16 and 32 units each
SLICES = (1, 7, 8, 9, 1216 * 8, 1216 * 8 + 1, 1216 * 16, 1216 * 16 + 1, 65536, 65537)


@pytest.mark.parametrize("slices", SLICES)
def test_chunk_edges(slices):
    n = slices * 512 - 5
    rs = np.random.RandomState(slices)
    pats = [b"\x07" * 9] + workloads.uniform_patterns(rs, 300, 256, 4, 20)
    text = rs.randint(0, 256, size=n, dtype=np.uint8)
    for at in (0, n // 3, n - min(n, 3000)):  # full slices
        text[at:at + 2500] = 7
    for i in rs.randint(0, max(1, n - 20), size=n // 400):
        p = np.frombuffer(pats[1 + i % 300], dtype=np.uint8)
        text[i:i + p.size] = p[:max(0, n - i)]
    w = workloads.Workload("chunks", 256, pats, text, workloads.single_segment(n))
    ref = oracle_keys(w)
    text_d, seg = to_device(w)
    with pfac.Table(pats, 256) as t:
        for opt in ({}, {"scan_kernel": 1}):
            keys = pfac.match(t, text_d, seg, capacity=ref.size + 64, **opt)
            assert_same(keys_np(keys), ref, f"{slices} slices {opt}")
            end = max(1, n - 4100)  # fewer units than the workspace is for
            keys = pfac.match(t, text_d, seg, capacity=ref.size + 64, starts_end=end, **opt)
            assert_same(keys_np(keys), ref[ref < (np.uint64(end) << np.uint64(24))], f"{slices} slices {opt}, starts")


@pytest.mark.parametrize("slices", SLICES[:-2])
def test_chunk_edges_dense_scan(slices):
    w = workloads.tiny_case(61, 4, 300, 3, 24, slices * 512 - 5)
    text, seg = to_device(w)
    ref = oracle_keys(w)
    with pfac.Table(w.patterns, 4) as t:
        assert_same(keys_np(pfac.match(t, text, seg, capacity=ref.size + 64)), ref, f"{slices} slices")
