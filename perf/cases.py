"""The calls that performance work on this library is measured on.

Each case is one match call (or match and verify) through the package's
public entry points, on inputs of the shapes that the benchmark, the tests and
the paper's evaluation use: uniform texts over alphabets of 4 to 256 symbols,
DNA-like texts with planted occurrences, network packets matched against
signature-like patterns, and the requests of a serving loop.  Texts and
patterns are drawn from the seed alone; planted occurrences never overlap, so
the inputs do not depend on the order of writes.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1704_02272_gb300 as pfac

MIB = 1 << 20


def listed() -> list:
    return [
        # One small packet batch against a large signature set, the call of a
        # latency-bound inspection loop: launches and fixed costs count.
        _case("packets-64KiB", "packets", 256, 20000, 65536, plants=0.005),
        # The plain workload (bytes, 1,000 patterns of 4 to 32 symbols, 1 MiB)
        # through the synchronous call that allocates its own workspace.
        _case("plain-1MiB", "uniform", 256, 1000, MIB, lo=4, hi=32, plants=2000 / MIB, call="match"),
        # One request of the serving workload: about two thousand packets of 64
        # to 9,000 bytes against 50,000 signatures.
        _case("request-9MB", "requests", 256, 50000, 9_283_507, plants=0.005),
        # IDS packets at full size: many short packets, short patterns that
        # really occur, 20,000 signatures.
        _case("ids-1GiB", "packets", 256, 20000, 1024 * MIB, plants=0.005),
        # DNA, the benchmark's default, with the autotuned plan it uses.
        _case("dna-256MiB", "uniform", 4, 10000, 256 * MIB, lo=8, hi=64, plants=0.001, tuned=True),
        # DNA of an odd size in pinned host memory, text in and keys out, with
        # the library's own plan.
        _case("dna-host-80MB", "uniform", 4, 10000, 80_000_003, lo=8, hi=64, plants=0.001, call="host"),
        # A sweep cell where about one position in twelve matches: emission and
        # ordering of the keys.
        _case("sweep-4x1k", "uniform", 4, 1000, 128 * MIB, lo=4, hi=64),
        # Protein-sized alphabet, medium pattern set.
        _case("sweep-20x10k", "uniform", 20, 10000, 256 * MIB, lo=4, hi=64),
        # Text-sized alphabet, the largest pattern count of the sweep.
        _case("sweep-64x100k", "uniform", 64, 100000, 128 * MIB, lo=4, hi=64),
        # All bytes, 1,000 patterns, 512 MiB: the sweep cell nearest to the
        # memory's rate.
        _case("sweep-256x1k", "uniform", 256, 1000, 512 * MIB, lo=4, hi=64),
        # The paper's throughput shape (52 letters, patterns of 20 symbols,
        # 100 MiB and an odd tail).
        _case("letters-100", "uniform", 52, 100, 100 * MIB + 77, lo=20, hi=20, plants=1000 / (100 * MIB)),
        # Prefix matching: candidates from a trie cut at 4 symbols, then the
        # verification that keeps the exact ones.
        _case("prefix-verify-64MiB", "packets", 256, 20000, 64 * MIB, plants=0.005, truncate=4,
              call="verify"),
    ]


def _case(name, shape, sigma, patterns, n_bytes, lo=2, hi=256, plants=0.0, call="async", tuned=False,
          truncate=0):
    return {"name": name, "shape": shape, "sigma": sigma, "patterns": patterns, "bytes": n_bytes,
            "lo": lo, "hi": hi, "plants": plants, "call": call, "tuned": tuned, "truncate": truncate}


def draw(rng) -> dict:
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("packets", "plain", "requests", "dna", "sweep", "sweep", "letters", "prefix"))
    if kind == "packets":
        c = _case("", "packets", 256, log(1000, 50000), log(1 << 14, 512 * MIB), plants=0.005)
    elif kind == "plain":
        c = _case("", "uniform", 256, log(100, 10000), log(1 << 14, 64 * MIB), lo=4, hi=32,
                  plants=2000 / MIB, call="match")
    elif kind == "requests":
        c = _case("", "requests", 256, log(5000, 50000), log(1 << 14, 19_000_000), plants=0.005)
    elif kind == "dna":
        c = _case("", "uniform", 4, log(1000, 20000), log(1 << 16, 256 * MIB), lo=8, hi=64,
                  plants=0.001, call=rng.choice(("async", "async", "host")))
        if c["call"] == "host":
            c["bytes"] = min(c["bytes"], 80_000_003)
    elif kind == "sweep":
        sigma = rng.choice((4, 20, 64, 256))
        n = log(1000, 3000 if sigma == 4 else 100000)
        top = {4: 48, 20: 128, 64: 128, 256: 256}[sigma]
        c = _case("", "uniform", sigma, n, log(1 << 16, top * MIB), lo=4, hi=64)
    elif kind == "letters":
        c = _case("", "uniform", 52, log(1, 1000), log(1 << 16, 100 * MIB), lo=20, hi=20, plants=1e-5)
    else:
        c = _case("", "packets", 256, log(1000, 20000), log(1 << 16, 64 * MIB), plants=0.005,
                  truncate=rng.choice((3, 4, 6, 8)), call="verify")
    del c["name"]
    return c


def _patterns(case, rs) -> list:
    """Distinct patterns: uniform lengths in [lo, hi] over the alphabet, or,
    for packets, signature-like ones (log-normal lengths with median 12, three
    of five printable)."""
    n, sigma = case["patterns"], case["sigma"]
    if case["shape"] == "uniform":
        lens = rs.randint(case["lo"], case["hi"] + 1, size=n)
        flat = rs.randint(0, sigma, size=int(lens.sum()), dtype=np.uint8)
    else:
        lens = np.clip(np.rint(rs.lognormal(math.log(12.0), 0.75, size=n)), case["lo"],
                       case["hi"]).astype(np.int64)
        flat = rs.randint(0, 256, size=int(lens.sum()), dtype=np.uint8)
        printable = np.repeat(rs.random_sample(n) < 0.6, lens)
        flat[printable] = 0x20 + flat[printable] % 95
    ends = np.cumsum(lens)
    raw = flat.tobytes()
    return list(dict.fromkeys(raw[e - m:e] for e, m in zip(ends.tolist(), lens.tolist())))


def _segments(case, rs) -> np.ndarray:
    """Segment offsets: one segment, IDS packets (40% of 64 to 128 bytes, 60%
    of 1,000 to 1,500) or a request's packets (64 to 9,000 bytes)."""
    n = case["bytes"]
    if case["shape"] == "uniform":
        return np.array([0, n], dtype=np.int64)
    if case["shape"] == "packets":
        m = n // 700 + 64
        lens = np.where(rs.random_sample(m) < 0.4, rs.randint(64, 129, size=m),
                        rs.randint(1000, 1501, size=m))
    else:
        lens = rs.randint(64, 9001, size=n // 4000 + 64)
    ends = np.cumsum(lens)
    return np.concatenate([[0], ends[ends < n], [n]]).astype(np.int64)


def _plant(case, rs, text, seg, pats):
    """Writes occurrences of random patterns at places that do not overlap:
    one in each of n equal slots of a uniform text, or one in a share of the
    packets."""
    n = case["bytes"]
    if case["shape"] == "uniform":
        count = int(round(case["plants"] * n))
        slot = max(n // max(count, 1), case["hi"])
        start = np.arange(min(count, n // slot), dtype=np.int64) * slot
        room = np.full(start.shape, slot, dtype=np.int64)
    else:
        pick = np.flatnonzero(rs.random_sample(len(seg) - 1) < case["plants"])
        start, room = seg[pick], seg[pick + 1] - seg[pick]
    if not len(start):
        return 0
    ids = rs.randint(0, len(pats), size=len(start))
    lens = np.array([len(p) for p in pats], dtype=np.int64)[ids]
    fits = lens <= room
    start, room, ids, lens = start[fits], room[fits], ids[fits], lens[fits]
    at = start + (rs.random_sample(len(start)) * (room - lens + 1)).astype(np.int64)
    total = int(lens.sum())
    if total:
        inside = np.arange(total, dtype=np.int64) - np.repeat(np.cumsum(lens) - lens, lens)
        where = torch.from_numpy(np.repeat(at, lens) + inside).to(text.device)
        what = np.frombuffer(b"".join(pats[j] for j in ids.tolist()), dtype=np.uint8)
        text[where] = torch.from_numpy(what.copy()).to(text.device)
    return len(start)


def _density(case) -> float:
    """Expected matches per position of a uniform text, from the case alone."""
    n, sigma, cut = case["patterns"], case["sigma"], case["truncate"] or 1 << 30
    if case["shape"] == "uniform":
        lens = range(case["lo"], case["hi"] + 1)
        return sum(n / len(lens) * float(sigma) ** -min(m, cut) for m in lens)

    def below(x):
        return 0.5 * (1.0 + math.erf((math.log(x) - math.log(12.0)) / 0.75 / math.sqrt(2.0)))

    share = {m: below(m + 0.5) - (below(m - 0.5) if m > case["lo"] else 0.0) for m in range(case["lo"], 12)}
    rest = 1.0 - sum(share.values())
    return n * (sum(s * 256.0 ** -min(m, cut) for m, s in share.items()) + rest * 256.0 ** -min(12, cut))


def _text(case, seed, pats, rs, seg):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    text = torch.randint(0, case["sigma"], (case["bytes"],), dtype=torch.uint8, device="cuda", generator=g)
    _plant(case, rs, text, seg, pats)
    return text


def prepare(case, seed) -> dict:
    rs = np.random.RandomState(seed & 0x7FFFFFFF)
    pats = _patterns(case, rs)
    seg_host = _segments(case, rs)
    text = _text(case, seed, pats, rs, seg_host)
    seg = torch.from_numpy(seg_host).to("cuda")
    table = pfac.Table(pats, case["sigma"], truncate_depth=case["truncate"])
    if case["tuned"]:
        sample = text[:min(case["bytes"], 128 * MIB)]
        pfac.autotune(table, sample, pfac.single_segment(sample.numel(), "cuda"))
    state = {"call": case["call"], "table": table, "text": text, "seg": seg}
    # room for the keys: the expected number and a good margin
    cap = int(1.1 * (_density(case) * case["bytes"] + 2.0 * _planted(case))) + 4096
    where = "cpu" if case["call"] == "host" else "cuda"
    state["out"] = torch.zeros(cap, dtype=torch.int64, device=where)
    if case["call"] == "host":
        state["text"] = text.to("cpu").pin_memory()
        state["seg"] = torch.from_numpy(seg_host).pin_memory()
        state["out"] = state["out"].pin_memory()
    else:
        state["count"] = torch.zeros(1, dtype=torch.int64, device="cuda")
    if case["call"] == "verify":
        state["exact"] = torch.zeros(cap, dtype=torch.int64, device="cuda")
    if case["call"] == "async":
        n_seg = seg.numel() - 1
        state["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
        state["workspace"] = torch.empty(pfac.workspace_bytes(table, text.numel(), n_seg),
                                         dtype=torch.uint8, device="cuda")
    return state


def run(state):
    """The keys are the first count entries of their buffer; what follows them
    stays as prepare left it."""
    t, text, seg, out = state["table"], state["text"], state["seg"], state["out"]
    if state["call"] == "host":
        return {"keys": out, "count": pfac.match_host(t, text, seg, out)}
    if state["call"] == "async":
        pfac.match_async(t, text, seg, out, state["count"], state["status"], state["workspace"])
        return {"keys": out, "count": state["count"], "status": state["status"]}
    n = pfac.match_into(t, text, seg, out)
    if state["call"] == "verify":
        pfac.verify_into(t, text, seg, out[:n], state["exact"], state["count"])
        return {"candidates": out, "keys": state["exact"], "count": state["count"]}
    return {"keys": out, "count": n}


def _planted(case) -> float:
    """About how many occurrences are planted."""
    n = case["bytes"]
    return case["plants"] * {"uniform": n, "packets": n / 788.0, "requests": n / 4532.0}[case["shape"]]


def work(case) -> dict:
    """The text and the segment offsets read once, the keys written once (and
    for prefix matching the candidates written and read)."""
    n = case["bytes"]
    segs = {"uniform": 1, "packets": n / 788.0, "requests": n / 4532.0}[case["shape"]]
    keys = 8.0 * (_density({**case, "truncate": 0}) * n + _planted(case))
    if case["truncate"]:
        keys += 16.0 * (_density(case) * n + _planted(case))
    return {"bytes": n + 8.0 * (segs + 1.0) + keys, "flops": 0.0}
