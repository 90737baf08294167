"""Timed cases of the public entry points (bos.orp, bos.sort, bos.Batch) over the range of their use.

A case is one call a program makes with device buffers, a workspace and (for batches) descriptors that it keeps.
Kinds:
  orp, sort    one array through bos.orp / bos.sort, output and workspace kept by the caller;
  merge        bos.sort with the comparison-based (merge) sort after the ORP;
  batch        bos.Batch.run: many arrays given afresh (descriptors written, launched, collected);
  graph        a prepared batch captured once in a CUDA graph: replay and collect.
The outputs are the records themselves, viewed as 64-bit words: bytes moved, no computed numbers.
"""
import numpy as np
import torch

from paper_2008_01765_gb300 import autotune, bos

DEV = "cuda"
KINDS_ONE = ("orp", "sort", "merge")


def listed():
    return [
        # the smallest serving request: launches and latency
        {"name": "sort_4k", "kind": "sort", "n": 1 << 12, "rec": 16, "Z": 512, "dist": "uniform"},
        # a small permutation of 8-byte records
        {"name": "orp_64k_rec8", "kind": "orp", "n": 1 << 16, "rec": 8, "Z": 512, "dist": "uniform"},
        # an ordinary request of ragged size
        {"name": "sort_1m_odd", "kind": "sort", "n": (1 << 20) + 3, "rec": 16, "Z": 512, "dist": "uniform"},
        # few distinct keys: the ties and large groups of a grouping column
        {"name": "sort_16m_dup", "kind": "sort", "n": 1 << 24, "rec": 16, "Z": 512, "dist": "dup1024"},
        # 32-bit keys, ragged
        {"name": "sort_25m_rec8", "kind": "sort", "n": 25_000_003, "rec": 8, "Z": 1024, "dist": "uniform"},
        # a bucket size that is no power of two, ragged
        {"name": "sort_40m_z768", "kind": "sort", "n": 40_000_001, "rec": 16, "Z": 768, "dist": "uniform"},
        # the largest serving request, permutation alone
        {"name": "orp_64m", "kind": "orp", "n": 1 << 26, "rec": 16, "Z": 1024, "dist": "uniform"},
        # the headline sort, at the largest size whose buffers fit the device three times
        {"name": "sort_512m", "kind": "sort", "n": 1 << 29, "rec": 16, "Z": 1024, "dist": "uniform"},
        # the composition with a comparison sort
        {"name": "merge_4m", "kind": "merge", "n": (1 << 22) + 5, "rec": 16, "Z": 512, "dist": "uniform"},
        # one batched launch of the serving loop: 64 small requests, ORP and sort mixed
        {"name": "batch_64_small", "kind": "batch", "arrays": 64, "lo": 12.0, "hi": 16.0, "rec": 16},
        # the batched workload, an eighth of its arrays: 2^10..2^20 records each, one CUDA graph
        {"name": "graph_512", "kind": "graph", "arrays": 512, "lo": 10.0, "hi": 20.0, "rec": 8},
    ]


def draw(rng):
    u = rng.random()
    rec = rng.choice((8, 16))
    if u < 0.7:
        kind = "merge" if u < 0.08 else rng.choice(("orp", "sort", "sort"))
        n = int(2.0 ** rng.uniform(12.0, 24.0 if kind == "merge" else 28.0))
        return {"kind": kind, "n": n | (1 if rng.random() < 0.5 else 0), "rec": rec,
                "Z": rng.choice((256, 512, 512, 768, 1024, 1024, 2048)),
                "dist": rng.choice(("uniform", "uniform", "uniform", "dup1024", "sorted", "equal"))}
    lo = rng.uniform(10.0, 13.0)
    if u < 0.85:
        return {"kind": "batch", "arrays": rng.randint(2, 64), "lo": lo, "hi": rng.uniform(lo + 0.5, 16.0), "rec": rec}
    return {"kind": "graph", "arrays": rng.randint(16, 512), "lo": lo, "hi": rng.uniform(lo + 0.5, 20.0), "rec": rec}


def _sizes(case):
    """Array sizes of a batch: floor(2^U), U uniform in [lo, hi]; a property of the case, not of the seed."""
    rng = np.random.Generator(np.random.PCG64(case["arrays"]))
    return np.floor(np.exp2(rng.uniform(case["lo"], case["hi"], size=case["arrays"]))).astype(np.int64)


def _records(n, rec, dist, seed):
    """n records {key, payload = index} as a flat uint8 CUDA tensor (the distributions of inputs.make_records)."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    dt, lo, hi = (torch.int32, -(1 << 31), (1 << 31) - 1) if rec == 8 else (torch.int64, -(1 << 63), (1 << 63) - 1)
    if dist == "equal":
        key = torch.full((n,), 0x5555555555555555 if rec == 16 else 0x55555555, dtype=dt, device=DEV)
    elif dist == "dup1024":
        table = torch.randint(lo, hi, (1024,), generator=g, dtype=dt, device=DEV)
        key = table[torch.randint(0, 1024, (n,), generator=g, device=DEV)]
    else:
        key = torch.randint(lo, hi, (n,), generator=g, dtype=dt, device=DEV)
        if dist == "sorted":  # ascending as unsigned keys
            key = key.sort().values
            key = torch.cat([key[key >= 0], key[key < 0]])
    r = torch.empty((n, 2), dtype=dt, device=DEV)
    r[:, 0] = key
    r[:, 1] = torch.arange(n, dtype=dt, device=DEV)
    return r.view(torch.uint8).reshape(-1)


def prepare(case, seed):
    kind, rec = case["kind"], case["rec"]
    if kind in KINDS_ONE:
        n = case["n"]
        x = _records(n, rec, case["dist"], seed)
        flags = bos.FLAG_MERGE_SORT if kind == "merge" else 0
        p = bos.params(rec, case["Z"], seed, flags=flags)
        return {"kind": kind, "x": x, "out": torch.empty_like(x), "rec": rec, "Z": case["Z"], "seed": seed + 1,
                "flags": flags, "ws": bos.alloc_workspace(bos.workspace_bytes(n, p), x.device)}
    sizes = _sizes(case)
    offs = np.zeros(sizes.size + 1, dtype=np.uint64)
    np.cumsum(sizes, out=offs[1:])
    x = _records(int(offs[-1]), rec, "uniform", seed)
    out = torch.empty_like(x)
    seeds = np.arange(1, sizes.size + 1, dtype=np.uint64) + np.uint64(seed * 1000)
    ops = np.ones(sizes.size, dtype=np.uint8)
    if kind == "batch":
        ops[::2] = 0
        Zs = np.full(sizes.size, 512, dtype=np.uint32)
    else:
        Zs = np.asarray(autotune.z_array(sizes, rec), dtype=np.uint32)
    b = bos.Batch(x, out, offs, seeds, ops, bos.params(rec, 512, 0), Zs=Zs)
    graph = None
    if kind == "graph":
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        b.prepare(stream)
        b.enqueue(stream)
        b.collect(stream)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream, capture_error_mode="relaxed"):
            b.enqueue(stream)
        torch.cuda.current_stream().wait_stream(stream)
    return {"kind": kind, "batch": b, "graph": graph}


def run(state):
    if state["kind"] in KINDS_ONE:
        fn = bos.orp if state["kind"] == "orp" else bos.sort
        out, info = fn(state["x"], state["rec"], Z=state["Z"], seed=state["seed"], flags=state["flags"],
                       out=state["out"], workspace=state["ws"])
        return {"out": out.view(torch.int64), "attempts": int(info.attempts)}
    b = state["batch"]
    if state["graph"] is not None:
        state["graph"].replay()
        attempts = b.collect()
    else:
        attempts = b.run()
    return {"out": b.out.view(torch.int64), "attempts": attempts}


def work(case):
    n = case["n"] if case["kind"] in KINDS_ONE else int(_sizes(case).sum())
    return {"bytes": 2.0 * n * case["rec"], "flops": 0.0}  # every record read once and written once

