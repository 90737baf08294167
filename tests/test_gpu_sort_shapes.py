"""The sort kernels at the sizes and key shapes where they change form: range classes of the on-chip sort
and their edges, crowded bins (LSD passes in shared memory), in-place ranges and LSD arrays of a batch,
and streaming / packed-tile passes of a batch next to the one-CTA-per-subproblem ones. Bit-exact against
the oracle, so no tolerance is involved."""
import numpy as np
import pytest

import oracle
from paper_2008_01765_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bos():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2008_01765_gb300 import _build
    _build.build()
    from paper_2008_01765_gb300 import bos as b
    b.lib()
    return b


def _keys(n, rec_bytes, shape, seed):
    recs = inputs.make_records(n, rec_bytes, "uniform", seed=seed)
    kt = recs["key"].dtype.type
    bits = recs["key"].dtype.itemsize * 8
    k = recs["key"].copy()
    rng = np.random.default_rng(seed)
    if shape == "clusters":  # uniform top 16 bits, the bits below from three values: crowded bins, ties
        low = rng.integers(0, 1 << (bits - 17), size=3, dtype=np.uint64).astype(kt)
        k = ((k >> kt(bits - 16)) << kt(bits - 16)) | low[rng.integers(0, 3, size=n)]
    elif shape == "two":  # two distinct keys
        k = np.where(rng.integers(0, 2, size=n) == 1, kt(1 << (bits - 1)), kt(7))
    elif shape == "equal":
        k[:] = kt(42)
    elif shape == "low":  # only the low byte varies
        k = k & kt(255)
    elif shape == "extremes":  # the smallest and the largest key among uniform ones
        k[::3] = kt(0)
        k[1::3] = np.iinfo(kt).max
    elif shape == "span":  # keys around a power of two: ranges that cross the top digits' borders
        k = (kt(1 << (bits - 1)) - kt(n // 2) + np.arange(n).astype(kt))[rng.permutation(n)]
    recs["key"] = k
    return recs


# the largest record counts of the range classes (16- and 8-byte records) and one more
EDGES = [(255, 16), (256, 16), (257, 8), (1056, 16), (1057, 8), (2112, 16), (2113, 16), (4352, 16), (4353, 16),
         (6656, 8), (6657, 8), (9216, 16), (9217, 16), (14848, 8), (14849, 8), (19456, 16), (28672, 8)]


@pytest.mark.parametrize("n,rec_bytes", EDGES)
def test_range_class_edges(bos, n, rec_bytes):
    for shape in ("uniform", "clusters", "two", "span"):
        recs = _keys(n, rec_bytes, shape, seed=n)
        ref, _ = oracle.sort(recs, 512, 5, method=oracle.CLOSED)
        out, info = bos.sort(bos.to_device(recs), rec_bytes, Z=512, seed=5)
        np.testing.assert_array_equal(bos.to_host(out, recs.dtype), ref, err_msg=shape)


# 4096-record tiles of a partition or LSD pass: the look-back's steps (7 single words, then one for eight
# tiles, 64 tiles a window) and ragged last tiles
@pytest.mark.parametrize("tiles,extra,rec_bytes", [(7, 0, 16), (7, 1, 8), (8, 1, 16), (9, -1, 16), (16, 0, 8), (63, 5, 16),
                                                   (72, 31, 16), (73, 0, 8), (137, -33, 16)])
def test_partition_tiles(bos, tiles, extra, rec_bytes):
    n = 4096 * tiles + extra
    for shape in ("uniform", "two", "low"):  # partitions; few and many values a digit in the LSD passes
        recs = _keys(n, rec_bytes, shape, seed=n)
        ref, _ = oracle.sort(recs, 512, 7, method=oracle.CLOSED)
        out, _ = bos.sort(bos.to_device(recs), rec_bytes, Z=512, seed=7)
        np.testing.assert_array_equal(bos.to_host(out, recs.dtype), ref, err_msg=shape)


# 4096-record runs and 2048-record chunks of the merge sort: ragged runs, lone left runs, ties across runs
@pytest.mark.parametrize("n,rec_bytes", [(7, 16), (4095, 16), (4096, 8), (4097, 16), (8193, 8), (12287, 16), (14336, 16),
                                         (65 * 4096 + 2049, 8), (65 * 4096 + 2049, 16)])
def test_merge_runs(bos, n, rec_bytes):
    for shape in ("uniform", "two", "equal", "extremes"):
        recs = _keys(n, rec_bytes, shape, seed=n)
        ref, _ = oracle.sort(recs, 512, 11, method=oracle.CLOSED)
        out, _ = bos.sort(bos.to_device(recs), rec_bytes, Z=512, seed=11, flags=bos.FLAG_MERGE_SORT)
        np.testing.assert_array_equal(bos.to_host(out, recs.dtype), ref, err_msg=shape)


@pytest.mark.parametrize("n,rec_bytes,shape", [
    (200001, 16, "clusters"), (200001, 8, "clusters"), (1 << 20, 16, "span"), (300007, 8, "span"), (100003, 16, "extremes"),
    (100003, 8, "low"), ((1 << 23) + 1, 16, "clusters"), (1 << 23, 8, "clusters"),
])
def test_ranges_of_skewed_keys(bos, n, rec_bytes, shape):
    recs = _keys(n, rec_bytes, shape, seed=3)
    ref, _ = oracle.sort(recs, 512, 9, method=oracle.CLOSED)
    out, _ = bos.sort(bos.to_device(recs), rec_bytes, Z=512, seed=9)
    np.testing.assert_array_equal(bos.to_host(out, recs.dtype), ref)


def test_8_byte_records_on_odd_addresses(bos):
    # input and output aligned to the record only: the bulk copies of the passes and ranges start inside
    import torch
    n = 70001
    recs = _keys(n, 8, "uniform", seed=8)
    buf, obuf = (torch.zeros(n * 8 + 16, dtype=torch.uint8, device="cuda") for _ in range(2))
    x, out = buf[8:8 + n * 8], obuf[8:8 + n * 8]
    x.copy_(bos.to_device(recs))
    ref, _ = oracle.sort(recs, 512, 4, method=oracle.CLOSED)
    bos.sort(x, 8, Z=512, seed=4, out=out)
    np.testing.assert_array_equal(bos.to_host(out.clone(), recs.dtype), ref)
    assert int(obuf[:8].sum()) == 0 and int(obuf[8 + n * 8:].sum()) == 0


@pytest.mark.parametrize("rec_bytes", [8, 16])
def test_batch_of_mixed_shapes(bos, rec_bytes):
    # every key shape at sizes on both sides of the batched rules, bucket sizes the streaming passes take and
    # ones they do not, ORP and sort; then the same batch replayed from a CUDA graph
    import torch
    shapes = ["uniform", "clusters", "two", "equal", "low", "extremes", "span"]
    sizes = [1, 0, 2112, 2113, 4096, 9216, 9217, 16384, 30000, 65536, 100003, 1 << 18, 3000, 20000]
    Zs = np.array([512, 512, 512, 64, 100, 512, 1024, 2048, 96, 512, 256, 1024, 768, 4096 if rec_bytes == 8 else 2048],
                  dtype=np.uint32)
    parts = [_keys(n, rec_bytes, shapes[j % len(shapes)], seed=j + 1) for j, n in enumerate(sizes)]
    recs = np.concatenate(parts)
    offs = np.zeros(len(sizes) + 1, dtype=np.uint64)
    np.cumsum(sizes, out=offs[1:])
    for rot in (0, 1):
        ops = ((np.arange(len(sizes)) + rot) % 3 != 0).astype(np.uint8)
        seeds = np.arange(11, 11 + len(sizes), dtype=np.uint64)
        x = bos.to_device(recs)
        out = torch.zeros_like(x)
        b = bos.Batch(x, out, offs, seeds, ops, bos.params(rec_bytes, 512, 0), Zs=Zs)
        att = b.run().copy()
        got = bos.to_host(out, recs.dtype)
        for j in range(len(sizes)):
            lo, hi = int(offs[j]), int(offs[j + 1])
            f = oracle.sort if ops[j] else oracle.orp
            ref, rinfo = f(recs[lo:hi], int(Zs[j]), int(seeds[j]), method=oracle.CLOSED)
            assert att[j] == (rinfo.attempts if hi > lo else 0), j
            np.testing.assert_array_equal(got[lo:hi], ref, err_msg=f"array {j} rot {rot}")
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        b.prepare(stream)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream, capture_error_mode="relaxed"):
            b.enqueue(stream)
        out.zero_()
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            graph.replay()
        stream.synchronize()
        done = bos.to_host(out, recs.dtype)  # arrays without an overflow are complete before collect
        for j in range(len(sizes)):
            lo, hi = int(offs[j]), int(offs[j + 1])
            if att[j] == 1:
                np.testing.assert_array_equal(done[lo:hi], got[lo:hi], err_msg=f"replay, array {j} rot {rot}")
        att2 = b.collect(stream)
        np.testing.assert_array_equal(att2, att)
        np.testing.assert_array_equal(bos.to_host(out, recs.dtype), got)


@pytest.mark.parametrize("rec_bytes,Z,n", [(16, 1024, 1 << 22), (16, 512, (1 << 21) + 9), (8, 1024, (1 << 22) - 3),
                                           (16, 2048, 1 << 21), (16, 768, 1 << 21), (8, 32, 1 << 12), (16, 1056, 300001)])
def test_stream_and_tile_passes(bos, rec_bytes, Z, n):
    # plans of the streaming and packed-tile passes over bucket sizes of one, two and four buckets a batch
    recs = inputs.make_records(n, rec_bytes, "uniform", seed=Z)
    for seed in (1, 2):
        try:
            ref, rinfo = oracle.orp(recs, Z, seed, max_attempts=16, method=oracle.CLOSED)
        except oracle.OracleError:
            with pytest.raises(bos.BosError):
                bos.orp(bos.to_device(recs), rec_bytes, Z=Z, seed=seed, max_attempts=16)
            continue
        out, info = bos.orp(bos.to_device(recs), rec_bytes, Z=Z, seed=seed, max_attempts=16)
        assert info.attempts == rinfo.attempts
        np.testing.assert_array_equal(bos.to_host(out, recs.dtype), ref)
