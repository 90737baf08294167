"""The pass kernels where they take their rare branches: batches that are redone in smaller rounds, subproblems
run in parts, middle passes of a batch."""
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


def test_redone_batches_write_every_chunk_once(bos):
    # Middle passes with k = 8 and 2048-slot batches, many subproblems per CTA: about one batch in 3400 runs
    # out of list places and is redone in smaller rounds, and 262144 batches differ from seed to seed in which.
    # The accesses must not: the digest (count and sum of a 64-bit mix of every one) is the same for two seeds
    # (every output position is written once, so the last pass adds the same whatever the loads are).
    import torch
    n, Z = 1 << 28, 512
    info = bos.plan(n, 8, Z, sort=False)
    assert (info.passes, info.stream_passes, info.max_k, info.L, info.max_cluster) == (3, 2, 8, 20, 1)
    x = torch.arange(2 * n, dtype=torch.int32, device="cuda").view(torch.uint8)
    out = torch.empty_like(x)
    ws = bos.alloc_workspace(bos.workspace_bytes(n, bos.params(8, Z, 1)))
    digests = []
    for seed in (1, 2):
        buf = torch.zeros(512, dtype=torch.int64, device="cuda")
        bos.trace_attach_digest(buf)
        try:
            _, info = bos.orp(x, 8, Z=Z, seed=seed, out=out, workspace=ws)
        finally:
            bos.trace_attach_digest(None)
        assert info.attempts == 1
        s = buf.cpu().numpy().view(np.uint64).reshape(-1, 2)
        with np.errstate(over="ignore"):
            digests.append((int(s[:, 0].sum()), int(s[:, 1].sum())))
    assert digests[0] == digests[1]


def _batch(bos, parts, rec_bytes, Zs, seeds):
    """Every array as ORP and as sort in one batch, each against the oracle alone."""
    import torch
    recs = np.concatenate(parts + parts)
    sizes = [len(p) for p in parts] * 2
    offs = np.zeros(len(sizes) + 1, dtype=np.uint64)
    np.cumsum(sizes, out=offs[1:])
    ops = np.repeat(np.array([0, 1], dtype=np.uint8), len(parts))
    x = bos.to_device(recs)
    b = bos.Batch(x, torch.zeros_like(x), offs, np.array(seeds * 2, dtype=np.uint64), ops, bos.params(rec_bytes, 512, 0),
                  Zs=np.array(Zs * 2, dtype=np.uint32))
    att = b.run()
    got = bos.to_host(b.out, recs.dtype)
    for j in range(len(sizes)):
        lo, hi = int(offs[j]), int(offs[j + 1])
        ref, rinfo = (oracle.sort if ops[j] else oracle.orp)(recs[lo:hi], (Zs * 2)[j], (seeds * 2)[j], method=oracle.CLOSED)
        assert att[j] == rinfo.attempts, j
        np.testing.assert_array_equal(got[lo:hi], ref, err_msg=f"array {j}")


@pytest.mark.parametrize("rec_bytes", [8, 16])
def test_batched_middle_passes(bos, rec_bytes):
    # a batch's streaming plan has 8 levels in its first pass and 4 in the last: a middle pass from L = 13 on;
    # batches of one, two and four buckets, beside arrays of two passes
    shapes = [(300000, 128), (5000, 512), ((1 << 20) + 3, 256), ((1 << 21) + 7, 512), (1 << 20, 512)]
    if rec_bytes == 8:
        shapes.append(((1 << 23) + 5, 1536))
    assert [bos.plan(n, rec_bytes, Z).L >= 13 for n, Z in shapes[:5]] == [True, False, True, True, False]
    parts = [inputs.make_records(n, rec_bytes, "uniform", seed=n) for n, _ in shapes]
    _batch(bos, parts, rec_bytes, [Z for _, Z in shapes], list(range(31, 31 + len(shapes))))


@pytest.mark.parametrize("seed", [52, 293])
def test_tile_pass_in_parts(bos, seed):
    # 512 full buckets of Z = 896: five levels in the streaming pass, four in the tile, which has room for 7408
    # 16-byte records; with these seeds a subproblem holds more and runs in parts
    n, Z = 256 * 896, 896
    info = bos.plan(n, 16, Z, k=5, sort=False)
    assert (info.L, info.passes, info.stream_passes, info.max_k, info.max_cluster) == (9, 2, 1, 5, 1)
    assert np.bincount(oracle.labels(n, seed, 0, 9) >> 4).max() > 7408
    recs = inputs.make_records(n, 16, "uniform", seed=seed)
    ref, rinfo = oracle.orp(recs, Z, seed, method=oracle.CLOSED)
    out, info = bos.orp(bos.to_device(recs), 16, Z=Z, seed=seed, k=5)
    assert info.attempts == rinfo.attempts == 1
    np.testing.assert_array_equal(bos.to_host(out, recs.dtype), ref)
    _batch(bos, [recs, recs[:70001]], 16, [Z, Z], [seed, 5])


@pytest.mark.parametrize("rec_bytes", [8, 16])
@pytest.mark.parametrize("count,n,Z,streams", [(1, 1 << 20, 512, False), (48, 1 << 17, 512, True), (64, 1 << 16, 64, False),
                                               (256, 1 << 12, 256, False), (2, (1 << 20) + 5, 1024, True)])
def test_batch_route(bos, rec_bytes, count, n, Z, streams):
    # streaming passes only where the batch has subproblems enough for them and buckets long enough (elsewhere
    # they took up to 4 times as long); the digest of the accesses tells the routes apart, the results agree
    import torch
    recs = inputs.make_records(count * n, rec_bytes, "uniform", seed=count)
    offs = np.arange(count + 1, dtype=np.uint64) * np.uint64(n)
    ops = np.zeros(count, dtype=np.uint8)
    seeds = np.arange(7, 7 + count, dtype=np.uint64)
    x = bos.to_device(recs)
    got, digest = [], []
    for flags in (0, bos.FLAG_NO_STREAM):
        b = bos.Batch(x, torch.zeros_like(x), offs, seeds, ops, bos.params(rec_bytes, Z, 0, flags=flags))
        buf = torch.zeros(512, dtype=torch.int64, device="cuda")
        bos.trace_attach_digest(buf)
        try:
            att = b.run()
        finally:
            bos.trace_attach_digest(None)
        assert att.max() == 1
        digest.append(buf.cpu().numpy().view(np.uint64).reshape(-1, 2)[:, 0].sum())
        got.append(bos.to_host(b.out, recs.dtype))
    assert (digest[0] != digest[1]) == streams
    np.testing.assert_array_equal(got[0], got[1])
    for j in (0, count - 1):
        ref, _ = oracle.orp(recs[j * n:(j + 1) * n], Z, int(seeds[j]), method=oracle.CLOSED)
        np.testing.assert_array_equal(got[0][j * n:(j + 1) * n], ref)
