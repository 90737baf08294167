"""The pass kernels where they take their rare branches: batches that are redone in smaller rounds, subproblems
run in parts, middle passes of a batch."""
import numpy as np
import pytest

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
