"""Host memory that the GPU reads or writes while a call runs: it outlives the work that uses it."""
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


def test_batch_descriptors_outlive_their_copy(bos):
    # The stream is busy when the batch is issued, so the copy of its descriptors runs long after it was
    # enqueued; the host bytes it reads must still be there.
    import torch
    sizes = [5000, 3, 2112, 40000, 0, 1 << 17] * 8
    recs = inputs.make_records(sum(sizes), 16, "uniform", seed=21)
    offs = np.zeros(len(sizes) + 1, dtype=np.uint64)
    np.cumsum(sizes, out=offs[1:])
    ops = (np.arange(len(sizes)) % 2).astype(np.uint8)
    seeds = np.arange(1, len(sizes) + 1, dtype=np.uint64)
    x = bos.to_device(recs)
    out = torch.zeros_like(x)
    b = bos.Batch(x, out, offs, seeds, ops, bos.params(16, 512, 0))
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    for _ in range(3):
        with torch.cuda.stream(stream):
            out.zero_()
            torch.cuda._sleep(40_000_000)  # about 20 ms
        b.run(stream)
        got = bos.to_host(out, recs.dtype)
        for j in range(len(sizes)):
            lo, hi = int(offs[j]), int(offs[j + 1])
            ref, _ = (oracle.sort if ops[j] else oracle.orp)(recs[lo:hi], 512, int(seeds[j]), method=oracle.CLOSED)
            np.testing.assert_array_equal(got[lo:hi], ref, err_msg=f"array {j}")
