"""Host memory that the GPU reads or writes while a call runs: it outlives the work that uses it, and calls
that find no slot of the shared pinned block are as good as those that do. What depends on the state of a
whole process runs in a child (this file with the function's name)."""
import ctypes
import os
import subprocess
import sys
import threading
import time

import numpy as np
import pytest

import oracle
from paper_2008_01765_gb300 import inputs

pytestmark = pytest.mark.gpu


SLOTS = 12


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


def _child(name, **env):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-m", "tests.test_gpu_host_state", name], cwd=root, env={**os.environ, **env},
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


def _keys(n, rec_bytes, shape):
    recs = inputs.make_records(n, rec_bytes, "uniform", seed=n)
    if shape == "two":  # crowds one value of the top digit from kCap on: LSD passes
        recs["key"] = recs["key"] & recs["key"].dtype.type(1 << 7)
    return recs


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


# every mode of the sort: on chip (classes 0 to 5), one partition, two partitions, LSD passes, one key
NO_SLOT_CASES = [(1, 16, "uniform"), (200, 8, "uniform"), (1000, 16, "uniform"), (2000, 8, "two"), (4096, 16, "uniform"),
                 (9000, 16, "two"), (19000, 16, "uniform"), (19000, 16, "two"), (28000, 8, "uniform"),
                 (70001, 16, "uniform"), (1 << 20, 8, "uniform"), (1 << 20, 16, "two"), ((1 << 23) + 1, 16, "uniform")]


def child_no_slot():
    import torch
    from paper_2008_01765_gb300 import bos
    jobs = []
    for n, rec, shape in NO_SLOT_CASES:
        recs = _keys(n, rec, shape)
        x = bos.to_device(recs)
        p = bos.params(rec, 512, 5)
        jobs.append((recs, rec, x, torch.empty_like(x), bos.alloc_workspace(bos.workspace_bytes(n, p))))
    for rec in (8, 16):  # every kernel of the sort once: loading one late may wait for the sleeping calls
        for n, shape in [(200, "uniform"), (1000, "uniform"), (2000, "uniform"), (4096, "uniform"), (9000, "uniform"),
                         (14000, "two"), (19000, "two"), (28000, "two"), (70001, "uniform"), (1 << 20, "two"),
                         (1 << 24, "uniform")]:
            bos.sort(bos.to_device(_keys(n, rec, shape)), rec, Z=512, seed=5)
    small = bos.to_device(_keys(64, 16, "uniform"))
    held = [(torch.cuda.Stream(), torch.empty_like(small), bos.alloc_workspace(1 << 20)) for _ in range(SLOTS)]
    main = torch.cuda.Stream()
    torch.cuda.synchronize()
    free = bos.lib().bos_selftest_host_slots

    def hold(stream, out, ws):  # a call that waits for its stream holds its slot meanwhile
        with torch.cuda.stream(stream):
            torch.cuda._sleep(1_000_000_000)  # about half a second
        bos.orp(small, 16, Z=512, seed=1, out=out, workspace=ws, stream=stream)

    assert free() == SLOTS
    threads = [threading.Thread(target=hold, args=h) for h in held]
    for t in threads:
        t.start()
    end = time.time() + 0.3
    while free() and time.time() < end:
        time.sleep(0.001)
    assert free() == 0
    infos = []
    for recs, rec, x, out, ws in jobs:
        infos.append(bos.sort(x, rec, Z=512, seed=5, out=out, workspace=ws, stream=main)[1])
        assert free() == 0, f"{len(recs)} x {rec}: the slots were not held long enough"
    for t in threads:
        t.join()
    assert free() == SLOTS
    modes = set()
    for (recs, rec, x, out, ws), info in zip(jobs, infos):
        ref, rinfo = oracle.sort(recs, 512, 5, method=oracle.CLOSED)
        assert info.attempts == rinfo.attempts
        modes.add(info.sort_mode)
        np.testing.assert_array_equal(bos.to_host(out, recs.dtype), ref, err_msg=f"{len(recs)} x {rec}")
    assert modes == {0, 1, 2, 3}


def test_sort_without_a_host_slot(bos):
    # twelve calls hold the twelve slots; a queue per stream, so that the others run meanwhile
    _child("child_no_slot", CUDA_DEVICE_MAX_CONNECTIONS="32")


def child_noalloc_first():
    from paper_2008_01765_gb300 import bos
    recs = _keys(5000, 16, "uniform")
    x = bos.to_device(recs)
    ref, _ = oracle.orp(recs, 512, 3, method=oracle.CLOSED)
    free = bos.lib().bos_selftest_host_slots
    for block in (0, SLOTS):  # before the block exists, and after bos_orp has made it
        for _ in range(2):
            out, _ = bos.orp_noalloc(x, 16, Z=512, seed=3)
            np.testing.assert_array_equal(bos.to_host(out, recs.dtype), ref)
            assert free() == block
        bos.orp(x, 16, Z=512, seed=3)
        assert free() == SLOTS


def test_noalloc_allocates_no_host_block(bos):
    # the process's first call is bos_orp_noalloc: the pinned block must not come into being
    _child("child_noalloc_first")


def child_failed_calls():
    import torch
    from paper_2008_01765_gb300 import bos
    recs = _keys(5000, 16, "uniform")
    x = bos.to_device(recs)
    out, ws = torch.empty_like(x), bos.alloc_workspace(1 << 24)
    ref, _ = oracle.sort(recs, 512, 3, method=oracle.CLOSED)
    bos.sort(x, 16, Z=512, seed=3, out=out, workspace=ws)
    bos.orp(x, 16, Z=512, seed=3, out=out, workspace=ws)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    rt = ctypes.CDLL("libcudart.so.13")
    handle, graph = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
    for j in range(2 * SLOTS):  # a call that synchronises cannot be captured: it fails halfway
        assert rt.cudaStreamBeginCapture(handle, 2) == 0  # 2: relaxed
        with pytest.raises(bos.BosError):
            (bos.sort if j % 2 else bos.orp)(x, 16, Z=512, seed=3, out=out, workspace=ws, stream=stream)
        assert rt.cudaStreamEndCapture(handle, ctypes.byref(graph)) != 0  # invalidated
        rt.cudaGetLastError()
        assert bos.lib().bos_selftest_host_slots() == SLOTS, j
    bos.sort(x, 16, Z=512, seed=3, out=out, workspace=ws, stream=stream)
    np.testing.assert_array_equal(bos.to_host(out, recs.dtype), ref)


def test_failed_calls_give_their_slots_back(bos):
    _child("child_failed_calls")


def child_reset():
    # no torch here: its allocator would not survive the reset
    from paper_2008_01765_gb300 import bos
    rt = ctypes.CDLL("libcudart.so.13")
    rt.cudaMalloc.argtypes = [ctypes.POINTER(ctypes.c_void_p), ctypes.c_size_t]
    rt.cudaHostAlloc.argtypes = [ctypes.POINTER(ctypes.c_void_p), ctypes.c_size_t, ctypes.c_uint]
    rt.cudaMemcpy.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int]
    L, n = bos.lib(), 5000
    recs = _keys(n, 16, "uniform")
    p = bos.params(16, 512, 3)
    need = bos.workspace_bytes(n, p)
    ref = {"bos_sort": oracle.sort(recs, 512, 3, method=oracle.CLOSED)[0]}
    ref["bos_orp"] = ref["bos_orp_noalloc"] = oracle.orp(recs, 512, 3, method=oracle.CLOSED)[0]

    def alloc(nbytes):
        q = ctypes.c_void_p()
        assert rt.cudaMalloc(ctypes.byref(q), nbytes) == 0
        return q

    def call(name):
        x, out, ws = alloc(n * 16), alloc(n * 16), alloc(need)
        assert rt.cudaMemcpy(x, recs.ctypes.data, n * 16, 1) == 0
        args = (x, out, n, ctypes.byref(p)) + ((None, None) if name == "bos_orp_noalloc" else (ws, need, None, None))
        assert getattr(L, name)(*args) == bos.OK, name
        got = np.zeros_like(recs)
        assert rt.cudaMemcpy(got.ctypes.data, out, n * 16, 2) == 0
        np.testing.assert_array_equal(got, ref[name], err_msg=name)

    for order in (("bos_sort", "bos_orp"), ("bos_orp", "bos_sort"), ("bos_orp_noalloc", "bos_sort")):
        call("bos_sort")
        assert L.bos_selftest_host_slots() == SLOTS
        assert rt.cudaDeviceReset() == 0
        mine = []  # pinned memory of the caller's, some of it where the library's block was
        for _ in range(8):
            q = ctypes.c_void_p()
            assert rt.cudaHostAlloc(ctypes.byref(q), 4096, 3) == 0  # portable, mapped
            ctypes.memset(q, 0x5A, 4096)
            mine.append(q)
        for name in order:
            call(name)
        assert L.bos_selftest_host_slots() == SLOTS
        assert all(ctypes.string_at(q, 4096) == b"\x5a" * 4096 for q in mine)


def test_host_block_after_a_device_reset(bos):
    # the reset ends the process's own context, and the pinned block with it
    _child("child_reset")


if __name__ == "__main__":
    globals()[sys.argv[1]]()
