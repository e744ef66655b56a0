"""Scans of a list of ids in CUDA graphs and around them: which kernels a capture records, what may be done with its
graph, and that a table or scratch that could not be had once is had by the next call."""
import ctypes

import numpy as np
import pytest

from paper_2008_05612_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KERNEL_NODE, GLOBAL_MODE = 0, 0


@pytest.fixture(scope="module")
def hp():
    import __graft_entry__

    __graft_entry__.build()
    import paper_2008_05612_gb300 as m

    if not torch.cuda.is_available():
        pytest.fail("CUDA is not available for a gpu-marked test")
    return m


class Capture:
    """call() captured on a stream of its own, through the CUDA runtime that torch has loaded; its outputs are of
    n ids."""

    def __init__(self, n, call):
        self.rt = ctypes.CDLL("libcudart.so.%s" % torch.version.cuda.split(".")[0])
        self.stream = torch.cuda.Stream()
        self.graph = ctypes.c_void_p()
        self.error = None
        with torch.cuda.stream(self.stream):  # blocks for the outputs, which torch keeps for this stream
            blocks = [torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(4)]
            del blocks
        torch.cuda.synchronize()
        ptr = ctypes.c_void_p(self.stream.cuda_stream)
        with torch.cuda.stream(self.stream):
            assert self.rt.cudaStreamBeginCapture(ptr, GLOBAL_MODE) == 0
            try:
                self.out = call()
            except Exception as e:
                self.error = e
            rc = self.rt.cudaStreamEndCapture(ptr, ctypes.byref(self.graph))
            self.rt.cudaGetLastError()
            if rc != 0 and self.error is None:
                self.error = RuntimeError(f"cudaStreamEndCapture: {rc}")

    def nodes(self):
        n = ctypes.c_size_t()
        assert self.rt.cudaGraphGetNodes(self.graph, None, ctypes.byref(n)) == 0
        arr = (ctypes.c_void_p * n.value)()
        assert self.rt.cudaGraphGetNodes(self.graph, arr, ctypes.byref(n)) == 0
        types = []
        for node in arr:
            t = ctypes.c_int()
            assert self.rt.cudaGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(t)) == 0
            types.append(t.value)
        return types

    def instance(self, graph=None):
        x = ctypes.c_void_p()
        rc = self.rt.cudaGraphInstantiate(ctypes.byref(x), graph or self.graph, ctypes.c_ulonglong(0))
        return rc, x

    def launch(self, x, stream=None):
        assert self.rt.cudaGraphLaunch(x, ctypes.c_void_p((stream or self.stream).cuda_stream)) == 0

    def destroy(self):
        assert self.rt.cudaGraphDestroy(self.graph) == 0


def ids_of(N, n, seed):
    return torch.from_numpy(inputs.sample_ids(N, n, seed=seed).view(np.int64)).cuda()


def warp_scan(hp, s, ids, **kw):
    """A scan that counts its pruning runs one warp per sequence (candidates of -1 prune nothing)."""
    cand = torch.full((ids.numel(), 1), -1, dtype=torch.int32, device="cuda")
    return hp.sequence_scan(s, ids, cand=cand, counters=torch.zeros(2, dtype=torch.int64, device="cuda"), **kw)


def test_a_table_that_found_no_memory_is_built_by_a_later_call(hp):
    other = hp.Structs((2, 2, 6))
    hp.sequence_scan(other, ids_of(24, 64, 1))  # every kernel is loaded
    s = hp.Structs((3, 3, 3))
    ids = ids_of(27, 64, 3)
    want = warp_scan(hp, s, ids)
    hog, size = [], torch.cuda.mem_get_info()[0]
    while size >= 1 << 21:  # all but a few MB of the device
        try:
            hog.append(torch.empty(size, dtype=torch.uint8, device="cuda"))
        except torch.OutOfMemoryError:
            size //= 2
    try:
        assert torch.cuda.mem_get_info()[0] < 1 << 23
        assert torch.equal(hp.sequence_scan(s, ids), want)
    finally:
        del hog
        torch.cuda.empty_cache()
    assert torch.equal(hp.sequence_scan(s, ids), want)
    later = Capture(64, lambda: hp.sequence_scan(s, ids))
    assert later.error is None
    assert later.nodes().count(KERNEL_NODE) == 2  # the scan and what resolves its ties, not the warp scan
    later.destroy()
