"""Scans of a list of ids in CUDA graphs and around them: which kernels a capture records, what may be done with its
graph, and that a table or scratch that could not be had once is had by the next call."""
import ctypes
import time

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


def runtime():
    """The CUDA runtime that torch has loaded."""
    return ctypes.CDLL("libcudart.so.%s" % torch.version.cuda.split(".")[0])


class Capture:
    """call() captured on a stream of its own; its outputs are of n ids."""

    def __init__(self, n, call):
        self.rt = runtime()
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
    rt = runtime()
    hog, size = [], torch.cuda.mem_get_info()[0]
    while size >= 1 << 21:  # all but a few MB of the device (torch's allocator takes 20 MB at a time)
        p = ctypes.c_void_p()
        if rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(size)) == 0:
            hog.append(p)
        else:
            rt.cudaGetLastError()
            size //= 2
    try:
        assert torch.cuda.mem_get_info()[0] < 1 << 23
        assert torch.equal(hp.sequence_scan(s, ids), want)
    finally:
        for p in hog:
            assert rt.cudaFree(p) == 0
    assert torch.equal(hp.sequence_scan(s, ids), want)
    later = Capture(64, lambda: hp.sequence_scan(s, ids))
    assert later.error is None
    assert later.nodes().count(KERNEL_NODE) == 2  # the scan and what resolves its ties, not the warp scan
    later.destroy()


@pytest.mark.parametrize("dims", [(5, 5), (3, 3, 3)])
@pytest.mark.parametrize("counted", [False, True])
def test_a_scan_makes_every_later_scan_capturable(hp, dims, counted):
    """The tensor-core scan and the warp scan have tables of their own; a capture of one after only the other has run."""
    s, ref = hp.Structs(dims), hp.Structs(dims)
    ids = ids_of(s.N, 5000, 11)
    cand = torch.zeros((5000, 1), dtype=torch.int32, device="cuda")
    cnt = torch.zeros(2, dtype=torch.int64, device="cuda")
    plain = lambda h: hp.sequence_scan(h, ids, aux=True)
    pruned = lambda h: hp.sequence_scan(h, ids, cand=cand, aux=True, counters=cnt)
    first, then = (pruned, plain) if not counted else (plain, pruned)
    want = plain(ref)
    first(s)
    c = Capture(5000, lambda: then(s))
    assert c.error is None, c.error
    for t in c.out:
        t.zero_()
    torch.cuda.synchronize()
    rc, x = c.instance()
    assert rc == 0
    c.launch(x)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(c.out, want))
    assert c.rt.cudaGraphExecDestroy(x) == 0
    c.destroy()


@pytest.mark.parametrize("n", [700, (1 << 19) + 131])  # one launch and two
def test_a_captured_scan_is_kernels_alone(hp, n):
    """So its graph may have two instances, side by side on two streams, and be a node of another graph."""
    s = hp.Structs((5, 5))
    ids = ids_of(25, n, 13)
    want = hp.sequence_scan(s, ids)
    c = Capture(n, lambda: hp.sequence_scan(s, ids))
    assert c.error is None, c.error
    assert set(c.nodes()) == {KERNEL_NODE}
    other, parent, node = torch.cuda.Stream(), ctypes.c_void_p(), ctypes.c_void_p()
    assert c.rt.cudaGraphCreate(ctypes.byref(parent), 0) == 0
    assert c.rt.cudaGraphAddChildGraphNode(ctypes.byref(node), parent, None, ctypes.c_size_t(0), c.graph) == 0
    (rc0, x0), (rc1, x1), (rc2, x2) = c.instance(), c.instance(), c.instance(parent)
    assert (rc0, rc1, rc2) == (0, 0, 0)
    c.destroy()  # the instances keep the scratch
    again = Capture(n, lambda: hp.sequence_scan(s, ids ^ 1))
    assert again.error is None
    for use in ([x0, x1], [x2]):
        c.out.zero_()
        torch.cuda.synchronize()
        for _ in range(5):
            for x, st in zip(use, (c.stream, other)):
                c.launch(x, st)
        torch.cuda.synchronize()
        assert torch.equal(c.out, want)
    for x in (x0, x1, x2):
        assert c.rt.cudaGraphExecDestroy(x) == 0
    assert c.rt.cudaGraphDestroy(parent) == 0
    again.destroy()


def test_captures_share_scratch_over_time_and_the_library_gives_it_back(hp):
    s = hp.Structs((5, 5))
    n = 1 << 19
    ids = ids_of(25, n, 17)
    hp.sequence_scan(s, ids)
    torch.cuda.synchronize()

    def one():
        c = Capture(n, lambda: hp.sequence_scan(s, ids))
        assert c.error is None
        rc, x = c.instance()
        assert rc == 0
        c.launch(x)
        torch.cuda.synchronize()
        assert c.rt.cudaGraphExecDestroy(x) == 0
        c.destroy()
        del c
        torch.cuda.empty_cache()
        time.sleep(0.02)  # the driver may end the scratch's use a little later
        return torch.cuda.mem_get_info()[0]

    first = one()
    free = [one() for _ in range(12)]
    assert first - min(free) < 3 * (28 << 20)  # not 12 blocks of 27 MB
    del s
    assert torch.cuda.mem_get_info()[0] >= min(free) + (27 << 20) - (2 << 20)


def test_the_library_keeps_one_launch_of_scratch_and_gives_it_back(hp):
    s = hp.Structs((5, 5))
    n = 1 << 19
    ids = ids_of(25, n, 19)
    want = hp.sequence_scan(s, ids)
    streams = [torch.cuda.Stream() for _ in range(4)]
    for _ in range(3):  # scans on several streams take scratch side by side
        outs = [hp.sequence_scan(s, ids, stream=st) for st in streams]
        torch.cuda.synchronize()
        assert all(torch.equal(o, want) for o in outs)
        held = torch.cuda.mem_get_info()[0]
    for _ in range(3):
        hp.sequence_scan(s, ids)
        torch.cuda.synchronize()
        assert torch.cuda.mem_get_info()[0] >= held
    held = torch.cuda.mem_get_info()[0]
    del s
    back = torch.cuda.mem_get_info()[0] - held
    assert (26 << 20) <= back <= (72 << 20)  # 27 MB kept of four times 27, and the tables
