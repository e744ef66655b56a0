"""The tensor-core scan against the warp scan, the oracle and the map kernel (whole numbers: equal), at the
edges of its blocks of 128 and 256 sequences, its tiles of 256 conformations and its launches."""
import numpy as np
import pytest

from paper_2008_05612_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hp():
    import __graft_entry__

    __graft_entry__.build()
    import paper_2008_05612_gb300 as m

    if not torch.cuda.is_available():
        pytest.fail("CUDA is not available for a gpu-marked test")
    yield m
    m.set_wait_limit(-1)


def ids_of(N, n, seed):
    ids = inputs.sample_ids(N, n, seed=seed)
    ids[: min(n, 2)] = np.array([0, (1 << N) - 1], dtype=np.uint64)[: min(n, 2)]  # every score 0; every score equal
    return ids


def warp_scan(hp, s, t, T):
    """The warp scan: candidates that prune nothing, with counters (gaps clipped at T)."""
    cand = torch.full((t.numel(), 1), -1, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(2, dtype=torch.int64, device="cuda")
    return hp.sequence_scan(s, t, cand=cand, aux=True, gap_threshold=T, gaps=True, counters=cnt)


@pytest.mark.parametrize("dims,n", [((5, 5), 1), ((5, 5), 128), ((5, 5), 129), ((2, 3, 4), 256), ((2, 3, 4), 257),
                                    ((3, 3, 3), 127), ((3, 3, 3), 4099), ((6, 6), 255), ((6, 6), 2049),
                                    ((4, 4), 65521), ((4, 5), 20011)])
def test_tensor_core_scan_equals_the_warp_scan(hp, dims, n):
    s = hp.Structs(dims)
    t = torch.from_numpy(ids_of(s.N, n, 17 + n).view(np.int64)).cuda()
    for T in (1, 5):
        want = warp_scan(hp, s, t, T)
        cnt = torch.zeros(2, dtype=torch.int64, device="cuda")
        got = hp.sequence_scan(s, t, aux=True, gap_threshold=T, gaps=True, counters=cnt)
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
        assert torch.equal(got[2].clamp(max=T), want[2])
        assert cnt.tolist() == [n * s.S_dir, 0]
        # pruned without counters: the same, gaps clipped at T
        cand = torch.zeros((n, 1), dtype=torch.int32, device="cuda")
        for a, b in zip(hp.sequence_scan(s, t, cand=cand, aux=True, gap_threshold=T, gaps=True), want):
            assert torch.equal(a, b)


def test_tensor_core_scan_gaps_equal_the_oracle(hp, obox):
    s = hp.Structs((5, 5))
    ids = ids_of(25, 3000, 5)
    _, aux, gap = obox((5, 5)).phenotypes(ids, aux=True, gaps=True)
    got = hp.sequence_scan(s, torch.from_numpy(ids.view(np.int64)).cuda(), aux=True, gap_threshold=7, gaps=True)
    np.testing.assert_array_equal(got[0].cpu().numpy(), np.where(gap >= 7, aux, -1))
    np.testing.assert_array_equal(got[1].cpu().numpy(), aux)
    np.testing.assert_array_equal(got[2].cpu().numpy(), gap)


def test_more_ids_than_one_launch_takes(hp):
    s = hp.Structs((5, 5))
    n = (1 << 19) + 131
    t = torch.from_numpy(ids_of(25, n, 3).view(np.int64)).cuda()
    assert torch.equal(hp.sequence_scan(s, t), hp.phenotype_map(s)[t])


def test_exact_when_waits_give_up_and_under_capture(hp):
    """A wait that gives up leaves the sequences to the resolving kernel; a captured scan replays."""
    s = hp.Structs((5, 5))
    t = torch.from_numpy(ids_of(25, 5000, 9).view(np.int64)).cuda()
    want = hp.sequence_scan(s, t, aux=True)
    hp.set_wait_limit(0)
    try:
        got = hp.sequence_scan(s, t, aux=True)
    finally:
        hp.set_wait_limit(-1)
    assert all(torch.equal(a, b) for a, b in zip(got, want))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = hp.sequence_scan(s, t, aux=True)
    for x in out:
        x.zero_()
    graph.replay()
    graph.replay()
    assert all(torch.equal(a, b) for a, b in zip(out, want))


@pytest.mark.parametrize("dims,begin,count,T", [((3, 3, 3), 12345, 150001, 1), ((3, 3, 3), (1 << 26) - 3, 7, 1),
                                                ((3, 3, 3), (1 << 22) + 1, (1 << 22) + 77, 1), ((3, 3, 3), 0, 1 << 14, 9),
                                                ((2, 3, 4), 777, 65535, 12), ((5, 5), 3, (1 << 20) + 9, 4),
                                                ((6, 6), (1 << 35) + 5, 4097, 2), ((4, 5), 0, 1 << 20, 1)])
def test_split_ranges_equal_the_map_kernel(hp, dims, begin, count, T):
    """A range split between the scan and the map kernel against the map kernel alone (a library with a shape set)."""
    s, k = hp.Structs(dims), hp.Structs(dims)
    k.set_tile_cfg(5, 256)
    out = [torch.full((count + 2,), -9, dtype=torch.int32, device="cuda") for _ in range(4)]
    hp.phenotype_map(s, begin, count, out=out[0][1:-1], aux=out[1][1:-1], gap_threshold=T)
    hp.phenotype_map(k, begin, count, out=out[2][1:-1], aux=out[3][1:-1], gap_threshold=T)
    assert torch.equal(out[0], out[2]) and torch.equal(out[1], out[3])
