"""The map kernel itself against the warp scan.  A library without a shape set divides its ranges, and ranges of many
conformations and few ids, or at a threshold above 1, then run on the tensor-core scan, as long lists of ids do: here a
shape is set on the library, which keeps the whole range on the map kernel, and the other side counts its pruning,
which keeps it on the warp scan.  Phenotypes and lowest minimisers are whole numbers: equal."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hp():
    import __graft_entry__

    __graft_entry__.build()
    import paper_2008_05612_gb300 as m

    if not torch.cuda.is_available():
        pytest.fail("CUDA is not available for a gpu-marked test")
    return m


@pytest.mark.parametrize("dims,begin,count,sample", [((3, 3, 3), 5 << 22, 1 << 20, 16), ((3, 3, 3), (3 << 20) + 77, 1500, 1),
                                                     ((6, 6), 7 << 30, 1 << 22, 64), ((2, 3, 4), 0, 1 << 24, 256),
                                                     ((5, 5), 12345, 1 << 16, 1)])
def test_map_kernel_equals_the_warp_scan(hp, dims, begin, count, sample):
    """404 tiles of conformations (3x3x3), 224 (6x6), a whole space (2x3x4) and ragged ranges, at every kind of threshold."""
    s = hp.Structs(dims)
    s.set_tile_cfg(5, 256)
    ids = torch.arange(begin, begin + count, sample, dtype=torch.int64, device="cuda")
    none = torch.full((ids.numel(), 1), -1, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(2, dtype=torch.int64, device="cuda")
    for T in (1, 2, 5, 13):
        aux = torch.empty(count, dtype=torch.int32, device="cuda")
        got = hp.phenotype_map(s, begin, count, aux=aux, gap_threshold=T)
        want, want_aux = hp.sequence_scan(s, ids, cand=none, aux=True, counters=cnt, gap_threshold=T)
        assert torch.equal(got[::sample], want) and torch.equal(aux[::sample], want_aux)
