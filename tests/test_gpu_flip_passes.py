"""The passes over a map's flips: neutral networks at the edges of their blocks (2^13 ids) and pass groups, and
the rows of the phi matrix on both sides of the longest row that one warp sorts, against the oracle."""
import numpy as np
import pytest

import oracle
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
    return m


def plateaus(N, S, seed, bits):
    """Phenotypes of the top `bits` bits (networks that cross blocks and pass groups), a quarter of the ids at -1."""
    g = np.arange(1 << N, dtype=np.uint64)
    p = (inputs.splitmix64((g >> np.uint64(max(N - bits, 0))) ^ np.uint64(seed)) % np.uint64(S)).astype(np.int32)
    p[inputs.splitmix64(g ^ np.uint64(seed + 5)) % np.uint64(4) == 0] = -1
    return p


@pytest.mark.parametrize("N", [1, 2, 3, 9, 10, 12, 14, 17, 18, 21, 22])
@pytest.mark.parametrize("offset", [0, 1])
def test_components_equal_the_oracle(hp, N, offset):
    S = 5
    phen_np = plateaus(N, S, 7 + N, 6)
    want_label, want_n = oracle.components(phen_np, N, S)
    buf = torch.empty((1 << N) + 1, dtype=torch.int32, device="cuda")  # an offset of one id: not 16-byte aligned
    phen = buf[offset: offset + (1 << N)]
    phen.copy_(torch.from_numpy(phen_np))
    out = torch.empty((1 << N) + 1, dtype=torch.int32, device="cuda")[offset: offset + (1 << N)]
    label, ncomp = hp.neutral_components(phen, N, S, out_label=out)
    np.testing.assert_array_equal(label.cpu().numpy(), want_label)
    np.testing.assert_array_equal(ncomp.cpu().numpy().astype(np.int64), np.asarray(want_n).astype(np.int64)[:S])


@pytest.mark.parametrize("N,S,hubs", [(14, 3000, 2), (13, 260, 1), (13, 255, 1), (12, 1023, 0), (12, 1024, 0), (15, 9000, 1)])
def test_phi_rows_of_every_length_equal_the_oracle(hp, N, S, hubs):
    """Random phenotypes, and `hubs` of them on half of the ids (rows of more than 256 entries)."""
    g = np.arange(1 << N, dtype=np.uint64)
    p = (inputs.splitmix64(g ^ np.uint64(N)) % np.uint64(S)).astype(np.int32)
    r = inputs.splitmix64(g ^ np.uint64(99)) % np.uint64(8)
    if hubs:
        p[r < 4] = (S - 1 - (g[r < 4] % np.uint64(hubs))).astype(np.int32)
    p[r == 7] = -1
    row_ptr, col, count = (t.cpu().numpy() for t in hp.phi_matrix(torch.from_numpy(p).cuda(), N, S))
    assert row_ptr[0] == 0 and row_ptr[S + 1] == len(col)
    for q in list(range(0, S, max(1, S // 300))) + [S - 1, -1]:
        want = np.asarray(oracle.neighbourhood(p, N, S, q)).astype(np.int64)
        a, b = row_ptr[q if q >= 0 else S], row_ptr[(q if q >= 0 else S) + 1]
        nz = np.flatnonzero(want)
        np.testing.assert_array_equal(col[a:b], nz)
        np.testing.assert_array_equal(count[a:b], want[nz])
