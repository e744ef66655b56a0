"""The order of equal logits in one top-k list: larger values that arrive after them move them down, and they stay
in the order of their classes (ties toward the lower class)."""
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
    return m


@pytest.mark.parametrize("S", [60, 100, 128])
@pytest.mark.parametrize("k", [4, 8, 16])
def test_displaced_equal_logits_keep_their_order(hp, S, k):
    """At most 128 classes are one list, which then holds the whole answer.  Most classes repeat one of a few rows of
    W3 and b3 at random (runs of equal logits that k cuts through), the rest are distinct."""
    N, H1, H2 = 27, 64, 64
    W1, b1, W2, b2, W3, b3 = (inputs.init_weights(sh, f, 50 + i) for i, (sh, f) in enumerate(
        [((H1, N), N), ((H1,), N), ((H2, H1), H1), ((H2,), H1), ((S, H2), H2), ((S,), H2)]))
    rng = np.random.default_rng(S + k)
    row = np.where(rng.random(S) < 0.8, rng.integers(0, S // 5, S), np.arange(S))
    net = hp.MLP(N, H1, H2, S, 512, [W1, b1, W2, b2, W3[row].copy(), b3[row].copy()])
    ids = torch.from_numpy(inputs.sample_ids(N, 500, seed=S).view(np.int64)).cuda()
    z = net.logits(ids).cpu().numpy()
    top = net.topk(ids, k).cpu().numpy()
    net.status()
    np.testing.assert_array_equal(top, np.argsort(-z, axis=1, kind="stable")[:, :k])
