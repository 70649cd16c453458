"""The select rounds where their number and their blocks change: linear indices on either side of
12 and 24 bits (one index digit more), counts of candidates on either side of what one block and
the whole grid take, all of them ties of one value.  Whole numbers: exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(64, 64), (17, 241), (4096, 4096), (4097, 4096)])
@pytest.mark.parametrize("extra", [0, 1, 1023, 1025])
def test_ties_cut_by_index(m, n, extra):
    """`extra` of the equal entries are wanted beside the larger ones: the first by linear index."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1309_0302_gb300 as G
    g = np.random.default_rng(m * n + extra)
    R = np.full(m * n, -1.0, np.float32)
    big = np.sort(g.choice(m * n, 60, replace=False))
    R[big] = 2.0
    rest = np.setdiff1d(np.arange(extra + 60), big)[:extra]
    want = np.sort(np.concatenate([big, rest]))
    idx, val = G.hard_threshold(torch.from_numpy(R.reshape(m, n)).cuda(), 60 + extra)
    assert np.array_equal(idx.cpu().numpy(), want)
    assert np.array_equal(val.cpu().numpy(), R[want])
