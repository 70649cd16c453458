"""The hard threshold's streaming passes and the ordered export from the support bitmap, at the
sizes where they can go wrong: columns that are no multiple of the eight a thread takes, more
candidates in a step than the staging buffer holds, supports of every density, several blocks
of bitmap words, and one that ends inside a word.  Integer comparisons: exact."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1309_0302_gb300 as G
    G.library()


@pytest.mark.parametrize("m,n", [(1, 1), (1, 33), (7, 8), (9, 15), (300, 1021), (1000, 4097), (2500, 1024)])
@pytest.mark.parametrize("frac", [0.0, 0.003, 0.5, 1.0])
def test_threshold_exact(m, n, frac):
    import torch

    import paper_1309_0302_gb300 as G
    g = np.random.default_rng(m + 7 * n)
    R = g.standard_normal((m, n)).astype(np.float32)
    R[g.random((m, n)) < 0.1] = 0.0
    R.ravel()[:: max(1, m * n // 50)] = 1.5          # ties
    k = int(round(frac * m * n))
    idx, val = G.hard_threshold(torch.from_numpy(R).cuda(), k)
    ri, rv = O.hard_threshold(R.astype(np.float64), k)
    assert np.array_equal(idx.cpu().numpy(), ri)
    assert np.array_equal(val.cpu().numpy(), rv.astype(np.float32))


@pytest.mark.parametrize("m,n,k", [(40, 33, 1), (513, 400, 30000), (2000, 1300, 1500)])
def test_context_export_in_order(m, n, k):
    """S of a context: ascending indices, values R there (bit for bit, from the dump of R)."""
    import torch

    import paper_1309_0302_gb300 as G
    g = torch.Generator(device="cuda").manual_seed(k)
    X = torch.randn(m, 3, generator=g, device="cuda") @ torch.randn(n, 3, generator=g, device="cuda").T
    X += torch.randn(m, n, generator=g, device="cuda")
    ctx = G.GoDec(X, torch.randn(n, 3, generator=g, device="cuda"), 3, k, 1, tol=0.0, max_iter=9)
    ctx.iterate(2)
    idx, val = ctx.S()
    R = ctx.residual()
    ctx.close()
    assert idx.numel() == k and bool((idx[1:] > idx[:-1]).all())
    assert torch.equal(val, R[:, :n].reshape(-1)[idx])
