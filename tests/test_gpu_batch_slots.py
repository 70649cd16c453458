"""Batches whose problems need more partial slots at a share of the SMs than on the whole
device: 128 row tiles over as many blocks take one slot each, over fewer blocks two (16384
rows); a large share of an uneven batch (8192 rows beside a small problem)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1309_0302_gb300 as G
    G.library()


@pytest.mark.parametrize("shapes", [[(16384, 300), (16384, 300)], [(300, 16384), (513, 400)],
                                    [(8192, 512), (300, 256)]])
@pytest.mark.parametrize("tune", [True, False])
def test_batch_of_whole_tiles(shapes, tune):
    """L of every problem as its own context gives it (grids change only the order of float32
    sums: 1e-5, as for the other batches)."""
    import torch

    import paper_1309_0302_gb300 as G
    g = torch.Generator(device="cuda").manual_seed(5)
    Xs, A1s, ks = [], [], []
    for m, n in shapes:
        X = torch.randn(m, 4, generator=g, device="cuda") @ torch.randn(n, 4, generator=g, device="cuda").T
        X += 1e-2 * torch.randn(m, n, generator=g, device="cuda")
        k = m * n // 100
        pos = torch.randperm(m * n, generator=g, device="cuda")[:k]
        X.view(-1)[pos] += 5.0 * torch.randn(k, generator=g, device="cuda")
        Xs.append(X)
        A1s.append(torch.randn(n, 4, generator=g, device="cuda"))
        ks.append(k)
    b = G.GoDecBatch(Xs, A1s, 4, ks, 1, tune=tune)
    try:
        b.iterate(4)
        for j, (X, A1, k) in enumerate(zip(Xs, A1s, ks)):
            one = G.GoDec(X, A1, 4, k, 1, tol=-1.0, max_iter=10)
            one.iterate(4)
            L, L1 = b.problem(j).L_dense().double(), one.L_dense().double()
            one.close()
            assert (L - L1).norm().item() <= 1e-5 * L1.norm().item(), j
    finally:
        b.close()
