"""The product over the split working copy (k_prod.cu) at the edges of its tiles: rows and K
around 64 and 128, every padded rank, tiles shared by many blocks and by one, and a matrix
above the size from which part of it is kept in L2.

Tolerance: both operands are split to 2^-24 relative and the dropped product of the low
terms is 2^-24; the tensor core adds at most 128 terms between drains, each addition off by
at most 2^-23 of the running sum.  For Gaussian data (running sums of about sqrt(K) against a
result of sqrt(K)) that is below 128 * 2^-23 / sqrt(128) = 1.4e-6 relative in the norm."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1309_0302_gb300 as G
    G.library()


@pytest.mark.parametrize("m,n,r", [(1, 1, 1), (64, 128, 8), (63, 129, 9), (65, 127, 17), (128, 1, 1), (1, 257, 1),
                                   (129, 191, 33), (257, 320, 48), (300, 130, 49), (191, 385, 57), (513, 640, 64),
                                   (20000, 65, 24), (130, 20001, 40), (5003, 5203, 50)])
def test_transposed_product(m, n, r):
    import torch

    import paper_1309_0302_gb300 as G
    g = torch.Generator(device="cuda").manual_seed(m * 31 + n)
    Z = torch.randn(m, n, generator=g, device="cuda")
    C = torch.randn(m, r, generator=g, device="cuda")
    W = G.mul_ZtC(Z, C).double()
    ref = Z.double().T @ C.double()
    assert (W - ref).norm().item() <= 1.4e-6 * ref.norm().item()


@pytest.mark.parametrize("m,n,r,q", [(129, 65, 3, 1), (255, 383, 57, 0), (5003, 5203, 9, 1)])
def test_chain_against_64_bits(m, n, r, q):
    """One L-step (products in both directions with normalisers and Gram partials) on a
    noiseless rank-r matrix: it is recovered, to the float32 products' error."""
    import torch

    import paper_1309_0302_gb300 as G
    g = torch.Generator(device="cuda").manual_seed(n)
    X = torch.randn(m, r, generator=g, device="cuda") @ torch.randn(n, r, generator=g, device="cuda").T
    ctx = G.GoDec(X, torch.randn(n, r, generator=g, device="cuda"), r, 0, q, tol=0.0, max_iter=4)
    ctx.iterate(3)   # exact path, then the lagged normalisers
    L = ctx.L_dense().double()
    ctx.close()
    assert (L - X.double()).norm().item() <= 1e-5 * X.double().norm().item()
