"""The residual of a matrix whose rows had to be copied to aligned ones has the matrix's own shape:
every entry X - L (float32 roundings of the terms and the tensor cores' two-term split: 2^-20 of the
sum of their magnitudes), no column of the copy's padding."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,r", [(200, 257, 3), (130, 66, 9), (64, 128, 4), (33, 1, 1)])
def test_residual_has_the_shape_of_x(m, n, r):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1309_0302_gb300 as G
    g = torch.Generator(device="cuda").manual_seed(n)
    X = torch.randn(m, n, generator=g, device="cuda")
    ctx = G.GoDec(X, torch.randn(n, r, generator=g, device="cuda"), r, m * n // 50, 1, tol=-1.0, max_iter=9)
    ctx.iterate(2)
    U, s, V = (t.double() for t in ctx.L())
    R = ctx.residual()
    ctx.close()
    assert R.shape == (m, n)
    size = X.double().abs() + (U.abs() * s) @ V.abs().T
    assert bool(((R.double() - (X.double() - (U * s) @ V.T)).abs() <= 2.0 ** -20 * size).all())
