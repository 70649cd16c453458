"""Dense L at the ranks where its kernel changes (4 and 8 are the register widths, above 8
the tensor cores) and at row and column counts that no tile divides.  Bound per element: r + 2
float32 roundings of the terms up to rank 8, |err| <= (r + 2) 2^-24 sum |u s v|; above, the
factors' 2^-23 splits and an accumulation that is not to nearest, 2^-20 of the same sum."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,r", [(65, 130, 1), (200, 127, 4), (129, 133, 5), (64, 128, 8), (190, 257, 9),
                                   (321, 140, 16), (140, 321, 17)])
def test_dense_l(m, n, r):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1309_0302_gb300 as G
    g = torch.Generator(device="cuda").manual_seed(r)
    X = torch.randn(m, r, generator=g, device="cuda") @ torch.randn(n, r, generator=g, device="cuda").T
    X += 0.1 * torch.randn(m, n, generator=g, device="cuda")
    ctx = G.GoDec(X, torch.randn(n, r, generator=g, device="cuda"), r, m * n // 50, 1, tol=0.0, max_iter=4)
    ctx.iterate(2)
    U, s, V = (t.double() for t in ctx.L())
    L = ctx.L_dense().double()[:, :n]
    ctx.close()
    size = (U.abs() * s) @ V.abs().T
    bound = (r + 2) * 2.0 ** -24 if r <= 8 else 2.0 ** -20
    assert bool(((L - (U * s) @ V.T).abs() <= bound * size + 1e-30).all())
