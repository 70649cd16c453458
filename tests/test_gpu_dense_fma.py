"""Dense L is one chain of r float32 fmas per entry at every rank: term l is (u_l sigma_l) v_l
with u_l sigma_l rounded, l ascending.  Compared for equality with that chain in float64 rounded
to float32 after every step.  That rounds twice, which differs from one rounding about once in
2^29 steps: at most 4 entries of a matrix may differ (5e6 steps at most), by one unit in the last
place of a partial sum.  Edges: 128 x 128 tiles, factors taken 32 columns at a time, rows of L
that are 16-byte aligned and not."""
import numpy as np
import pytest

from gpu_helpers import fma32, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,r", [(1, 1, 1), (200, 127, 4), (129, 132, 8), (130, 257, 9), (128, 128, 16), (257, 140, 31),
                                   (140, 321, 32), (300, 131, 33), (256, 260, 50), (127, 384, 64)])
def test_dense_l_is_a_float32_chain(m, n, r):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1309_0302_gb300 as G
    g = torch.Generator(device="cuda").manual_seed(r)
    X = torch.randn(m, r, generator=g, device="cuda") @ torch.randn(n, r, generator=g, device="cuda").T
    X += 0.1 * torch.randn(m, n, generator=g, device="cuda")
    ctx = G.GoDec(X, torch.randn(n, r, generator=g, device="cuda"), r, m * n // 50, 1, tol=0.0, max_iter=4)
    ctx.iterate(2)
    U, s, V = (to_np(t) for t in ctx.L())
    L = to_np(ctx.L_dense())
    ctx.close()
    assert U.shape[1] == r and L.shape == (m, n)
    Us = U * s
    want = np.zeros((m, n), np.float32)
    for l in range(r):
        want = fma32(Us[:, l, None], V[None, :, l], want)
    off = L != want
    assert off.sum() <= 4
    size = np.abs(Us).astype(np.float64) @ np.abs(V).T.astype(np.float64)
    assert (np.abs(L.astype(np.float64) - want)[off] <= 2.0 ** -23 * size[off]).all()
