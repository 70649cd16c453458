"""The sparse first projection subtracts the float32 values of S themselves: X A1 - S A1 is, row by
row, the chain of float32 fmas over S's entries in column order that starts from X A1.  X and A1 are
small integers, so that X A1 is exact (terms below 2^11, sums below 2^24); the chain is emulated in
float64 and must be met to the bit but for one double rounding in 2^29 (at most 2 entries)."""
import numpy as np
import pytest

from gpu_helpers import fma32, to_gpu, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,r,density", [(129, 65, 3, 0.05), (300, 257, 8, 0.3), (70, 640, 9, 1.0)])
def test_projection_is_the_chain(m, n, r, density):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1309_0302_gb300 as G
    g = np.random.default_rng(m)
    X = (g.integers(-8, 9, (m, r)) @ g.integers(-8, 9, (r, n)) + g.integers(-50, 51, (m, n))).astype(np.float32)
    A1 = g.integers(-4, 5, (n, r)).astype(np.float32)
    ctx = G.GoDec(to_gpu(X), to_gpu(A1), r, max(1, int(density * m * n)), 1, tol=-1.0, max_iter=9,
                  flags=G.FLAG_SPARSE_FIRST)
    try:
        for _ in range(3):
            ctx.iterate(1)
            P = to_np(ctx.first_projection())
            idx, val = (to_np(t) for t in ctx.S())
            want = X @ A1
            assert np.array_equal(want, X.astype(np.float64) @ A1.astype(np.float64))
            rows, cols = idx // n, idx % n
            start = np.searchsorted(rows, np.arange(m + 1))
            for step in range(np.diff(start).max()):
                live = start[:-1] + step < start[1:]
                e = start[:-1][live] + step
                want[live] = fma32(-val[e][:, None], A1[cols[e]], want[live])
            assert (P != want).sum() <= 2
        assert ctx.info()["iter"] == 3
    finally:
        ctx.close()


def test_needs_the_flag():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1309_0302_gb300 as G
    ctx = G.GoDec(torch.randn(40, 32, device="cuda"), torch.randn(32, 3, device="cuda"), 3, 20, 1, tol=-1.0, max_iter=9)
    try:
        ctx.iterate(1)
        with pytest.raises(G.GodecError):
            ctx.first_projection()
    finally:
        ctx.close()
