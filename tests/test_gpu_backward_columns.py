"""The backward's sparse products and low-rank values take four columns at a time where rows are
16-byte aligned: ranks on both sides of that (1 and 5 to 7 with a remainder, 8 without), three
steps so that both sparse products and both evaluations run.  Against the float64 gradient on the
same supports; tolerance 1e-4 as for the other gradients (float32 through T solves whose error is
of order 6e-8 cond(Y2), cond(Y2) below 1e3 on these inputs)."""
import numpy as np
import pytest

import oracle as O
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,r", [(70, 91, 1), (130, 97, 5), (97, 130, 7), (161, 128, 8)])
def test_gradient_by_rank(m, n, r):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1309_0302_gb300 as G
    T = 3
    d = synth.small_case(m, n, r, 0.03, r, 0, tag=f"bwc{r}")
    g = np.random.default_rng(r)
    Lstar = g.standard_normal((m, r)) @ g.standard_normal((n, r)).T
    X, A1 = torch.from_numpy(d["X"]).cuda(), torch.from_numpy(d["A1"]).cuda()
    ctx = G.GoDec(X, A1, r, d["k"], 0, tol=0.0, max_iter=T)
    masks = []
    for _ in range(T):
        ctx.iterate(1)
        masks.append(ctx.S()[0].cpu().numpy())
    ctx.close()
    Xg = X.clone().requires_grad_(True)
    ((G.unrolled_godec(Xg, A1, r, d["k"], T) - torch.from_numpy(Lstar).float().cuda()) ** 2).sum().backward()
    ref = O.unrolled_vjp(d["X"].astype(np.float64), d["A1"].astype(np.float64), d["k"], T, Lstar, masks)
    got = Xg.grad.cpu().numpy().astype(np.float64)
    assert float(np.linalg.norm(got - ref) / np.linalg.norm(ref)) <= 1e-4
