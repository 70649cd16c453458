"""An S-step that writes entries of the working copy X - S beyond the range of its scale: the copy is
rebuilt from X and S at a new scale, whichever form runs.

X is close to 1 with one column whose odd rows have the other sign, and the test vector (or the item
feature) lies so that the row space it spans has half its weight on that column: L is about
(1 + sqrt(n)) / 2 there, sixteen and more times max |X|, and S takes the column.  The scale puts
max |X| at 2^12 at least, the range ends at 2^15.

Bar for LinGoDec: 1e-5, as in its parity test (one product of one-signed rows, up to 128 additions
between drains that are off by 2^-23 of the running sum: below 128 2^-24 = 7.6e-6).  For the power
chain the direction e_COL + 1/sqrt(n) comes out of a sum over the rows of terms of about +1/2 and -1/2
in turn, whose partial sums stay below 1/2 + (its result): off by 2^-24 (128 + 2 sqrt(n)) of the result
at most, and as much again for the two float16 terms of the +-1/2 at 2^-23: the bar is
2^-23 (128 + 2 sqrt(n)), 3.1e-5 for the widest.  The first iteration, before any rescale, comes closest
(the small entries of the test vector are added to one of about 1/2: 2.2e-5 of 2.3e-5, with a float32
working copy 2.2e-5 too); those on a rebuilt copy are below 1e-6."""
import numpy as np
import pytest

import oracle as O
import oracle.lingodec as LG
from gpu_helpers import lfro_rel, s_common_rel, to_gpu, to_np

pytestmark = pytest.mark.gpu

COL = 7
SHAPES = [(300, 1000), (130, 4097), (257, 2050)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1309_0302_gb300 as G
    G.library()


def _matrix(m, n):
    X = np.ones((m, n))
    X[1::2, COL] = -1.0
    X += 1e-3 * np.random.default_rng(m).standard_normal((m, n))
    return (X / np.abs(X).max()).astype(np.float32)


def _test_vector(n):
    """a with X a = p1 on the even rows and -1/2 on the odd ones, p1 = 1/2 + 1/sqrt(n): X^T X a is
    then the direction e_COL + 1/sqrt(n)."""
    p1, p2 = 0.5 + 1.0 / np.sqrt(n), -0.5
    a = np.full((n, 1), (p1 - (p1 - p2) / 2) / (n - 1))
    a[COL] = (p1 - p2) / 2
    return a.astype(np.float32)


def _follow(X, A1, k, step, state):
    """Four iterations, each against one float64 step from the S before it; the first must leave the
    working copy beyond its range."""
    S = (np.zeros(0, np.int64), np.zeros(0))
    for t in range(4):
        step()
        ref = O.godec_step(X, A1, S[0], S[1], k, 0)
        U, s, V, i, v = state()
        bar = 2.0 ** -23 * (128 + 2 * np.sqrt(X.shape[1]))
        assert lfro_rel(U, s, V, ref["U"], ref["sigma"], ref["V"]) <= bar, t
        e, flips = s_common_rel(i, v, ref["S_idx"], ref["S_val"])
        assert e <= bar and flips == 0, t
        Z = X.astype(np.float64)
        Z.ravel()[i] -= v
        assert np.abs(Z).max() >= 8.0 * np.abs(X).max()
        S = (i, v)


def _state(g):
    U, s, V = (to_np(t).astype(np.float64) for t in g.L())
    i, v = g.S()
    return U, s, V, to_np(i), to_np(v).astype(np.float64)


@pytest.mark.parametrize("m,n", SHAPES)
@pytest.mark.parametrize("sparse_first", [False, True])
def test_rescale_plain(m, n, sparse_first):
    import paper_1309_0302_gb300 as G
    X, A1 = _matrix(m, n), _test_vector(n)
    g = G.GoDec(to_gpu(X), to_gpu(A1), 1, m, 0, tol=-1.0, max_iter=9, flags=G.FLAG_SPARSE_FIRST if sparse_first else 0)
    try:
        _follow(X, A1, m, lambda: g.iterate(1), lambda: _state(g))
        g.reset()   # and once more from the first scale
        _follow(X, A1, m, lambda: g.iterate(1), lambda: _state(g))
    finally:
        g.close()


def test_rescale_in_a_batch():
    import paper_1309_0302_gb300 as G
    X, A1 = _matrix(*SHAPES[0]), _test_vector(SHAPES[0][1])
    other = np.random.default_rng(1).standard_normal((200, 90)).astype(np.float32)
    b = G.GoDecBatch([to_gpu(X), to_gpu(other)], [to_gpu(A1), to_gpu(other[:90, :3])], [1, 3], [X.shape[0], 50], [0, 1])
    try:
        _follow(X, A1, X.shape[0], lambda: b.iterate(1), lambda: _state(b.problem(0)))
        assert b.problem(1).info()["iter"] == 4
    finally:
        b.close()


@pytest.mark.parametrize("m,n", SHAPES)
def test_rescale_lingodec(m, n):
    import paper_1309_0302_gb300 as G
    X, lam = _matrix(m, n), 0.75
    F = np.full((n, 1), 1.0 / np.sqrt(n))
    F[COL] += 1.0
    F = F.astype(np.float32)
    g = G.LinGoDec(to_gpu(X), to_gpu(F), 1, lam)
    try:
        g.iterate(4)
        W = to_np(g.W()).astype(np.float64)
        i, v = (to_np(t) for t in g.S())
    finally:
        g.close()
    ref = LG.lingodec(X.astype(np.float64), F.astype(np.float64), 1, lam, 4)
    assert np.abs(X - ref["S"]).max() >= 8.0 * np.abs(X).max()
    assert np.linalg.norm(W - ref["W"]) <= 1e-5 * np.linalg.norm(ref["W"])
    assert np.array_equal(i, np.flatnonzero(ref["S"]))
    assert np.linalg.norm(v - ref["S"].ravel()[i]) <= 1e-5 * np.linalg.norm(ref["W"] @ F.T.astype(np.float64))
