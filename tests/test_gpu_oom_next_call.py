"""The call after one that ran out of device memory does not report that error again: the getters and
iterations of another context, and the row copy of an unaligned matrix, whose checks look at the last
CUDA error."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("refused,left", [("context", 128 << 20), ("backward", 400 << 20)])
@pytest.mark.parametrize("then", ["L_dense", "iterate", "reset", "threshold"])
def test_next_call_after_out_of_memory(refused, left, then):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1309_0302_gb300 as G
    g = torch.Generator(device="cuda").manual_seed(1)
    X = torch.randn(8192, 8192, generator=g, device="cuda")   # 256 MB, and as much for a working copy
    A1 = torch.randn(8192, 8, generator=g, device="cuda")
    other = G.GoDec(X[:128, :128].contiguous(), A1[:128].contiguous(), 8, 100, 1, tol=-1.0, max_iter=9)
    other.iterate(2)
    L = other.L_dense()
    odd = X[:64, :65].contiguous()
    picked = G.hard_threshold(odd, 10)
    torch.cuda.synchronize()
    G.trim_scratch()
    torch.cuda.empty_cache()
    filler = torch.empty(torch.cuda.mem_get_info()[0] - left, dtype=torch.uint8, device="cuda")
    try:
        with pytest.raises(G.GodecError) as e:
            if refused == "backward":
                G.backward(X, A1, 1, [], gU=A1[:, :2], gV=A1[:, :2])
            else:
                G.GoDec(X, A1, 8, 1000, 1)
        assert e.value.status == 3
        if then == "L_dense":
            assert torch.equal(other.L_dense(), L)
        elif then == "iterate":
            other.iterate(1)
            assert other.info()["iter"] == 3
        elif then == "reset":
            other.reset()
        else:
            assert all(torch.equal(a, b) for a, b in zip(G.hard_threshold(odd, 10), picked))
    finally:
        del filler
        torch.cuda.empty_cache()
        other.close()
