"""A call that runs out of device memory reports it and leaves no CUDA error behind for the next
call: after a refused gradient and a refused context, products and torch's own launches work."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call,left", [("backward", 400 << 20), ("context", 128 << 20)])
def test_out_of_memory_is_reported_once(call, left):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1309_0302_gb300 as G
    g = torch.Generator(device="cuda").manual_seed(1)
    # 256 MB, and as much for a working copy (the gradient's result too)
    X = torch.randn(8192, 8192, generator=g, device="cuda")
    A1 = torch.randn(8192, 8, generator=g, device="cuda")
    want = X @ A1
    torch.cuda.synchronize()
    G.trim_scratch()
    torch.cuda.empty_cache()
    filler = torch.empty(torch.cuda.mem_get_info()[0] - left, dtype=torch.uint8, device="cuda")
    try:
        with pytest.raises(G.GodecError) as e:
            if call == "backward":
                G.backward(X, A1, 1, [], gU=want[:, :2], gV=A1[:, :2])
            else:
                G.GoDec(X, A1, 8, 1000, 1)
        assert e.value.status == 3
        # before any other call could report it: a launch of torch's, then one of the library's
        small = G.mul_ZB(X[:256], A1)
        assert bool(torch.isfinite(small + 1.0).all())
    finally:
        del filler
        torch.cuda.empty_cache()
    assert (G.mul_ZB(X, A1) - want).norm().item() <= 1e-2 * want.norm().item()
