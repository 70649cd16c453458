"""The scratch that calls without a context leave in the library's pool goes back to the device
on request, and the calls work as before after it."""
import pytest

pytestmark = pytest.mark.gpu


def test_trim_gives_memory_back():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1309_0302_gb300 as G
    Z, C = torch.randn(4000, 4000, device="cuda"), torch.randn(4000, 8, device="cuda")
    W = G.mul_ZtC(Z, C)   # a 64 MB copy of Z is part of its scratch
    torch.cuda.synchronize()
    kept = torch.cuda.mem_get_info()[0]
    G.trim_scratch()
    assert torch.cuda.mem_get_info()[0] - kept >= 64_000_000
    G.trim_scratch()
    assert torch.equal(G.mul_ZtC(Z, C), W)
