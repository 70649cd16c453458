"""A product that a bounded wait made give up says so in its result: the calls do not synchronise
and have no status for it.  The self-test withholds the first block's loads, so that its waits run
out after about 40 ms; the rows of the tiles it had a share of become NaN (one tile, and several of
which it would have completed some), the others are as without it, and the next call is whole."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,r", [(700, 600, 20), (40000, 100, 64), (130, 20000, 8), (100, 64, 3)])
@pytest.mark.parametrize("trans", [0, 1])
def test_given_up_tiles_are_nan(m, n, r, trans):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1309_0302_gb300 as G
    g = torch.Generator(device="cuda").manual_seed(m)
    rows, K = (n, m) if trans else (m, n)
    Z = torch.randn(m, n, generator=g, device="cuda")
    B = torch.randn(K, r, generator=g, device="cuda")
    whole = (G.mul_ZtC if trans else G.mul_ZB)(Z, B)
    Y = torch.zeros(rows, r, device="cuda")
    st = G.library().godec_mul_check_timeout(Z.data_ptr(), m, n, Z.stride(0), B.data_ptr(), r, Y.data_ptr(), trans,
                                             torch.cuda.current_stream().cuda_stream)
    assert st == 0
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    geo = (G.prod_geometry if trans else G.tc_geometry)(rows, K, nsm)
    share = (geo["S"] // geo["G"] - 1) // geo["ks"] + 1     # row tiles of the first block's stages
    lost = min(128 * share, rows)
    # a tile that others complete from this block's full share may be whole again; none is here,
    # for the block gives up before its first stage
    assert bool(Y[:lost].isnan().all())
    assert torch.equal(Y[lost:], whole[lost:])
    assert torch.equal((G.mul_ZtC if trans else G.mul_ZB)(Z, B), whole)
