"""A bounded wait that gave up is reported by the call whose result it spoils, not by the next
one: the residual (its kernel leaves tiles unwritten) and an iteration.  The wait is the
self-test's, on an mbarrier that nothing arrives on; afterwards the context goes on."""
import numpy as np
import pytest

import synth
from gpu_helpers import to_gpu, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["residual", "iterate"])
def test_timeout_is_reported_at_once(call):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1309_0302_gb300 as G
    d = synth.small_case(300, 260, 5, 0.03, 5, 1, tag="timeout_report")
    g = G.GoDec(to_gpu(d["X"]), to_gpu(d["A1"]), d["r"], d["k"], d["q"], tol=-1.0, max_iter=50)
    try:
        g.iterate(2)
        R = to_np(g.residual())
        g.queue_timeout()
        with pytest.raises(G.GodecError) as e:
            g.residual() if call == "residual" else g.iterate(1)
        assert e.value.status == 5 and "gave up" in str(e.value)
        assert g.info()["iter"] == 2
        assert np.array_equal(to_np(g.residual()), R)
        g.iterate(1)
        assert g.info()["iter"] == 3
    finally:
        g.close()
