"""Work split of the product over the working copy (host logic): more SMs never mean fewer
CTAs, a whole device leaves 24 SMs to the kernels beside a chain, and every stage has an owner."""
import numpy as np
import pytest

import paper_1309_0302_gb300 as G


@pytest.mark.parametrize("rows,K", [(10000, 10000), (16384, 300), (300, 16384), (129, 65)])
def test_more_sms_never_fewer_ctas(rows, K):
    grids = [G.prod_geometry(rows, K, n)["G"] for n in range(17, 161)]
    assert all(a <= b for a, b in zip(grids, grids[1:]))
    S = G.prod_geometry(rows, K, 152)["S"]
    assert G.prod_geometry(rows, K, 152)["G"] == min(S, 128)
    assert G.prod_geometry(rows, K, 100)["G"] == min(S, 96)


@pytest.mark.parametrize("nsm", [1, 16, 100, 110, 121, 152])
def test_partial_slots_cover_every_tile(nsm):
    for rows, K in [(16384, 300), (8192, 512), (333, 12345), (1, 1)]:
        g = G.prod_geometry(rows, K, nsm)
        owner = ((np.arange(g["S"], dtype=np.int64) + 1) * g["G"] - 1) // g["S"]
        per_tile = [len(set(owner[t * g["ks"]:(t + 1) * g["ks"]])) for t in range(g["tiles"])]
        assert max(per_tile) == g["maxseg"]


def test_bad_arguments():
    for args in [(0, 10, 4), (10, 0, 4), (10, 10, 0)]:
        with pytest.raises(G.GodecError):
            G.prod_geometry(*args)
