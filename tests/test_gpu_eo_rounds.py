"""Edge-once rounds in one launch (short lists) and per round (long ones): the same
output as the oracle on either side of the switch and across it."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sg():
    import paper_1912_08950_gb300 as m

    return m


# scale 8: a list of a few hundred; 12: all rounds in one launch; 15: the last
# ones; a capacity of 50,000 lists windows, each finished in one launch
@pytest.mark.parametrize("scale,cap", [(8, 0), (12, 0), (12, 50000), (15, 0)])
@pytest.mark.parametrize("kern,p", [("tr_eo", 0.2), ("tr_eo", 1.0), ("tr_eo_maxw", 0.6), ("tr_eo_mincount", 0.6)])
def test_rounds(sg, scale, cap, kern, p):
    g = gg.attach_weights(gg.rmat(scale, 16, seed=scale), seed=1)
    ctx = sg.Context(0)
    ctx.set_eo_list_capacity(cap)
    G = sg.Graph.from_csr(ctx, g)
    H = sg.compress(G, kern, p, 11)
    off, col, w = H.download()
    rounds = ctx.stats()["eo_rounds"]
    H.free()
    G.free()
    ctx.close()
    o_off, o_col, o_w = oracle.compress(g, kern, p, 11)
    assert np.array_equal(off, o_off) and np.array_equal(col, o_col)
    assert np.array_equal(w.view(np.uint32), o_w.view(np.uint32))
    assert rounds >= 1
