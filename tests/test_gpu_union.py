"""The union kernels' two passes (lists streamed until their edge is deleted, then
the live arcs of the deleted edges' ends) at the sizes where they change: list
lengths around the short-list limits, table chunks and the hub launch."""
import numpy as np
import pytest
import torch

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sg():
    import paper_1912_08950_gb300 as m

    return m


@pytest.fixture(scope="module")
def ctx(sg):
    c = sg.Context(0)
    yield c
    c.close()


def _equal(sg, ctx, g, kern, p, seed):
    G = sg.Graph.from_csr(ctx, g)
    H = sg.compress(G, kern, p, seed)
    off, col, w = H.download()
    H.free()
    G.free()
    o_off, o_col, o_w = oracle.compress(g, kern, p, seed)
    assert np.array_equal(off, o_off) and np.array_equal(col, o_col)
    if o_w is not None:
        assert np.array_equal(w.view(np.uint32), o_w.view(np.uint32))


# out-degrees up to n - 1: lists of 128, 129, 130 elements, windows that end and
# wrap inside a block, one arc beyond them, and many lists above the limit
@pytest.mark.parametrize("n,q", [(129, 1.0), (130, 1.0), (131, 1.0), (162, 1.0), (300, 0.9), (420, 0.7)])
@pytest.mark.parametrize("kern,p", [("tr_random", 0.02), ("tr_random", 0.5), ("tr_random", 1.0), ("tr_p2", 0.3),
                                    ("tr_mincount", 0.4), ("tr_maxw", 1.0)])
def test_dense(sg, ctx, n, q, kern, p):
    g = gg.complete(n) if q == 1.0 else gg.gnp(n, q, seed=n)
    _equal(sg, ctx, gg.attach_weights(g, seed=n) if kern == "tr_maxw" else g, kern, p, 7)


# 75 vertices of out-degree above 1024 (chunked tables) and 175 (a hub launch)
@pytest.mark.parametrize("n,p", [(1100, 0.01), (1200, 0.005), (1200, 0.01)])
def test_hubs(sg, ctx, n, p):
    i = np.triu_indices(n, 1)
    g = gg.csr_from_edges(n, torch.from_numpy(i[0].astype(np.int64)), torch.from_numpy(i[1].astype(np.int64)))
    _equal(sg, ctx, g, "tr_random", p, 3)
