"""One pass or two for a union kernel: either side of every line of the rule, the passes that
ran (the second one's launches have names of their own), and the oracle's output on both."""
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


def _passes(sg, g, kern, p, seed=5):
    ctx = sg.Context(0)
    G = sg.Graph.from_csr(ctx, g)
    ctx.set_profiling(True)
    H = sg.compress(G, kern, p, seed)
    off, col, w = H.download()
    two = ctx.kernel_time("tri_rest")[1] > 0
    H.free()
    G.free()
    ctx.close()
    o_off, o_col, o_w = oracle.compress(g, kern, p, seed)
    assert np.array_equal(off, o_off) and np.array_equal(col, o_col)
    if o_w is not None:
        assert np.array_equal(w.view(np.uint32), o_w.view(np.uint32))
    return 2 if two else 1


def _isolated(g, n):
    return gg.CSR(n, torch.cat([g.off, g.off[-1:].expand(n - g.n)]).contiguous(), g.col, g.w)


def _copies(c, n):
    """c cliques of n."""
    a, b = (torch.from_numpy(x.astype(np.int64)) for x in np.triu_indices(n, 1))
    base = (torch.arange(c) * n)[:, None]
    return gg.csr_from_edges(c * n, (base + a).reshape(-1), (base + b).reshape(-1))


# c cliques of n: lists of up to n - 1, W = c n (n - 1) (n - 2) / 6 elements, (n - 2) / 3 per arc
@pytest.mark.parametrize("c,n,kern,p,passes", [
    (24, 257, "tr_random", 0.5, 1), (24, 258, "tr_random", 0.5, 2),         # longest list 256, 257
    (10, 300, "tr_random", 0.2710, 1), (10, 300, "tr_random", 0.2713, 2),   # s W = 1.1993e9, 1.2006e9
    (10, 300, "tr_mincount", 0.2710, 1), (10, 300, "tr_mincount", 0.2713, 2),
    (10, 300, "tr_p2", 0.1355, 1), (10, 300, "tr_p2", 0.1357, 2),           # 1.1993e9, 1.2011e9
    (30, 300, "tr_maxw", 0.752, 1), (30, 300, "tr_maxw", 0.754, 2),         # 9.98e9, 1.001e10
    (1, 1300, "tr_random", 0.00923, 1), (1, 1300, "tr_random", 0.00925, 2),  # s = 3.994, 4.002; and a hub launch
    (10, 300, "tr_random", 1.0, 2), (10, 300, "tr_random", 0.0, 1), (12, 289, "tr_p2", 1.0, 2),
    (1, 200, "tr_random", 0.75, 1), (1, 200, "tr_random", 0.76, 1), (1, 200, "tr_maxw", 1.0, 1), (1, 200, "tr_p2", 1.0, 1),
    (1, 1100, "tr_random", 0.05, 2), (1, 1200, "tr_mincount", 0.05, 2),     # tables in chunks; a hub launch
])
def test_cliques(sg, c, n, kern, p, passes):
    g = _copies(c, n)
    assert _passes(sg, gg.attach_weights(g, seed=2) if kern == "tr_maxw" else g, kern, p) == passes


# 44.55 M elements, 32 per vertex on 1,392,218 vertices
@pytest.mark.parametrize("n,passes", [(1392000, 2), (1392500, 1)])
def test_isolated_vertices(sg, n, passes):
    assert _passes(sg, _isolated(_copies(10, 300), n), "tr_random", 0.5) == passes


# out-degrees above the hub launch's table (4096 entries): tables in chunks in both passes.
# 1.3e10 triangles are too many for the oracle: against a batch of this one graph, which
# takes one pass
@pytest.mark.parametrize("kern,p", [("tr_random", 0.5), ("tr_random", 0.005), ("tr_p2", 0.01)])
def test_out_degrees_above_the_hub_table(sg, kern, p):
    n = 4300
    off = torch.arange(n + 1, dtype=torch.int64, device="cuda") * (n - 1)
    i = torch.arange(n * (n - 1), device="cuda")
    row, col = i // (n - 1), i % (n - 1)
    ctx = sg.Context(0)
    ctx.set_profiling(True)
    G = sg.Graph.from_csr(ctx, gg.CSR(n, off, (col + (col >= row)).to(torch.int32)))
    H = sg.compress(G, kern, p, 9)
    assert ctx.kernel_time("tri_rest")[1] > 0
    batch = sg.Batch(ctx, [G])
    ctx.reset_profile()
    B = batch.compress([kern], [p], [9])[0]
    assert ctx.kernel_time("tri_rest")[1] == 0
    for mine, other in zip(H.download()[:2], B.download()[:2]):
        assert np.array_equal(mine, other)
    H.free()
    batch.free()
    G.free()
    ctx.close()
