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


# a clique of n: lists of up to n - 1, (n - 2) / 3 elements per arc
@pytest.mark.parametrize("n,kern,p,passes", [
    (257, "tr_random", 0.5, 1), (258, "tr_random", 0.5, 2),          # longest list 256, 257
    (300, "tr_random", 0.0503, 1), (300, "tr_random", 0.0504, 2),    # p W / m 4.998, 5.006
    (300, "tr_mincount", 0.0503, 1), (300, "tr_mincount", 0.0504, 2),
    (300, "tr_p2", 0.0251, 1), (300, "tr_p2", 0.0252, 2),            # 2.49, 2.504
    (300, "tr_maxw", 0.1510, 1), (300, "tr_maxw", 0.1511, 2),        # 14.999, 15.009
    (300, "tr_random", 1.0, 2), (300, "tr_maxw", 1.0, 2), (300, "tr_random", 0.0, 1),
    (200, "tr_random", 0.75, 1), (200, "tr_random", 0.76, 1), (200, "tr_maxw", 1.0, 1), (200, "tr_p2", 1.0, 1),
])
def test_cliques(sg, n, kern, p, passes):
    g = gg.complete(n)
    assert _passes(sg, gg.attach_weights(g, seed=2) if kern == "tr_maxw" else g, kern, p) == passes


# 44,850 arcs of a clique of 300, 4.455 M elements: below 51.2 elements per arc beside 43,200
# arcs of cliques of 10, below 32 per vertex on 139,500 vertices
@pytest.mark.parametrize("name,passes", [("with 900 cliques of 10", 2), ("with 1100 cliques of 10", 1),
                                         ("in 139000", 2), ("in 139500", 1)])
def test_dilution(sg, name, passes):
    k = gg.complete(300)
    if name.startswith("with"):
        g = gg.disjoint_union(k, *([gg.complete(10)] * int(name.split()[1])))
    else:
        g = _isolated(k, int(name.split()[1]))
    assert _passes(sg, g, "tr_random", 0.5) == passes


# 175 vertices of out-degree above 1024: a hub launch in both passes; 75: chunked tables
@pytest.mark.parametrize("n", [1100, 1200])
def test_hubs(sg, n):
    assert _passes(sg, gg.complete(n), "tr_random", 0.05) == 2


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
