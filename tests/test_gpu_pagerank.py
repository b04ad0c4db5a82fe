"""PageRank with y in degree order and in vertex order (few iterations) against the
FP64 oracle, on rows of every length class and more vertices than a CTA keeps."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sg():
    import paper_1912_08950_gb300 as m

    return m


# R-MAT 17: 131,072 vertices, isolated ones, hub rows of several chunks; one
# star whose centre has 8193 arcs (a chunk of one); 33 rows of 32 and 33 arcs
@pytest.mark.parametrize("iters", [1, 2, 3, 4, 5, 50])
@pytest.mark.parametrize("name", ["rmat17", "star8193", "k33", "k34", "pairs"])
def test_against_oracle(sg, name, iters):
    g = {"rmat17": lambda: gg.rmat(17, 16, seed=3), "star8193": lambda: gg.star(8193), "k33": lambda: gg.complete(33),
         "k34": lambda: gg.disjoint_union(gg.complete(34), gg.complete(33), gg.path(5)),
         "pairs": lambda: gg.from_edge_list(1001, [(2 * i, 2 * i + 1) for i in range(300)])}[name]()
    ctx = sg.Context(0)
    G = sg.Graph.from_csr(ctx, g)
    x, r = sg.pagerank(G, 0.85, iters)
    x2, r2 = sg.pagerank(G, 0.85, iters)
    x, x2 = x.cpu().numpy(), x2.cpu().numpy()
    ref, rr = oracle.pagerank(g, 0.85, iters)
    G.free()
    ctx.close()
    assert np.array_equal(x, x2) and r == r2
    # FP32 values: a few ulp per update, contracted by the damping (below 1e-5)
    assert np.all(np.abs(x.astype(np.float64) - ref) <= 1e-5 * ref)
    assert abs(r - rr) <= 2e-5
