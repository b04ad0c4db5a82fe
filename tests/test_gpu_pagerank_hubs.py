"""PageRank's longest rows: sums of many parts, added by whichever warp comes last."""
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


def _biclique(a, b):
    """a hubs joined to each of b leaves (all hub rows b long, all leaf rows a long)."""
    off = torch.cat([torch.arange(a, dtype=torch.int64) * b, a * b + torch.arange(b + 1, dtype=torch.int64) * a])
    col = torch.cat([(a + torch.arange(b, dtype=torch.int32)).repeat(a), torch.arange(a, dtype=torch.int32).repeat(b)])
    return gg.CSR(a + b, off, col)


# one row of 74 chunks (few chunks: each in eight parts, 592 in all) and 20 rows of 62
# (1240 chunks: whole ones)
@pytest.mark.parametrize("a,b", [(1, 600001), (20, 500000)])
def test_rows_of_many_parts(sg, a, b):
    g = _biclique(a, b)
    ctx = sg.Context(0)
    G = sg.Graph.from_csr(ctx, g)
    x = sg.pagerank(G, 0.85, 6)[0].cpu().numpy()
    for _ in range(4):
        assert np.array_equal(x, sg.pagerank(G, 0.85, 6)[0].cpu().numpy())
    G.free()
    ctx.close()
    ref, _ = oracle.pagerank(g, 0.85, 6)
    # a part adds 32 values per lane, 5 + 8 steps of its trees, then 74 parts: 123
    # roundings with those of the update, 7.4e-6 of the value, contracted by 0.85
    assert np.all(np.abs(x.astype(np.float64) - ref) <= 5e-5 * ref)


# y in vertex order up to 98,304 vertices, in degree order (its first 32,768 entries in shared
# memory) above, from four iterations on
@pytest.mark.parametrize("iters", [3, 4, 7])
@pytest.mark.parametrize("n", [98303, 98304, 98305, 98307])
def test_either_side_of_the_degree_order(sg, n, iters):
    core = gg.rmat(16, 16, seed=5)
    g = gg.CSR(n, torch.cat([core.off, core.off[-1:].expand(n - core.n)]).contiguous(), core.col)
    ctx = sg.Context(0)
    G = sg.Graph.from_csr(ctx, g)
    x = sg.pagerank(G, 0.85, iters)[0].cpu().numpy()
    G.free()
    ctx.close()
    ref, _ = oracle.pagerank(g, 0.85, iters)
    # hub rows of one chunk: 32 + 5 + 8 roundings, the update's and the dangling sum's few more
    assert np.all(np.abs(x.astype(np.float64) - ref) <= 2e-5 * ref)
