"""PageRank of a CSR that is not symmetric (a graph is taken as it is unless validation
is asked for): an arc into a vertex with no arcs of its own adds nothing."""
import numpy as np
import pytest
import torch

import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sg():
    import paper_1912_08950_gb300 as m

    return m


def _one_way(n, sinks, deg, seed):
    """Vertices n - sinks .. n - 1 have no arcs; the others `deg` each, any head."""
    rng = np.random.default_rng(seed)
    rows = n - sinks
    col = np.concatenate([np.sort(rng.choice(n, deg, replace=False)) for _ in range(rows)])
    off = np.minimum(np.arange(n + 1), rows) * deg
    return gg.CSR(n, torch.from_numpy(off.astype(np.int64)), torch.from_numpy(col.astype(np.int32)))


@pytest.mark.parametrize("iters", [1, 3, 4, 10])
@pytest.mark.parametrize("n,sinks,deg", [(7, 1, 3), (3000, 1000, 8), (2500, 40, 60), (1500, 500, 1100)])
def test_head_without_arcs(sg, n, sinks, deg, iters):
    g = _one_way(n, sinks, deg, seed=n)
    off, col, _ = g.numpy()
    d = np.diff(off)
    x = np.full(n, 1.0 / n)
    for _ in range(iters):
        y = np.where(d > 0, x / np.maximum(d, 1), 0.0)
        sums = np.add.reduceat(np.append(y[col], 0.0), np.minimum(off[:-1], len(col)))
        x = 0.15 / n + 0.85 * (np.where(d > 0, sums, 0.0) + x[d == 0].sum() / n)
    ctx = sg.Context(0)
    big = sg.Graph.from_csr(ctx, gg.rmat(14, 16, seed=1))
    G = sg.Graph.from_csr(ctx, g)
    sg.pagerank(big, 0.85, 5)  # what it leaves in the freed scratch is not zero
    got = sg.pagerank(G, 0.85, iters)[0].cpu().numpy()
    big.free()
    G.free()
    ctx.close()
    # at most 1100 terms a row, 35 of them one after another, and some ten steps more: 45 roundings an
    # iteration, 2.7e-6, contracted by 0.85
    assert np.all(np.abs(got.astype(np.float64) - x) <= 2e-5 * x)
