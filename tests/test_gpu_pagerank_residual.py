"""The PageRank residual's FP64 sum has one order: where its terms carry more bits than
FP64 adds exactly (damping 1, values from 2^-40 to 1) it must still repeat bit for bit."""
import math

import numpy as np
import pytest

import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sg():
    import paper_1912_08950_gb300 as m

    return m


@pytest.mark.parametrize("damping", [1.0, 0.99999])
@pytest.mark.parametrize("iters", [1, 2, 5])
@pytest.mark.parametrize("name", ["star", "rmat", "small"])
def test_repeats(sg, name, iters, damping):
    g = {"star": lambda: gg.star(1300007), "rmat": lambda: gg.rmat(18, 4, seed=9), "small": lambda: gg.rmat(6, 4, seed=9)}[name]()
    ctx = sg.Context(0)
    G = sg.Graph.from_csr(ctx, g)
    runs = [sg.pagerank(G, damping, iters) for _ in range(8)]
    x = runs[0][0].cpu().numpy().astype(np.float64)
    if iters > 1:
        before = sg.pagerank(G, damping, iters - 1)[0].cpu().numpy().astype(np.float64)
    else:
        before = np.full(g.n, np.float64(np.float32(1.0 / g.n)))
    G.free()
    ctx.close()
    assert len({r for _, r in runs}) == 1
    # every term is exact in FP64; the sum takes at most ceil(n / 256) + 16 + 256 additions of it
    exact = math.fsum(np.abs(x - before))
    assert abs(runs[0][1] - exact) <= (g.n // 256 + 273) * 2.0**-53 * exact
