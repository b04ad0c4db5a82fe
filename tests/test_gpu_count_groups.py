"""Triangle counts per vertex and per edge, and edge-once compression, where light
vertices stream groups of 32 short lists as one sequence: out-degrees and in-lists around the group and slab
sizes, and lists left out because the other end streams them."""
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


def _joined(k, r):
    """A clique of k vertices, r further vertices joined to all of it, and a path through those."""
    i = np.triu_indices(k, 1)
    lo, hi = [i[0]], [i[1]]
    for x in range(r):
        lo.append(np.arange(k))
        hi.append(np.full(k, k + x))
    if r > 1:
        lo.append(k + np.arange(r - 1))
        hi.append(k + 1 + np.arange(r - 1))
    return gg.csr_from_edges(k + r, torch.from_numpy(np.concatenate(lo).astype(np.int64)),
                             torch.from_numpy(np.concatenate(hi).astype(np.int64)))


def _same(sg, G, g, p):
    for kern in ("tr_mincount", "tr_eo", "tr_eo_mincount"):
        off, col, _ = sg.compress(G, kern, p, 5).download()
        o_off, o_col, _ = oracle.compress(g, kern, p, 5)
        assert np.array_equal(off, o_off) and np.array_equal(col, o_col)


@pytest.mark.parametrize("k,r", [(3, 0), (32, 0), (33, 0), (34, 0), (64, 0), (65, 0), (66, 0), (9, 31), (9, 32),
                                 (9, 33), (31, 70), (33, 150), (20, 400)])
def test_joined(sg, ctx, k, r):
    g = _joined(k, r)
    G = sg.Graph.from_csr(ctx, g)
    assert np.array_equal(sg.vertex_triangle_counts(G).cpu().numpy(), oracle.vertex_triangle_counts(g))
    _same(sg, G, g, 1.0)


@pytest.mark.parametrize("n,q", [(60, 0.5), (150, 0.3), (150, 0.6), (900, 0.05)])
def test_random(sg, ctx, n, q):
    g = gg.gnp(n, q, seed=n)
    G = sg.Graph.from_csr(ctx, g)
    assert np.array_equal(sg.vertex_triangle_counts(G).cpu().numpy(), oracle.vertex_triangle_counts(g))
    _same(sg, G, g, 0.5)
