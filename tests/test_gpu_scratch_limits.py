"""Triangle kernels where device memory is short: what fits a call that marks in one
pass and allocates its output afterwards must still run, with the same result."""
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


def _one_pass_peak(n, nnz, weighted, kernel):
    """Bytes of the arrays of a call that marks in one pass over all lists: row map,
    orientation and reverse list, then the larger of the marking's arrays (a byte of
    flag per edge; heavy and in-degree lists, counters of min-count) and of the rebuild's
    (the flags again, the output, keep bits, prefixes)."""
    m, nc = nnz // 2, -(-nnz // 256)
    base = 4 * (nc + 1) + 8 * (n + 1) + 4 * nnz + 4 * (8 * nc + 1) + 8 * (nc + 1) + 8 * (nnz - m)
    if kernel == "tr_maxw":
        base += 4 * nnz
    mark = m + 8 * n + 1664 + (4 * m if kernel == "tr_mincount" else 0)
    out = 8 * (n + 1) + 4 * nnz * (2 if weighted else 1)
    rebuild = m + m // 8 + out + 4 * (8 * nc + 1) + 8 * (nc + 1) + 8 * (nc // 1024 + 2)
    return base + max(mark, rebuild)


def _padded(g, n):
    """g with isolated vertices up to n."""
    off = torch.cat([g.off, g.off[-1:].expand(n - g.n)])
    return gg.CSR(n, off.contiguous(), g.col, g.w)


def _cliques(c, n):
    """c cliques of n."""
    a, b = (torch.from_numpy(x.astype(np.int64)) for x in np.triu_indices(n, 1))
    base = (torch.arange(c) * n)[:, None]
    return gg.csr_from_edges(c * n, (base + a).reshape(-1), (base + b).reshape(-1))


# two passes when there is room, their vertex records in the orientation's unused half (mean degrees
# 299 and 8.4) or not (2.4); one pass in any case (0.3); all too large for the scratch to be one allocation
GRAPHS = {
    "deg299": lambda: _cliques(16, 300),
    "deg8.4": lambda: _padded(_cliques(16, 300), 170000),
    "deg2.4": lambda: _padded(_cliques(16, 300), 600000),
    "deg0.3": lambda: _padded(gg.rmat(14, 16, seed=1), 1400000),
}


@pytest.mark.parametrize("kernel", ["tr_random", "tr_maxw", "tr_p2", "tr_mincount"])
@pytest.mark.parametrize("name", list(GRAPHS))
def test_fits_where_one_pass_fits(sg, name, kernel):
    g = gg.attach_weights(GRAPHS[name](), seed=1) if kernel == "tr_maxw" else GRAPHS[name]()
    limit = _one_pass_peak(g.n, g.nnz, g.w is not None, kernel)
    ctx = sg.Context(0)
    ctx.set_profiling(True)
    G = sg.Graph.from_csr(ctx, g)
    sg.compress(G, kernel, 0.5, 3).free()
    assert (ctx.kernel_time("tri_rest")[1] > 0) == (name != "deg0.3" and kernel != "tr_maxw")
    ctx.set_alloc_limit(limit)
    H = sg.compress(G, kernel, 0.5, 3)
    ctx.set_alloc_limit(limit // 4)
    with pytest.raises(sg.SgError):
        sg.compress(G, kernel, 0.5, 3)
    ctx.set_alloc_limit(0)
    off, col, w = H.download()
    H.free()
    G.free()
    ctx.close()
    o_off, o_col, _ = oracle.compress(g, kernel, 0.5, 3)
    assert np.array_equal(off, o_off) and np.array_equal(col, o_col)


def test_nothing_is_left_behind(sg):
    """Limits at which one or another optional array does not fit: every call works, and
    what it allocated before it gave up on a second pass is freed."""
    g = GRAPHS["deg299"]()
    low = _one_pass_peak(g.n, g.nnz, False, "tr_random")
    ctx = sg.Context(0)
    G = sg.Graph.from_csr(ctx, g)
    sizes = set()
    for _ in range(2):  # the first time also loads the kernels, which takes memory
        ctx.synchronize()
        before = sg.device_free_memory(0)
        for k in range(300):  # (the marking's peak lies 1.2 m below the rebuild's)
            ctx.set_alloc_limit(low - 2 * g.m + k * g.m // 100)
            try:
                H = sg.compress(G, "tr_random", 0.5, 3)
            except sg.SgError:
                assert k < 200  # below the one-pass peak
                continue
            sizes.add(H.nnz)
            H.free()
        ctx.set_alloc_limit(0)
        ctx.synchronize()
    assert len(sizes) == 1
    assert sg.device_free_memory(0) >= before
    G.free()
    ctx.close()


# limits around the 256 MB (and a quarter of headroom) of a small graph's triangle list: below it, just above it
# with little left for the rounds' own lists, and with room for everything
@pytest.mark.parametrize("kernel", ["tr_eo", "tr_eo_maxw", "tr_eo_mincount"])
@pytest.mark.parametrize("one_launch", [True, False])
def test_edge_once_list_leaves_room(sg, kernel, one_launch):
    g = gg.attach_weights(gg.rmat(12, 16, seed=12), seed=1)
    o_off, o_col, _ = oracle.compress(g, kernel, 1.0, 3)
    ctx = sg.Context(0)
    ctx.set_eo_one_launch(one_launch)
    G = sg.Graph.from_csr(ctx, g)
    for mb in (60, 120, 261, 262, 263, 264, 266, 268, 270, 275, 280, 290, 300, 320, 325, 330, 340, 400):
        ctx.release_workspace()
        ctx.set_alloc_limit(mb << 20)
        H = sg.compress(G, kernel, 1.0, 3)
        ctx.release_workspace()
        ctx.set_alloc_limit(0)
        off, col, _ = H.download()
        H.free()
        assert np.array_equal(off, o_off) and np.array_equal(col, o_col), mb
    G.free()
    ctx.close()


def test_pagerank_of_a_dense_graph(sg):
    """Scratch that depends on the vertices, with what the arcs add well below 1/64 byte
    each: the lists of long rows hold no more rows than there are."""
    g = gg.complete(6000)
    ctx = sg.Context(0)
    G = sg.Graph.from_csr(ctx, g)
    x, r = sg.pagerank(G, 0.85, 6)
    ctx.set_alloc_limit(44 * g.n + g.nnz // 256 + (256 << 10))
    x2, r2 = sg.pagerank(G, 0.85, 6)
    ctx.set_alloc_limit(0)
    G.free()
    ctx.close()
    assert torch.equal(x, x2) and r == r2
