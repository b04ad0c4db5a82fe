"""Which launches the edge-once rounds take: short lists in one cluster launch, long
ones a few launches per round and the short rest in one.  Lists of ragged lengths, so
that the lanes of a warp leave the rounds' loops at different times."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu

ONE_LAUNCH = 1 << 20  # list slots up to which the rounds left run in one launch


@pytest.fixture(scope="module")
def sg():
    import paper_1912_08950_gb300 as m

    return m


def _run(sg, g, kern, p, one_launch=True):
    ctx = sg.Context(0)
    if not one_launch:
        ctx.set_eo_one_launch(False)
    ctx.set_profiling(True)
    G = sg.Graph.from_csr(ctx, g)
    H = sg.compress(G, kern, p, 7)
    off, col, _ = H.download()
    launches = {k: ctx.kernel_time(k)[1] for k in ("tri_eo_rounds", "tri_eo_fresh_reserve", "tri_eo_list_reserve")}
    stats = ctx.stats()
    H.free()
    G.free()
    ctx.close()
    o_off, o_col, _ = oracle.compress(g, kern, p, 7)
    assert np.array_equal(off, o_off) and np.array_equal(col, o_col)
    return launches, stats


# one triangle; 35; some 10^4; 66 thousand (a warp may leave 31 slots of each of six
# buckets empty: 905 thousand on 4864 warps, which still fits beside them)
@pytest.mark.parametrize("name", ["k3", "k7", "rmat8", "rmat10"])
@pytest.mark.parametrize("kern", ["tr_eo", "tr_eo_maxw", "tr_eo_mincount"])
def test_short_list_takes_one_launch(sg, name, kern):
    g = {"k3": lambda: gg.complete(3), "k7": lambda: gg.complete(7), "rmat8": lambda: gg.rmat(8, 16, seed=2),
         "rmat10": lambda: gg.rmat(10, 16, seed=12)}[name]()
    launches, stats = _run(sg, gg.attach_weights(g, seed=1), kern, 1.0)
    assert stats["eo_listed"] > 0 and stats["eo_list_passes"] == 1
    assert launches == {"tri_eo_rounds": 1, "tri_eo_fresh_reserve": 0, "tri_eo_list_reserve": 0}


def test_long_list_ends_in_one_launch(sg):
    launches, stats = _run(sg, gg.rmat(15, 24, seed=15), "tr_eo", 1.0)
    assert stats["eo_listed"] > ONE_LAUNCH
    assert launches["tri_eo_fresh_reserve"] >= 1 and launches["tri_eo_rounds"] == 1


# as on a device that cannot host the cluster: every round in launches of its own
@pytest.mark.parametrize("name", ["k7", "rmat10"])
@pytest.mark.parametrize("kern", ["tr_eo", "tr_eo_maxw", "tr_eo_mincount"])
def test_without_the_cluster(sg, name, kern):
    g = {"k7": lambda: gg.complete(7), "rmat10": lambda: gg.rmat(10, 16, seed=12)}[name]()
    launches, stats = _run(sg, gg.attach_weights(g, seed=1), kern, 1.0, one_launch=False)
    assert launches["tri_eo_rounds"] == 0 and launches["tri_eo_fresh_reserve"] >= 1
