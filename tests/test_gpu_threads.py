"""Contexts used by several threads at once."""
import threading

import pytest

import graphgen as gg


@pytest.mark.gpu
def test_concurrent_calls_of_different_sizes():
    """Threads with graphs of different sizes: what a launch needs of a kernel's
    process-wide limits must not depend on what another thread launches."""
    import paper_1912_08950_gb300 as sg

    sizes = [gg.complete(9), gg.rmat(10, 8, seed=1), gg.rmat(13, 16, seed=2), gg.rmat(15, 16, seed=3)]
    errors = []

    def work(g):
        try:
            ctx = sg.Context(0)
            G = sg.Graph.from_csr(ctx, g)
            first = None
            for _ in range(25):
                H = sg.compress(G, "tr_random", 0.05, 1)
                d = sg.divergence(G, H, iters=5)
                first = first or (H.nnz, d)
                assert (H.nnz, d) == first
                H.free()
            G.free()
            ctx.close()
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(g,)) for g in sizes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
