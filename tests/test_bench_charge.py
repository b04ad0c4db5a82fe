"""What the bench charges an enumeration: no byte for probes that were not made."""
import bench

def test_forward_probes_follow_the_share_streamed():
    # the headline's graph: W = 4.1e11, W+ = 1.17e12; two passes stream 0.32 of W
    work = {"probes": 410_000_000_000, "forward_probes": 1_170_000_000_000}
    assert bench.charged_forward_probes(work, work["probes"]) == work["forward_probes"]
    assert bench.charged_forward_probes(work, work["probes"] // 4) == work["forward_probes"] / 4
    assert bench.charged_forward_probes({"probes": 0, "forward_probes": 0}, 0) == 0
