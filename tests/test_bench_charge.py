"""What the bench charges an enumeration: no byte for probes that were not made."""
import os
import re

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_forward_probes_follow_the_share_streamed():
    # the headline's graph: W = 4.1e11, W+ = 1.17e12; two passes stream 0.32 of W
    work = {"probes": 410_000_000_000, "forward_probes": 1_170_000_000_000}
    assert bench.charged_forward_probes(work, work["probes"]) == work["forward_probes"]
    assert bench.charged_forward_probes(work, work["probes"] // 4) == work["forward_probes"] / 4
    assert bench.charged_forward_probes({"probes": 0, "forward_probes": 0}, 0) == 0


def test_every_launch_of_the_step_is_listed():
    """Each name under which the triangle kernels launch is one of the bench's, or has one as its prefix."""
    src = open(os.path.join(ROOT, "paper_1912_08950_gb300", "csrc", "sg_triangles.cu")).read()
    names = set(re.findall(r'SG_LAUNCH\(c, "(\w+)"\)', src)) | set(re.findall(r'"(tri_\w+)"', src))
    assert names
    missing = {x for x in names if not any(x.startswith(k) for k in bench.KERNEL_NAMES)}
    assert not missing, missing
