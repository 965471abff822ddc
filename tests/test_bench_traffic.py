"""The benchmark reports a launch's measured DRAM bytes while the kernels' source is the one they were measured on: both
ends of that source have to be found where the benchmark looks for them, and cover the kernels."""
import os

import bench


def test_the_kernels_source_is_found():
    assert bench.kernel_sha(bench.M2L_TRAFFIC["src"]) is not None
    with open(os.path.join(bench.ROOT, bench.M2L_TRAFFIC["src"])) as f:
        s = f.read()
    part = s[s.index(bench.KERNEL_BEGIN):s.index(bench.KERNEL_END)]
    assert "k_m2l_tc(" in part and "k_m2l_tc_pair(" in part and "pair_tile(" in part
