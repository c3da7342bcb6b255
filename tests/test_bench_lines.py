"""What bench.py says of the history convolution beside its times (no device needed)."""
import os
import re

import bench
from paper_1808_00270_gb300 import build as B


def test_the_source_hash_covers_the_convolution():
    """Every file with a kernel of the convolution, so that a measured traffic is
    not reported for kernels edited since."""
    kernel = re.compile(r"__global__[^;{]*?\b(?:hist_conv\w*|conv_\w+|b_conv\w*)\(", re.S)
    files = {f for f in os.listdir(B.CSRC) if kernel.search(open(os.path.join(B.CSRC, f)).read())}
    assert {"history.cuh", "k_history_blk.cu"} <= files <= set(bench.CONV_SOURCES)


def test_bytes_of_a_step():
    n, m, nacc = 1000, 101, 2
    whole = n * (4 * 3 * 100 + 4 * 3 * nacc)
    assert bench.conv_bytes(n, m, 4, nacc, False, 0, 64, 1, 0) == whole
    # 16 steps from slot 40 of one range of 100: rows 0 .. 39 once for the block,
    # 40 .. 99 by each step; parts written and read, sums written
    got = bench.conv_bytes(n, m, 4, nacc, False, 40, 16, 1, 16)
    assert abs(got - n * (12 * (40 / 16 + 60) + 12 * nacc * 3)) < 1e-6 * got
    # two ranges, steps of 8 from slot 0: the second range is complete in the parts
    got = bench.conv_bytes(n, m, 2, nacc, False, 0, 8, 2, 8)
    assert abs(got - n * (6 * (50 + 50 / 8) + 12 * nacc * 3)) < 1e-6 * got
