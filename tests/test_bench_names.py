"""What bench.py states about the sweep kernels agrees with their sources and summaries (no GPU)."""
import os
import re

import bench

CSRC = os.path.join(bench.ROOT, "paper_1711_02146_gb300", "csrc")


def test_gaussian_kernel_is_the_one_that_is_launched():
    source = open(os.path.join(CSRC, "pa_sweep_gauss.cu")).read()
    shape = re.search(r"case 10: e = launch_g_t<([0-9, ]+)>", source).group(1).replace(" ", "")
    assert bench.GAUSS_KERNEL == f"k_sweep_g<{shape}>"


def test_traffic_is_reported_for_the_profiled_shapes():
    tail = bench.tail_kernel(10, {"words": 16, "threads": 320, "ctas_per_sm": 2})
    traffic, _ = bench.step_traffic(tail=tail)
    # a step writes rows of 1000 bits, padded to 1024, for 1e6 replicas, and reads as many; the writes
    # that stay in L2 may not show, nor the reads that find them there
    assert traffic is not None and 32e6 < traffic < 2 * 1.1 * 128e6
    assert bench.step_traffic(kernel="k_sweep<10,8,160,3>", tail=tail) == (None, False)
    assert bench.step_traffic() == (None, False)  # without its second launch
