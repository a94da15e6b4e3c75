"""The FP64 kernel's operations per point in the bench line: what it issues on the FP64 pipe, which
from N = 2 is without the D sums (fixed point) and at N = 1 with them."""
import bench
from paper_1604_08501_gb300 import workload as wl


def test_flops_per_point_of_the_fp64_kernel():
    for N, flops in ((1, bench.flops_per_node_fp64(2)), (2, bench.FP64_PIPE_FLOPS_NATIVE),
                     (7, bench.FP64_PIPE_FLOPS_NATIVE)):
        roof, _ = bench.roofline_entries(f"vol_rhs_fp64_kernel<{N + 1}>", 1.0, wl.make_workload(N, 1, seed=0))
        assert roof["flops_per_point"] == flops
