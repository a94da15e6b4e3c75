"""Every evaluation kernel of the library carries a name that numa_vol_kernel_name reports, so that
the name a handle gives finds the kernel it launches in a profiler."""
import re
import subprocess

from paper_1604_08501_gb300 import build

REPORTED = [r"vol_rhs_fp64_kernel<[2-8], ", r"vol_rhs_df64_kernel<[2-8], ", r"vol_rhs_mixed_kernel<[2-8], ",
            r"vol_rhs_mixed_tc_kernel\(", r"vol_rhs_high_kernel<(9|1[0-6]), (double|float), "]


def test_kernel_names():
    out = subprocess.run(["nm", "-C", build.build()], check=True, capture_output=True, text=True).stdout
    names = set(re.findall(r"vol_rhs_\w*kernel[<(].{12}", out))   # the stubs' names and first arguments
    strays = {n for n in names if not any(re.match(r, n) for r in REPORTED)}
    assert not strays, strays
    for r in REPORTED:
        assert any(re.match(r, n) for n in names), r
