"""The benchmark's operation counts against what the kernels form."""
import os
import re

import bench

CSRC = os.path.join(os.path.dirname(os.path.abspath(bench.__file__)), "paper_1605_08423_gb300", "csrc")


def test_derivative_rows_count_what_both_kernels_form():
    """Four rows (gradient, Laplacian) of N G x n multiply-adds an electron, SIMT and tensor-core."""
    src = open(os.path.join(CSRC, "k_orbitals.cu")).read()
    rows = int(re.search(r"if \(grad\) launch_orb<(\d)>", src).group(1))
    for use_tc in (False, True):
        f = bench._flops_per_launch("orbitals_meas", W=3, N=64, n=32, B=128, G=2, acc_ratio=0.5, use_tc=use_tc)
        assert f == 2.0 * rows * 3 * 64 * 128 * 32
