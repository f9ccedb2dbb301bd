"""bench.py's table of kernel groups: every group its profiled pass reads has a row, and DRAM figures stand only beside kernels
that are the captured ones."""

import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_every_profiled_group_has_a_row():
    prof = {k: (2.0, 5) for k in bench.PROFILE_GROUPS}
    work = {k: (1e9, 1e9) for k in bench.PROFILE_GROUPS}
    kernels, _ = bench.kernel_rooflines(prof, work, 5, 4096, 6809.3, "measured", "tf32ir", 2070.0, tensor_peak=838.0)
    assert set(bench.PROFILE_GROUPS) - set(kernels) == {"status"}
    assert set(bench.DRAM_BYTES_PER_ELEMENT_STEP) <= {"lu_tc_diag", "restrict"}


def test_the_adjoint_product_takes_the_binding_roof():
    """4.3 ms a step of the 64 x 64 benchmark: 7.7 GB and 3.9e11 useful flops, issued three times.  The issued flops bind."""
    prof = {"adjoint": (5 * 4.3, 5), "gemv": (1.0, 10)}
    work = {"adjoint": (5 * 7.7e9, 5 * 3.9e11), "gemv": (1e9, 0.0)}
    kernels, roof = bench.kernel_rooflines(prof, work, 5, 4096, 6809.3, "measured", "tf32ir", 2070.0, tensor_peak=838.0)
    row = kernels["adjoint"]
    assert row["frac_hbm"] == pytest.approx(7.7e9 / 4.3e-3 / 1e9 / 6809.3)
    assert row["frac_tensor_issued"] == pytest.approx(3 * 3.9e11 / 4.3e-3 / 1e12 / 838.0)
    assert row["bound"] == roof["bound"] == "tensor" and roof["kernel"] == "adjoint"
