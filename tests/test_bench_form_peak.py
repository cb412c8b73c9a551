"""The bench's peaks of the summed forms, on the CPU: from the operations of a
register and row and the measured issue rates."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


@pytest.mark.parametrize("kernel,n_max,n_add,about", [("k_inter_local16", 3.5, 3, 7942), ("k_inter_glob16", 3, 1, 11370)])
def test_form_peak(kernel, n_max, n_add, about):
    r = bench.form_peak(kernel, 1.98, 3.907, 152, 2070.0, 7000.0)
    cycles = n_max / 1.98 + n_add / 3.907   # per packed register and row, 32 lanes, 2 cells
    assert r["form_peak"] == pytest.approx(152 * 2070e6 * 64 / cycles / 1e9, abs=0.1)
    assert r["form_peak"] == pytest.approx(about, rel=1e-3)
    assert r["form_frac"] == pytest.approx(7000.0 / r["form_peak"], abs=1e-4)


def test_every_summed_kernel_is_a_score_kernel():
    assert {k for _, k, *_ in bench.SUB_KERNELS.values()} <= set(bench.SUMMED_OPS)
