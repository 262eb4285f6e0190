"""The FP64 sweep's one-sided derivatives on the host: no less accurate than with double-precision indicators.

fp64_pairs_check.cu compiles the kernels' own header for the host.  Over random lines with sharp kinks, rounded
corners and steep slopes on grids of the sizes the library is used at, neither the rms nor the largest error against
extended precision may exceed that of the same formulas all in double (by more than the 5 % by which the largest of
some hundred thousand errors may differ where both round in the last place).
"""
import os
import subprocess

import pytest

from paper_1909_13263_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def errors(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("pairs") / "check")
    subprocess.run([build._nvcc(), "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-w", "-Xcompiler", "-ffp-contract=off",
                    "-I", build.CSRC, "-o", exe, os.path.join(HERE, "fp64_pairs_check.cu")], check=True)
    rows = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split("\n")
    return {tuple(map(int, r.split()[:2])): tuple(map(float, r.split()[2:])) for r in rows if r}


@pytest.mark.parametrize("weights", [0, 1], ids=["arclength", "jp"])
@pytest.mark.parametrize("family", [0, 1, 2], ids=["kink", "corner", "slope"])
def test_errors_are_no_larger_than_the_double_forms(errors, family, weights):
    largest, largest_double, rms, rms_double = errors[family, weights]
    assert rms <= rms_double and largest <= 1.05 * largest_double
