"""The scaled conversion and the quarter of csrc/hw_fixed.h, compiled for the host, against exact integer products and
IEEE arithmetic: every magnitude, constants at both ends of the range, subnormal and special values.

The product keeps at least 60 bits and is at most 3 of its units low (fx_mulhi_u drops below two, the constant's product
none more), 2^-6 of the result's last place, so the rounded result is within 1/2 + 2^-5 of a unit; the quarter is exact
or correctly rounded."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2208_01260_gb300", "csrc")


@pytest.mark.parametrize("seed", [1, 2])
def test_scaled_conversion_and_quarter(tmp_path, seed):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I" + CSRC,
                    os.path.join(HERE, "fixed_scale_check.cpp"), "-o", exe], check=True)
    worst, wrong, quarters = subprocess.run([exe, "400000", str(seed)], capture_output=True, text=True,
                                            check=True).stdout.split()
    assert float(worst) <= 0.5 + 2.0 ** -5 and int(wrong) == 0 and int(quarters) == 0, (worst, wrong, quarters)
