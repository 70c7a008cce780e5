"""The block fixed-point reconstruction and limiter of the CUDA kernels (csrc/hw_fixed.h), compiled for the
host, against the scheme's formulas in long double: smooth and rough data, jumps in values and in single
derivatives, flat data, data far below epsilon, and zero.

The FP64 form rounds a handful of sums of the stencil's scale, each by up to half of 2^-53 of it (the weighted
value five times, the limited one, from differences twice as large, about ten). The fixed-point form has to stay
below the first of them: 1 and 4 units of 2^-53 of the stencil's largest entry."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2208_01260_gb300", "csrc")


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_fixed_point_reconstruction(tmp_path, seed):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "fixed_check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I" + CSRC, os.path.join(HERE, "fixed_check.cpp"),
                    "-o", exe], check=True)
    r = subprocess.run([exe, "100000", str(seed)], capture_output=True, text=True, check=True)
    *kinds, last = [line.split() for line in r.stdout.splitlines()]
    assert len(kinds) == 8
    for k, (value, limited) in enumerate(kinds):
        assert float(value) <= 1.0 and float(limited) <= 4.0, (k, value, limited)
    rcp, wrong, bad = last
    assert float(rcp) <= -58 and int(wrong) == 0 and int(bad) == 0, last
