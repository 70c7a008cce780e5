"""Grids of any spacing a problem may have keep the fixed-point form: the range of the spacings' factors (csrc/hw_fixed.h,
compiled for the host), and right-hand side and stages on both sides of it against the oracle. A factor outside the
range costs four times the time, so the range is as wide as the conversion allows."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2208_01260_gb300 import scenarios as S

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2208_01260_gb300", "csrc")


def test_range_of_the_factors(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I" + CSRC,
                    os.path.join(HERE, "fixed_scale_range_check.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe, "7"], capture_output=True, text=True, check=True).stdout.split()
    assert r == ["0", "0", "0"], r


@pytest.mark.gpu
@pytest.mark.parametrize("lx,ly", [(1e-14, 1e-15), (1e27, 1e26), (1e-30, 1e-30), (1e31, 1e31), (1.0, 1e31)])
@pytest.mark.parametrize("char", [1, 0])
def test_spacings_against_oracle(orc, lx, ly, char):
    """On either side: 1e-14 to 1e27 units a side in fixed point, 1e-30 and 1e31 on the FP64 pipe. The bounds are those of
    the other parity tests, 1e-12 of the group's scale with derivatives in units of the spacing."""
    import paper_2208_01260_gb300 as hw
    from _parity import G, normwise, oracle_grid, oracle_state
    from test_gpu_scaled_faces import _stretched
    sc = _stretched(37, 26, S.REFLECTIVE if char else S.PERIODIC, lx, ly)
    g, p = oracle_grid(orc, sc), orc.make_params(char_decomp=char)
    st, stat = oracle_state(orc, sc)
    unit = [1.0] * 3 + [sc.dx] * 3 + [sc.dy] * 3
    eta = np.abs(st[0]).max()
    s = hw.Solver.from_scenario(sc, hw.make_params(char_decomp=char))

    def scaled(a):
        return [np.asarray(x) * u for x, u in zip(a, unit)]

    errs = normwise(scaled(s.rhs()), scaled(orc.rhs2d(g, p, st, stat)[0]), [G * eta * eta / min(sc.dx, sc.dy)] * 3)
    assert max(errs) <= 1e-12, errs
    dt, base = orc.cfl_dt2d(g, p, st, stat), None
    for k in (1, 2, 3):
        ref, b, _ = orc.stage2d(g, p, k, dt, st, stat, base)
        base = b if k == 1 else base
        s.rk3_stage(k, dt)
        errs = normwise(scaled(s.state()), scaled(ref), [eta] * 3)
        assert max(errs) <= 1e-12, (k, errs)
        st = ref
        s.set_state(ref)
    s.close()
