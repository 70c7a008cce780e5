"""The 1D scheme's single-launch forms (csrc/hw_step1d.cu): whole steps of a small grid in one launch (at most 248
and 504 nodes in blocks of 31 and 63), one launch per stage beyond, on both sides of each limit and on grids whose
last block holds a single node. Both forms run the same stage code, so a run equals the caller's own loop of
cfl_dt and rk3_step (one launch per stage on every size) to the per-stage tolerance of the parity tests; the stage
itself is held to the oracle there and in test_gpu_1d_forms.py."""
import dataclasses

import numpy as np
import pytest

from paper_2208_01260_gb300 import scenarios as S
from _parity import normwise, oracle_grid, oracle_state, stage_scales

pytestmark = pytest.mark.gpu


def _scenario(nx, bc, s=1.0):
    """A smooth flow over a wavy bottom, periodic on [0, 1], depths times s and discharges times s^(3/2)."""
    sc = S.accuracy1d(nx)
    v = s * np.sqrt(s)
    return dataclasses.replace(sc, bc_x=bc, h=sc.h * s, hu=sc.hu * v, b=sc.b * s,
                               deriv=[sc.deriv[0] * s, sc.deriv[1] * v, sc.deriv[2] * s])


@pytest.mark.parametrize("nx", [2, 3, 31, 32, 63, 218, 248, 249, 442, 504, 505, 1000])
@pytest.mark.parametrize("bc,char", [(S.PERIODIC, 1), (S.REFLECTIVE, 1), (S.OUTFLOW, 0)])
def test_run_equals_steps(nx, bc, char):
    import paper_2208_01260_gb300 as hw
    sc = _scenario(nx, bc)
    a, b = (hw.Solver.from_scenario(sc, hw.make_params(char_decomp=char)) for _ in range(2))
    t, n = a.advance(5)
    tb = 0.0
    for _ in range(5):
        dt = b.cfl_dt()
        b.rk3_step(dt)
        tb += dt
    assert n == 5 and abs(t - tb) <= 1e-13 * tb
    scl = stage_scales(b.state(), [sc.b, sc.deriv[2]])
    assert max(normwise(a.state(), b.state(), scl)) <= 1e-12
    assert max(normwise(a.base(), b.base(), scl)) <= 1e-12
    # an end time inside the third further step, then nothing left to do
    dt = a.cfl_dt()
    end = t + 2.5 * dt
    t2, n2 = a.advance(10 ** 6, t_end=end)
    assert 3 <= n2 <= 4 and abs(t + t2 - end) <= 1e-12 * end
    assert a.advance(10, t_end=end) == (0.0, 0)
    a.close()
    b.close()


@pytest.mark.parametrize("nx", [40, 600])
def test_depth_error_is_reported(nx):
    import paper_2208_01260_gb300 as hw
    sc = _scenario(nx, S.PERIODIC)
    s = hw.Solver.from_scenario(sc, hw.make_params())
    st = s.state()
    st[0][nx // 2] = sc.b[nx // 2] - 0.1
    s.set_state(st)
    with pytest.raises(hw.HwError):
        s.advance(1)
    s.close()


@pytest.mark.parametrize("scale", [1e-60, 1e-20, 1e-6, 1e5, 1e9])
@pytest.mark.parametrize("char", [1, 0])
def test_scaled_stage_matches_oracle(orc, scale, char):
    import paper_2208_01260_gb300 as hw
    _stage(orc, hw, _scenario(70, S.PERIODIC, scale), char)


@pytest.mark.parametrize("tiny", [1e-260, 1e-312])
@pytest.mark.parametrize("char", [1, 0])
def test_fallback_matches_oracle(orc, tiny, char):
    """Discharges, or all derivatives, of half of the grid below the fixed-point form's exponents: the limiter and
    (component-wise) the reconstruction take the FP64 pipe there."""
    import paper_2208_01260_gb300 as hw
    sc = _scenario(70, S.PERIODIC)
    f = np.where(np.arange(70) < 30, tiny, 1.0)
    _stage(orc, hw, dataclasses.replace(sc, hu=sc.hu * f, deriv=[sc.deriv[0], sc.deriv[1] * f, sc.deriv[2]]), char)


def _stage(orc, hw, sc, char):
    g, p = oracle_grid(orc, sc), orc.make_params(char_decomp=char)
    st, stat = oracle_state(orc, sc)
    dt = orc.cfl_dt1d(g, p, st, stat)
    s = hw.Solver.from_scenario(sc, hw.make_params(char_decomp=char))
    s.rk3_stage(1, dt)
    ref, _, _ = orc.stage1d(g, p, 1, dt, st, stat)
    errs = normwise(s.state(), ref, stage_scales(ref, [sc.b, sc.deriv[2]]))
    assert max(errs) <= 1e-12, errs
    s.close()
