"""The sweeps' and the limiter's fixed-point form (csrc/hw_fixed.h) over the range of magnitudes: a smooth 2D
flow scaled by powers of ten (depths by s, discharges by s^(3/2)), depths of many scales in one grid, and data
that takes interfaces and nodes back to the FP64 pipe, against the oracle at the per-stage tolerance of the
parity tests. epsilon is absolute, so the scales also run from weights that epsilon
makes linear to weights that it does not reach."""
import dataclasses

import numpy as np
import pytest

from paper_2208_01260_gb300 import scenarios as S
from _parity import normwise, oracle_grid, oracle_state, stage_scales

pytestmark = pytest.mark.gpu


def _scaled(nx, ny, bc, s):
    """Bumps, a hump and a rotating current on nx x ny nodes, depths times s (a number or a plane)."""
    sc = S.hump2d(nx, ny, 17, bc=bc)
    x, y = S.axis(nx, 0.0, 1.0, bc)[None, :], S.axis(ny, 0.0, 1.0, bc)[:, None]
    k, v = 2.0 * np.pi, s * np.sqrt(s)
    hu, hv = 0.2 * np.sin(k * x) * np.cos(k * y), -0.1 * np.cos(k * x) * np.sin(k * y)
    d = [sc.deriv[0] * s, v * 0.2 * k * np.cos(k * x) * np.cos(k * y), v * 0.1 * k * np.sin(k * x) * np.sin(k * y),
         sc.deriv[3] * s, -v * 0.2 * k * np.sin(k * x) * np.sin(k * y), -v * 0.1 * k * np.cos(k * x) * np.cos(k * y),
         sc.deriv[6] * s, sc.deriv[7] * s]
    return dataclasses.replace(sc, h=sc.h * s, hu=hu * v, hv=hv * v, b=sc.b * s, deriv=[p + 0.0 * sc.h for p in d])


@pytest.mark.parametrize("scale", [1e-100, 1e-60, 1e-20, 1e-6, 1.0, 1e5, 1e9])
@pytest.mark.parametrize("char", [1, 0])
def test_scaled_stage_matches_oracle(orc, scale, char):
    import paper_2208_01260_gb300 as hw
    _check(orc, hw, _scaled(37, 26, S.REFLECTIVE if char else S.PERIODIC, scale), char)


def test_depths_of_many_scales_in_one_grid(orc):
    """Depths fall from 1 to 1e-5 across the grid in steps of ten: interfaces between nodes of different scale. (The
    limiter divides by the node's wave speed, so the scheme's own conditioning grows like its inverse there.)"""
    import paper_2208_01260_gb300 as hw
    nx = 36
    s = np.repeat(10.0 ** -np.arange(6.0), nx // 6)[None, :]
    _check(orc, hw, _scaled(nx, 20, S.REFLECTIVE, s), 1, stages=(1,))  # the scheme has no wet/dry treatment


@pytest.mark.parametrize("tiny", [1e-260, 1e-312])
@pytest.mark.parametrize("char", [1, 0])
def test_fallback_matches_oracle(orc, tiny, char):
    """The y-discharge scaled below the fixed-point form's exponents (also to subnormal numbers) on half of the
    grid: there the x-sweep and the limiter take the FP64 pipe, next to interfaces and nodes that do not."""
    import paper_2208_01260_gb300 as hw
    sc = _scaled(40, 23, S.REFLECTIVE, 1.0)
    f = np.where(np.arange(40) < 20, tiny, 1.0)[None, :]
    sc = dataclasses.replace(sc, hv=sc.hv * f, deriv=[p * f if q in (2, 5) else p for q, p in enumerate(sc.deriv)])
    _check(orc, hw, sc, char, stages=(1,))


def _check(orc, hw, sc, char, stages=(1, 2, 3)):
    g, p = oracle_grid(orc, sc), orc.make_params(char_decomp=char)
    st, stat = oracle_state(orc, sc)
    dt = orc.cfl_dt2d(g, p, st, stat)
    s = hw.Solver.from_scenario(sc, hw.make_params(char_decomp=char))
    base = None
    for k in stages:
        ref, base_out, _ = orc.stage2d(g, p, k, dt, st, stat) if k == 1 else orc.stage2d(g, p, k, dt, st, stat, base)
        base = base_out if k == 1 else base
        s.rk3_stage(k, dt)
        got = s.state()
        errs = normwise(got, ref, stage_scales(ref, [sc.b, sc.deriv[6], sc.deriv[7]]))
        assert max(errs) <= 1e-12, (k, errs)
        st = ref
        s.set_state(ref)
    s.close()
