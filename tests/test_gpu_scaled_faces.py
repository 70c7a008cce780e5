"""The interface values carry the spacings' factors: right-hand side and stages on domains of 1e-9 to 1e9 units (the factors in
fixed point) and 1e15 and 1e-15 units (factors outside its range: every interface takes the FP64 pipe), uneven in x and y,
against the oracle at the tolerances of the parity tests (1e-12 of the group's scale, with derivatives in units of the
spacing, as the scheme holds them)."""
import dataclasses

import numpy as np
import pytest

from paper_2208_01260_gb300 import scenarios as S
from _parity import G, normwise, oracle_grid, oracle_state

pytestmark = pytest.mark.gpu


def _stretched(nx, ny, bc, lx, ly):
    sc = S.hump2d(nx, ny, 23, bc=bc)
    x, y = S.axis(nx, 0.0, 1.0, bc)[None, :], S.axis(ny, 0.0, 1.0, bc)[:, None]
    k = 2.0 * np.pi
    hu, hv = 0.2 * np.sin(k * x) * np.cos(k * y), -0.1 * np.cos(k * x) * np.sin(k * y)
    d = [sc.deriv[0], 0.2 * k * np.cos(k * x) * np.cos(k * y), 0.1 * k * np.sin(k * x) * np.sin(k * y),
         sc.deriv[3], -0.2 * k * np.sin(k * x) * np.sin(k * y), -0.1 * k * np.cos(k * x) * np.cos(k * y),
         sc.deriv[6], sc.deriv[7]]
    s = [lx, lx, lx, ly, ly, ly, lx, ly]
    return dataclasses.replace(sc, hu=hu, hv=hv, deriv=[(p + 0.0 * sc.h) / q for p, q in zip(d, s)], x0=0.0, x1=lx, y0=0.0, y1=ly)


@pytest.mark.parametrize("lx,ly", [(1e-9, 1e-8), (1.0, 3e3), (1e9, 1e7), (1e15, 1e15), (1.0, 1e15), (1e-15, 1.0)])
@pytest.mark.parametrize("char", [1, 0])
def test_stretched_domain(orc, lx, ly, char):
    import paper_2208_01260_gb300 as hw
    sc = _stretched(37, 26, S.REFLECTIVE if char else S.PERIODIC, lx, ly)
    g, p = oracle_grid(orc, sc), orc.make_params(char_decomp=char)
    st, stat = oracle_state(orc, sc)
    unit = [1.0] * 3 + [sc.dx] * 3 + [sc.dy] * 3

    def scaled(a):
        return [np.asarray(x) * u for x, u in zip(a, unit)]

    eta = np.abs(st[0]).max()
    s = hw.Solver.from_scenario(sc, hw.make_params(char_decomp=char))
    ref, _ = orc.rhs2d(g, p, st, stat)
    errs = normwise(scaled(s.rhs()), scaled(ref), [G * eta * eta / min(sc.dx, sc.dy)] * 3)
    assert max(errs) <= 1e-12, errs
    dt = orc.cfl_dt2d(g, p, st, stat)
    base = None
    for k in (1, 2, 3):
        ref, b, _ = orc.stage2d(g, p, k, dt, st, stat) if k == 1 else orc.stage2d(g, p, k, dt, st, stat, base)
        base = b if k == 1 else base
        s.rk3_stage(k, dt)
        errs = normwise(scaled(s.state()), scaled(ref), [eta] * 3)
        assert max(errs) <= 1e-12, (k, errs)
        st = ref
        s.set_state(ref)
    s.close()
