"""Stage 2 of the Runge-Kutta step rounds as 3/4 base + (U + dt R)/4: U + dt R once, of which a quarter is left, and the sum
once. With uniform roundings of 2^-53 at most that is a root mean square of sqrt(1 + 1/16) / sqrt(12) = 0.298 units in the
last place of the result (values in [1, 2)); a second full rounding makes it 0.408. Over thousands of nodes the mean
is within 2% of that, so 0.33 tells the two apart. The sizes take the three launch shapes of the node update."""
import numpy as np
import pytest

from paper_2208_01260_gb300 import scenarios as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(64, 66), (180, 201), (300, 270)])
@pytest.mark.parametrize("char", [1, 0])
def test_stage2_rounding(nx, ny, char):
    import paper_2208_01260_gb300 as hw
    sc = S.hump2d(nx, ny, seed=81, bc=S.REFLECTIVE)
    s = hw.Solver.from_scenario(sc, hw.make_params(char_decomp=char))
    st = s.state()
    # a surface that moves everywhere, above 1 and below 2
    x, y = np.linspace(0.0, 1.0, nx)[None, :], np.linspace(0.0, 1.0, ny)[:, None]
    st[0] = st[0] + 0.4 + 0.1 * np.cos(7.0 * x + 1.0) * np.cos(5.0 * y)
    st[1] = 0.3 * np.sin(6.0 * x) * np.cos(4.0 * y + 0.5)
    st[2] = 0.2 * np.cos(5.0 * x) * np.sin(7.0 * y)
    s.set_state(st)
    dt = s.cfl_dt()
    s.rk3_stage(1, dt)
    base, U = s.base()[0].astype(np.longdouble), s.state()[0].astype(np.longdouble)
    R = s.rhs()[0].astype(np.longdouble)
    s.rk3_stage(2, dt)
    got = s.state()[0]
    s.close()
    want = (3 * base + U + np.longdouble(dt) * R) / 4
    assert got.min() >= 1.0 and got.max() < 2.0
    err = ((got - want) * 2.0 ** 52).astype(np.float64)
    assert np.abs(err).max() <= 0.5 + 0.125 + 0.01
    assert np.sqrt(np.mean(err ** 2)) <= 0.33, np.sqrt(np.mean(err ** 2))
