"""A depth that becomes non-positive inside a 1D run is reported once a stage uses that state, not before: the launches that
write a state find its flags, the stage that reads it raises them (within a cluster's run of steps at 40 nodes, from
launch to launch at 300 and 600 nodes by graph and without; 300 nodes are one cluster of five blocks, 600 a launch per
stage). The oracle says at which stage of which step a run at an unstable CFL number first writes a bad depth; the first
depths are well away from 0 on either side, so rounding does not move that stage."""
import numpy as np
import pytest

from paper_2208_01260_gb300 import scenarios as S

pytestmark = pytest.mark.gpu


def _scenario(nx):
    x = np.arange(nx) / nx
    k = 2.0 * np.pi * (nx // 8)
    h, m, z = 0.5 + 0.2 * np.cos(k * x), 0.3 * np.sin(k * x), np.zeros(nx)
    deriv = [-0.2 * k * np.sin(k * x), 0.3 * k * np.cos(k * x), z]
    return h, m, z, deriv


def _first_bad(orc, nx, cfl, char):
    """(step, stage) of the first output with a depth that is not positive."""
    g = orc.make_grid(nx, 1, 0.0, 1.0, bc_x=S.PERIODIC)
    p = orc.make_params(char_decomp=char, cfl=cfl)
    h, m, b, deriv = _scenario(nx)
    st, stat = orc.to_state1d(h, m, b, deriv)
    for n in range(1, 12):
        dt, base = orc.cfl_dt1d(g, p, st, stat), None
        for k in (1, 2, 3):
            st, b1, _ = orc.stage1d(g, p, k, dt, st, stat, base)
            base = b1 if k == 1 else base
            low = st[0].min()
            if low < 1e-3:
                assert low < -1e-3, low
                return n, k
    raise AssertionError("no bad depth")


@pytest.mark.parametrize("graph", [True, False])
@pytest.mark.parametrize("nx,cfl,char", [(40, 1.0, 1), (40, 1.8, 1), (40, 1.2, 0), (300, 1.4, 0), (300, 2.0, 1), (600, 1.6, 1),
                                         (600, 2.0, 0), (600, 1.8, 0), (300, 2.2, 0)])
def test_flags_are_raised_by_the_stage_that_reads(orc, nx, cfl, char, graph):
    import paper_2208_01260_gb300 as hw
    n, k = _first_bad(orc, nx, cfl, char)
    assert (n, k) != (1, 1)
    reported = n if k < 3 else n + 1  # the step whose stage reads the bad depth

    def run(steps):
        s = hw.Solver(hw.make_grid(nx, 1, 0.0, 1.0, bc_x=S.PERIODIC, dim=1), hw.make_params(char_decomp=char, cfl=cfl))
        h, m, b, deriv = _scenario(nx)
        hw.hw_init(s.h, h, m, None, b, deriv)
        try:
            s.advance(steps, use_graph=graph)
        finally:
            s.close()

    if reported > 1:
        run(reported - 1)
    with pytest.raises(hw.HwError) as e:
        run(reported)
    assert e.value.code in (-2, -3)  # the depth, or what follows from it within the step
