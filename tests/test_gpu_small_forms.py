"""The small-grid forms of the sweeps (two lanes per interface) and of the node update (split over warps) around the edges
of their tiles (64 records: 61 x-interfaces, 29 rows of 2 columns; 64 nodes) and on both sides of the size where the
general forms take over, without and with data that goes back to the FP64 pipe, against the oracle at the per-stage
tolerance of the parity tests; and a run against the same run profiled, which takes the sweeps' general form: the same
values bit for bit."""
import numpy as np
import pytest

from paper_2208_01260_gb300 import scenarios as S
from _parity import normwise, oracle_grid, oracle_state, stage_scales, tiny_derivatives

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(5, 4), (57, 3), (61, 29), (62, 30), (3, 64), (33, 58), (170, 171), (171, 171)])
@pytest.mark.parametrize("bc,char,lim,tiny", [(S.REFLECTIVE, 1, 1, False), (S.PERIODIC, 0, 1, False), (S.OUTFLOW, 1, 0, False),
                                              (S.REFLECTIVE, 1, 1, True)])
def test_stages_and_run(orc, nx, ny, bc, char, lim, tiny):
    import paper_2208_01260_gb300 as hw
    sc = S.hump2d(nx, ny, seed=37, bc=bc)
    if tiny:
        sc = tiny_derivatives(sc, 1e-312)
    g, po = oracle_grid(orc, sc), orc.make_params(char_decomp=char, limiter=lim)
    p = hw.make_params(char_decomp=char, limiter=lim)
    st, stat = oracle_state(orc, sc)
    dt = orc.cfl_dt2d(g, po, st, stat)
    s, base = hw.Solver.from_scenario(sc, p), None
    for k in (1,) if tiny else (1, 2, 3):
        ref, b, _ = orc.stage2d(g, po, k, dt, st, stat) if k == 1 else orc.stage2d(g, po, k, dt, st, stat, base)
        base = b if k == 1 else base
        s.rk3_stage(k, dt)
        errs = normwise(s.state(), ref, stage_scales(ref, stat))
        assert max(errs) <= 1e-12, (k, errs)
        st = ref
        s.set_state(ref)
    s.close()
    a, b = hw.Solver.from_scenario(sc, p), hw.Solver.from_scenario(sc, p)
    hw.hw_set_profiling(b.h, True)
    a.advance(3)
    b.advance(3)
    for x, y in zip(a.state(), b.state()):
        assert np.array_equal(x, y)
    a.close()
    b.close()
