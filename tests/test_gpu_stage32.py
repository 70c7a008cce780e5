"""The single-precision stage as one launch (csrc/hw_stage32.cu) on grids around its 16 x 16 tiles' edges against the same
stage in three launches (csrc/hw_kernels2d.cu; a profiled solver takes those, which the single-precision parity tests
hold to the oracle), stage by stage and over a few CFL steps, at those tests' tolerance (2e-5 normwise)."""
import numpy as np
import pytest

from paper_2208_01260_gb300 import scenarios as S
from _parity import normwise, oracle_grid, oracle_state, stage_scales

pytestmark = pytest.mark.gpu
TOL32 = 2e-5


@pytest.mark.parametrize("nx,ny", [(2, 3), (15, 17), (16, 16), (17, 15), (18, 14), (31, 33), (47, 2), (3, 50)])
@pytest.mark.parametrize("bc,char", [(S.REFLECTIVE, 1), (S.PERIODIC, 0), (S.OUTFLOW, 1)])
def test_stage_in_one_launch(orc, nx, ny, bc, char):
    import paper_2208_01260_gb300 as hw
    sc = S.hump2d(nx, ny, seed=31, bc=bc)
    p = hw.make_params(precision=hw.HW_FP32, char_decomp=char)
    g, po = oracle_grid(orc, sc), orc.make_params(char_decomp=char)
    st, stat = oracle_state(orc, sc)
    dt = orc.cfl_dt2d(g, po, st, stat)
    a, b = hw.Solver.from_scenario(sc, p), hw.Solver.from_scenario(sc, p)
    hw.hw_set_profiling(b.h, True)
    for k in (1, 2, 3):
        a.rk3_stage(k, dt)
        b.rk3_stage(k, dt)
        assert max(normwise(a.state(), b.state(), stage_scales(a.state(), stat))) <= TOL32, k
    a.advance(4)
    b.advance(4)
    assert max(normwise(a.state(), b.state(), stage_scales(a.state(), stat))) <= TOL32
    assert np.isfinite(np.stack(a.state())).all()
    a.close()
    b.close()
