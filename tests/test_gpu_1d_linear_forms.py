"""The 1D kernels of the linear weights in their two forms: up to 4864 interfaces four lanes of a warp share one, up to 9728
nodes two lanes share one, above that a thread each. Right-hand side and stages against the oracle on both sides of
either limit and on the smallest grids, at the bounds of the other parity tests (a group is held to 1e-12 of its scale,
or to ten times the oracle's own change when eta moves by one unit in the last place, whichever is larger)."""
import numpy as np
import pytest

from paper_2208_01260_gb300 import scenarios as S
from _parity import normwise, oracle_grid, oracle_state, rhs_scales, stage_scales
from test_gpu_1d_forms import _ulp, _within

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("char", [1, 0])
@pytest.mark.parametrize("nx", [2, 3, 33, 4863, 4864, 9728, 9729])
def test_1d_linear_forms_against_oracle(nx, char, orc):
    import paper_2208_01260_gb300 as hw
    sc = S.perturbed1d(n=nx, perturb=0.05) if nx < 100 else S.accuracy1d(nx)
    g = oracle_grid(orc, sc)
    p = orc.make_params(eps_w=sc.eps_w, linear_weights=1, char_decomp=char)
    st, stat = oracle_state(orc, sc)
    s = hw.Solver.from_scenario(sc, hw.make_params(eps_w=sc.eps_w, linear_weights=1, char_decomp=char))
    ref, moved = orc.rhs1d(g, p, st, stat)[0], orc.rhs1d(g, p, _ulp(st), stat)[0]
    scales = rhs_scales(st, stat, sc.dx)
    _within(normwise(s.rhs(), ref, scales), normwise(moved, ref, scales), "rhs")
    dt = orc.cfl_dt1d(g, p, st, stat)
    base = None
    for k in (1, 2, 3):
        ref, b, _ = orc.stage1d(g, p, k, dt, st, stat, base)
        moved = orc.stage1d(g, p, k, dt, _ulp(st), stat, base)[0]
        base = b if k == 1 else base
        s.rk3_stage(k, dt)
        scales = stage_scales(st, stat)
        _within(normwise(s.state(), ref, scales), normwise(moved, ref, scales), k)
        st = ref
        s.set_state(ref)
    s.close()
