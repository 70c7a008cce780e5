"""The reverse sweeps' tiles (csrc/hw_adjoint.cu: 61 x-interfaces over flattened rows; 16 rows of y-interfaces of 4 columns
over flattened columns) on grids whose lines end anywhere in a tile: the directional derivative of the gauge loss from the
adjoint against the oracle's dual numbers at the tolerance of the adjoint tests (1e-7)."""
import numpy as np
import pytest

from paper_2208_01260_gb300 import scenarios as S
from test_gpu_adjoint import _eq_static, _oracle_problem, _smooth_direction

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(12, 12), (57, 13), (61, 16), (13, 58), (65, 15), (30, 17)])
@pytest.mark.parametrize("bc", [S.REFLECTIVE, S.PERIODIC, S.OUTFLOW])
def test_directional_derivative(orc, nx, ny, bc):
    import paper_2208_01260_gb300 as hw
    import torch
    from paper_2208_01260_gb300 import adjoint as A
    sc = S.hump2d(nx, ny, seed=73, hump_max=0.05, bc=bc)
    g, p, st, stat, dts, gidx, obs = _oracle_problem(sc, 2, 5, 6)
    solver = hw.Solver.from_scenario(sc, hw.make_params())
    state, static, _, _ = _eq_static(sc)
    A.load_problem(solver, state, static)
    gs, gb = torch.empty_like(state), torch.empty_like(static)
    loss, _ = A.hw_adjoint_run(solver.h, dts, gidx, obs, A.HW_ADJ_TAPE, [gs[q] for q in range(9)], [gb[q] for q in range(3)])
    for seed in (6, 7):
        dst, dstat = _smooth_direction(sc, seed)
        L, dL = orc.gauge_loss_dual2d(g, p, st, stat, dst, dstat, dts, gidx, obs)
        assert abs(loss - L) <= 1e-10 * abs(L)
        gv = float((gs.cpu().numpy() * np.stack(dst)).sum() + (gb.cpu().numpy() * np.stack(dstat)).sum())
        assert abs(gv - dL) <= 1e-7 * abs(dL) + 1e-12, (gv, dL)
    solver.close()
