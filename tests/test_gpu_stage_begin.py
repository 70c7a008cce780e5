"""Alpha of all grids of a batch, and the ring exchange with alpha of all blocks of a decomposed grid, each in one
launch: at the edges of their work items (1024 nodes), at the thinnest blocks and with walls, wraps and copies on
either side of a block, corners included."""
import dataclasses

import numpy as np
import pytest

from paper_2208_01260_gb300 import scenarios as S
from _parity import normwise, stage_scales

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graph", [False, True])
def test_batch_alpha_item_edges(graph):
    """31x33 = 1023, 32x32 = 1024, 41x25 = 1025 and 32x64 = 2048 nodes, the smallest grid, and a larger one. alpha is
    an exact maximum, so the step of each grid is the single solver's (to the tolerances of the batched tests)."""
    import paper_2208_01260_gb300 as hw
    shapes = [(31, 33), (32, 32), (41, 25), (32, 64), (4, 4), (130, 67)]
    scs = [S.hump2d(nx, ny, seed=70 + k, hump_max=0.05) for k, (nx, ny) in enumerate(shapes)]
    b = hw.BatchedSolver(scs)
    b.run(4, use_graph=graph)
    t, steps = b.times()
    assert list(steps) == [4] * len(scs)
    for i, sc in enumerate(scs):
        s = hw.Solver.from_scenario(sc, hw.make_params())
        ts, _ = s.advance(4, use_graph=False)
        assert abs(ts - t[i]) <= 1e-14 * t[i]
        ref = s.state()
        assert max(normwise(b.state(i), ref, stage_scales(ref, [sc.b, sc.deriv[6], sc.deriv[7]]))) <= 1e-12
    b.close()


@pytest.mark.parametrize("bcx", [S.PERIODIC, S.REFLECTIVE, S.OUTFLOW])
@pytest.mark.parametrize("bcy", [S.PERIODIC, S.REFLECTIVE, S.OUTFLOW])
@pytest.mark.parametrize("nx,ny,px,py", [(8, 9, 4, 4), (67, 35, 2, 2), (66, 64, 1, 2), (70, 131, 3, 1)])
def test_blocks_equal_grid(bcx, bcy, nx, ny, px, py):
    import paper_2208_01260_gb300 as hw
    sc = dataclasses.replace(S.hump2d(nx, ny, seed=81, bc=bcx, hump_max=0.05), bc_y=bcy)
    ref = hw.Solver.from_scenario(sc, hw.make_params())
    dd = hw.DecomposedSolver(sc, px, py)
    assert ref.advance(3) == dd.advance(3)
    for a, b in zip(ref.state(), dd.state()):
        assert np.array_equal(a, b)
    dd.close()
    ref.close()
