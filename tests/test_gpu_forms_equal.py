"""Forms of one computation chosen by the grid's size give the same values, bit for bit: the single-precision stage in one
launch against its three kernels (a profiled solver takes those), at sizes with every remainder of the 16 x 16 tile; and
the adjoint's forward pass, whose recorded states must not depend on the form: a periodic problem of 96 x 64 nodes (split
sweeps and node update) and the same repeated to 192 x 192 (split sweeps, node blocks of 64) and 384 x 256 (neither), with
spacings of 2^-6 so that the repeated grid's constants are the same."""
import dataclasses

import numpy as np
import pytest

from paper_2208_01260_gb300 import scenarios as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(2, 2), (16, 16), (17, 33), (31, 15), (47, 2), (3, 50), (130, 97), (257, 240)])
@pytest.mark.parametrize("bc,char,limiter", [(S.PERIODIC, 1, 1), (S.REFLECTIVE, 0, 1), (S.OUTFLOW, 1, 0)])
def test_single_precision_stage(nx, ny, bc, char, limiter):
    import paper_2208_01260_gb300 as hw
    sc = S.hump2d(nx, ny, seed=91, bc=bc)
    out = []
    for profile in (False, True):
        s = hw.Solver.from_scenario(sc, hw.make_params(precision=hw.HW_FP32, char_decomp=char, limiter=limiter))
        hw.hw_set_profiling(s.h, profile)
        dt = 0.5 * s.cfl_dt()
        states = []
        for k in (1, 2, 3, 1):
            s.rk3_stage(k, dt)
            states += s.state() + s.base()
        out.append(states)
        s.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def _tiled(nx, ny):
    """A flow of period 1.5 x 1 on nx x ny nodes of spacing 2^-6."""
    lx, ly = nx / 64.0, ny / 64.0
    X, Y = np.meshgrid(np.arange(nx) % 96 / 64.0, np.arange(ny) % 64 / 64.0)
    a, c = 2.0 * np.pi / 1.5, 2.0 * np.pi
    b = 0.3 + 0.2 * np.cos(a * X) * np.sin(c * Y)
    bx, by = -0.2 * a * np.sin(a * X) * np.sin(c * Y), 0.2 * c * np.cos(a * X) * np.cos(c * Y)
    eta, ex, ey = 1.0 + 0.05 * np.sin(2 * a * X + c * Y), 0.1 * a * np.cos(2 * a * X + c * Y), 0.05 * c * np.cos(2 * a * X + c * Y)
    m, mx, my = 0.2 * np.sin(a * X) * np.cos(c * Y), 0.2 * a * np.cos(a * X) * np.cos(c * Y), -0.2 * c * np.sin(a * X) * np.sin(c * Y)
    w, wx, wy = -0.1 * np.cos(a * X), 0.1 * a * np.sin(a * X), np.zeros_like(X)
    sc = S.hump2d(nx, ny, seed=92, bc=S.PERIODIC)
    return dataclasses.replace(sc, h=eta - b, hu=m, hv=w, b=b, deriv=[ex - bx, mx, wx, ey - by, my, wy, bx, by], x0=0.0, x1=lx,
                               y0=0.0, y1=ly)


@pytest.mark.parametrize("limiter", [1, 0])
def test_recorded_states(limiter):
    import paper_2208_01260_gb300 as hw
    from paper_2208_01260_gb300 import adjoint as A
    steps, dt = 3, None
    values = []
    for nx, ny in ((96, 64), (192, 192), (384, 256)):
        s = hw.Solver.from_scenario(_tiled(nx, ny), hw.make_params(limiter=limiter))
        dt = 0.5 * s.cfl_dt() if dt is None else dt
        i, j = np.meshgrid(np.arange(96), np.arange(64))
        nodes = (j * nx + i).ravel().astype(np.int32)
        values.append(A.hw_gauge_loss(s.h, [dt] * steps, nodes, np.ones((steps, nodes.size)))[1])
        s.close()
    for v in values[1:]:
        assert np.array_equal(v, values[0])
