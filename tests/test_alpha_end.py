"""The end of the one-launch exact pass of alpha (k_alpha2d_exact<true>, double grids above 2^18 nodes).

The last block to arrive clears the slots, the coarse maxima m32 among them, for the next launch. A block may
therefore arrive only after all of its warps have read m32, in a tile that it skips as in one that it evaluates:
otherwise a late warp finds zero thresholds, evaluates its nodes and leaves their keys in slots that the next launch
takes for zero, and a fallen maximum is reported at its former value.
"""
import os
import re

import numpy as np
import pytest

from conftest import ROOT
from paper_2208_01260_gb300 import scenarios as S


def test_every_warp_reads_the_thresholds_before_its_block_arrives():
    """On the source: on the way from the reads of m32 to the arrival there is a barrier outside every branch."""
    src = open(os.path.join(ROOT, "paper_2208_01260_gb300", "csrc", "hw_kernels2d.cu")).read()
    src = re.sub(r"//[^\n]*", "", src)
    body = src[src.index("k_alpha2d_exact("):]
    body = body[body.index("{") + 1:]
    reads = [m.start() for m in re.finditer(r"m32\[", body)][:2]
    end = body.index("alpha_block_done(")
    assert reads[-1] < end
    depth, barrier = 0, None
    for i, c in enumerate(body[:end]):
        depth += (c == "{") - (c == "}")
        if depth == 0 and re.match(r"[;}\s]__syncthreads\(\)", body[i:]):
            barrier = i
    assert barrier is not None and barrier > reads[-1]
    # the barrier's statement is no branch's own: what stands before it ends a statement or a block
    assert body[:barrier + 1].rstrip()[-1] in ";}"
    # and no return between it and the arrival
    assert "return" not in body[barrier:end]


@pytest.mark.gpu
def test_alpha_of_a_fallen_maximum():
    """600 x 451 nodes (above 2^18) at rest but one fast node, then without it, in turn: alpha and the step are the
    state's own every time. All tiles but the fast node's are skipped in the first state."""
    import paper_2208_01260_gb300 as hw
    nx, ny = 600, 451
    assert nx * ny > 1 << 18
    sc = S.hump2d(nx, ny, seed=75, bc=S.REFLECTIVE)
    s = hw.Solver.from_scenario(sc, hw.make_params())
    slow = s.state()
    for q in (1, 2):
        slow[q] = np.zeros_like(slow[q])
    fast = [p.copy() for p in slow]
    fast[1][300, 77] = 40.0
    fast[2][300, 77] = -60.0
    want = []
    for st in (fast, slow):
        t = hw.Solver.from_scenario(sc, hw.make_params())  # its first reduction: no earlier maximum
        t.set_state(st)
        want.append(t.alpha())
        t.close()
    h = slow[0] - sc.b
    c = np.sqrt(9.812 * h)
    assert abs(want[1][0] - c.max()) <= 1e-14 * c.max() and abs(want[1][1] - c.max()) <= 1e-14 * c.max()
    for _ in range(50):
        for st, w in ((fast, want[0]), (slow, want[1])):
            s.set_state(st)
            assert s.alpha() == w
            assert s.alpha() == w
    s.close()
