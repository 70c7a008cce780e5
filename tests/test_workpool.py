"""The memory an adjoint call keeps for the next one (csrc/hw_workpool.h), compiled for the host against a memory of fixed
size: a call never fails, nor gets less, for what an earlier call or another solver has left."""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2208_01260_gb300", "csrc")


def test_pool_rules(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "check")
    subprocess.run([cxx, "-O1", "-g", "-std=c++17", "-Wall", "-Werror", "-I" + CSRC, os.path.join(HERE, "workpool_check.cpp"), "-o", exe],
                   check=True)
    r = subprocess.run([exe], capture_output=True, text=True, check=True)
    assert r.stdout.strip() == "0", r.stderr


@pytest.mark.gpu
def test_modes_in_turn():
    """Tape, snapshots and the loss alone in turn on one solver, with a second solver's calls between: each gives what a
    fresh solver gives."""
    import torch

    import paper_2208_01260_gb300 as hw
    from paper_2208_01260_gb300 import adjoint as A
    from paper_2208_01260_gb300 import scenarios as S
    sc = S.hump2d(70, 52, seed=83, bc=S.REFLECTIVE)
    idx, steps = np.array([5, 900, 2222], dtype=np.int32), 6
    obs = np.ones((steps, 3))

    def run(s, dt, snapshots):
        gs = [torch.empty(52, 70, dtype=torch.float64, device="cuda") for _ in range(9)]
        gt = [torch.empty(52, 70, dtype=torch.float64, device="cuda") for _ in range(3)]
        loss = A.hw_adjoint_run(s.h, [dt] * steps, idx, obs, snapshots, gs, gt)
        return loss[0] if isinstance(loss, tuple) else loss

    s, t = hw.Solver.from_scenario(sc), hw.Solver.from_scenario(sc)
    dt = 0.9 * s.cfl_dt()
    losses = []
    for mode in (A.HW_ADJ_TAPE, 2, 5, A.HW_ADJ_AUTO, 0, A.HW_ADJ_TAPE):
        for x in (s, t):
            losses.append(run(x, dt, mode))
            losses.append(A.hw_gauge_loss(x.h, [dt] * steps, idx, obs))
    assert len({float(x[0] if isinstance(x, tuple) else x) for x in losses}) == 1, losses
    s.close()
    t.close()
