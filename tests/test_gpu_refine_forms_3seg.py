"""The refine's two forms in free-space FP32 IK of 3 segments, whose line is 48 * 4 * 152 candidates: a call on either
side of it and its two halves below it agree bit for bit."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle as O
from gpu_util import orc_robot, targets_dev
from paper_2607_11340_gb300 import api, lib, synth

pytestmark = pytest.mark.gpu

LINE = 48 * 4 * 152


@pytest.mark.parametrize("K,extra", [(8, 0), (8, 1), (7, 1), (4, 33)])
def test_refine_forms_agree(K, extra):
    n = 3
    P = LINE // K + extra                                    # (8, 0) is the last on its side
    spec = dataclasses.replace(synth.ROBOT_FAMILY, L=synth.ROBOT_FAMILY.L[:n])
    ik = dataclasses.replace(synth.IK_3SEG, S=16, n_final=K, k_init=6, k_final=12)
    rb = orc_robot(spec)
    tg64, _ = synth.ik_workload(spec, 64, "pose", lambda x: O.fk(rb, x)[0], seed=n)
    tg = np.tile(tg64, (P // 64 + 1, 1))[:P]                 # seeds differ by index: every row is its own problem
    tg[5, 0] = 4.0                                           # out of reach: the damping grows until it stops

    def solve(lo, hi):
        s = api.IkSolver(spec, ik, synth.WEIGHTS, lib.CR_TASK_IK6, hi - lo, None, lib.CR_F32)
        o = s.solve(targets_dev(tg[lo:hi]), p0=lo)
        torch.cuda.synchronize()
        return o

    whole, a, c = solve(0, P), solve(0, P // 2), solve(P // 2, P)
    for f in ("u", "cost", "pos_err", "rot_err", "success"):
        assert torch.equal(getattr(whole, f), torch.cat([getattr(a, f), getattr(c, f)], -1)), f
