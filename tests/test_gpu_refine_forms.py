"""The refine's two forms in free-space FP32 IK of up to 4 segments: more than 32 * 4 * 152 candidates (conversions
and comparisons kept off the FP64 pipe) and fewer. Both round the same values in the same order, so a call on either
side of the line and its two halves below it agree bit for bit."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle as O
from gpu_util import orc_robot, targets_dev
from paper_2607_11340_gb300 import api, lib, synth

pytestmark = pytest.mark.gpu

LINE = 32 * 4 * 152


@pytest.mark.parametrize("n", [1, 2, 3, 4])
@pytest.mark.parametrize("K,extra", [(8, 0), (8, 1), (7, 1), (4, 33)])
def test_refine_forms_agree(n, K, extra):
    P = LINE // K + extra                                    # P * K <= LINE only for (8, 0): the last of the old form
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
