"""The ragged batch's joint phase at 3 to 6 segments: a block to a path item (up to two per SM) against a warp to an
item (more), which add in the same order."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle as O
from gpu_util import orc_robot
from paper_2607_11340_gb300 import api, synth

pytestmark = pytest.mark.gpu

HS = [2, 31, 32, 33, 64, 65, 127, 128]


def _fk_backbone(n, U):
    spec = dataclasses.replace(synth.ROBOT_FAMILY, L=synth.ROBOT_FAMILY.L[:n])
    return O.fk(orc_robot(spec), U, backbone=True)


@pytest.mark.parametrize("n", [3, 4, 5, 6])
def test_block_and_warp_forms_agree(n):
    N = 2 * torch.cuda.get_device_properties(0).multi_processor_count + 6
    items = np.array([[1, n, 2 if i >= 2 * len(HS) else HS[i % len(HS)], 16, 4 * (i % 3)] for i in range(N)])
    items, tg, sph, _ = synth.ragged_workload(N, _fk_backbone, seed=n, items=items)
    ik = dataclasses.replace(synth.IK_RAGGED, k_init=8, k_final=6, n_final=4)

    def solve(lo, hi):
        b = api.BatchSolver(synth.ROBOT_FAMILY, items[lo:hi], ik, synth.WEIGHTS, k_warm=4, k_joint=6, seeds_per_unit=32,
                            seed_regs=1, p0=lo)
        w = items[:, 2].cumsum()
        s = items[:, 4].cumsum()
        b.set_inputs(tg[w[lo] - items[lo, 2]:w[hi - 1]], sph[s[lo] - items[lo, 4]:s[hi - 1]])
        b.run()
        torch.cuda.synchronize()
        return b

    whole, a, c = solve(0, N), solve(0, N // 2), solve(N // 2, N)
    for f in ("u", "cost", "pos", "rot", "flags"):
        assert torch.equal(getattr(whole, f), torch.cat([getattr(a, f), getattr(c, f)])), f
