"""The ragged batch's joint phase in its two forms: a warp to a path item (more than 304 path items of a segment
count) and a block to an item (fewer). Both add in the same order, so the whole batch and its parts agree bit for
bit, at waypoint counts around the rounds of 32 and at the ends of the range."""
import numpy as np
import pytest
import torch

import oracle as O
from gpu_util import orc_robot
from paper_2607_11340_gb300 import api, synth
import dataclasses

pytestmark = pytest.mark.gpu

HS = [2, 31, 32, 33, 64, 65, 127, 128]


def _fk_backbone(n, U):
    spec = dataclasses.replace(synth.ROBOT_FAMILY, L=synth.ROBOT_FAMILY.L[:n])
    return O.fk(orc_robot(spec), U, backbone=True)


@pytest.mark.parametrize("n", [1, 2])
def test_block_and_warp_forms_agree(n):
    N = 310
    items = np.array([[1, n, 2 if i >= 3 * len(HS) else HS[i % len(HS)], 16, 4 * (i % 3)] for i in range(N)])
    items, tg, sph, _ = synth.ragged_workload(N, _fk_backbone, seed=5, items=items)
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

    whole, a, c = solve(0, N), solve(0, 150), solve(150, N)
    for f in ("u", "cost", "pos", "rot", "flags"):
        assert torch.equal(getattr(whole, f), torch.cat([getattr(a, f), getattr(c, f)])), f
