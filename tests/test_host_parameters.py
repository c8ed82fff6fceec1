"""Forms in which a caller may hand over the robot's lengths and radii, on the host (no GPU): everything that indexes
to one number per segment."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2607_11340_gb300 import api, lib, synth

L = [0.12, 0.10, 0.08]


@pytest.mark.parametrize("form", [tuple, list, np.array, torch.tensor,
                                  lambda v: [torch.tensor(x, dtype=torch.float64) for x in v],
                                  lambda v: torch.tensor(v, dtype=torch.float64)[:, None]])
def test_robot_lengths(form):
    spec = synth.RobotSpec(L=form(L), rc=0.005, umax=0.01, lmin=0.05, lmax=0.2)
    r = api.robot_struct(spec)
    np.testing.assert_allclose(r.L[:3], L, rtol=1e-7)
    assert list(r.L[3:]) == [0.0] * (lib.CR_MAX_SEG - 3) and list(r.r_c[:3]) == [0.005] * 3
    assert list(r.l_max[:3]) == [0.2] * 3


@pytest.mark.parametrize("form", [lambda v: v, lambda v: v[:, None], lambda v: v.float(), lambda v: torch.cat([v, v]),
                                  lambda v: v.numpy()])
def test_cost_parameters(form, monkeypatch):
    seen = []
    monkeypatch.setattr(lib, "cr_cost_grad", lambda robot, *a: seen.append(robot))
    spec = synth.RobotSpec(L=tuple(L), rc=0.005, umax=0.01)
    v = form(torch.tensor(L, dtype=torch.float64))
    api.IkCost.apply(torch.zeros(9, 4), v, 0.05 * v, (spec, dataclasses.make_dataclass("S", ["c"])(None), None))
    np.testing.assert_allclose(seen[0].L[:3], L, rtol=1e-7)
    np.testing.assert_allclose(seen[0].r_c[:3], [0.05 * x for x in L], rtol=1e-7)


@pytest.mark.parametrize("v", [torch.ones(2), torch.ones(3, 2), torch.ones(())])
def test_too_few_or_too_many(v, monkeypatch):
    monkeypatch.setattr(lib, "cr_cost_grad", lambda robot, *a: None)
    spec = synth.RobotSpec(L=tuple(L), rc=0.005, umax=0.01)
    with pytest.raises((IndexError, TypeError, ValueError, RuntimeError)):
        api.IkCost.apply(torch.zeros(9, 4), v, v, (spec, dataclasses.make_dataclass("S", ["c"])(None), None))
