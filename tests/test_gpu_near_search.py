"""The search for near obstacles leaves out no pair within reach: every position of its words and chunks, and in
FP64, where it runs on an FP32 chain and table, also bends, sizes and spheres that FP32 cannot follow."""
import dataclasses

import numpy as np
import pytest
import torch

from gpu_util import targets_dev
from paper_2607_11340_gb300 import api, lib, synth

pytestmark = pytest.mark.gpu

B = 33                                                        # a warp and a lane


def _coll(spec, u, sph, w=synth.WEIGHTS, prims=None):
    """The clearance rows' cost of each state, from the kernel."""
    task = api.task_struct(lib.CR_TASK_IK6, targets_dev(np.tile([0.0, 0.0, 0.1, 1.0, 0.0, 0.0, 0.0], (B, 1))), 1, w)
    coll = api.cost_grad(api.robot_struct(spec), api.Scene(sph, prims=prims), task, u, grad=True, coll=True)[1]
    return coll.double().cpu().numpy()


def _samples(spec, u):
    return api.fk(api.robot_struct(spec), u, backbone=True)[1].double().cpu().numpy()  # [n nb][3][B]


def _near(rng, bb, n_o, spread, r_lo, r_hi):
    """n_o spheres about backbone samples."""
    c = bb[rng.integers(0, bb.shape[0], n_o), :, rng.integers(0, B, n_o)] + rng.normal(0, 1, (n_o, 3)) * spread
    return np.concatenate([c, rng.uniform(r_lo, r_hi, (n_o, 1))], axis=1)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("n,n_o", [(1, 1), (1, 31), (2, 32), (3, 33), (4, 63), (4, 64), (5, 65), (6, 97), (4, 130),
                                   (2, 256)])
def test_every_position_is_found(n, n_o, dtype):
    """The clearance cost among n_o spheres is the sum of the costs among each one alone; both add the same
    non-negative terms, at most n * n_b * n_o of them, so they agree to two roundings a term."""
    spec = dataclasses.replace(synth.ROBOT_FAMILY, L=synth.ROBOT_FAMILY.L[:n])
    rng = np.random.default_rng(100 * n + n_o)
    u = torch.as_tensor(synth.hexagon_states(rng, B, n, spec.umax).T.copy(), dtype=dtype, device="cuda")
    sph = _near(rng, _samples(spec, u), n_o, 0.004, 0.004, 0.01)
    alone = sum(_coll(spec, u, sph[j:j + 1]) for j in range(n_o))
    assert (alone > 0).any()
    err = np.abs(_coll(spec, u, sph) - alone)
    assert (err <= 2 * n * spec.nb * n_o * torch.finfo(dtype).eps * alone).all(), err.max()


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_largest_set_of_primitives(dtype):
    """256 primitives, the most a scene takes: with the FP32 table they fill the shared memory of a launch. The sum
    over its halves, as above."""
    n = 3
    spec = dataclasses.replace(synth.ROBOT_FAMILY, L=synth.ROBOT_FAMILY.L[:n])
    rng = np.random.default_rng(3)
    u = torch.as_tensor(synth.hexagon_states(rng, B, n, spec.umax).T.copy(), dtype=dtype, device="cuda")
    pr = synth.prims_uniform(rng, 128, 128, [-0.2, -0.2, 0.0], [0.2, 0.2, 0.35], 0.004, 0.01, 0.01, 0.04)
    assert len(pr) == 256
    parts = _coll(spec, u, None, prims=pr[:128]) + _coll(spec, u, None, prims=pr[128:])
    assert (parts > 0).any()
    err = np.abs(_coll(spec, u, None, prims=pr) - parts)
    assert (err <= 2 * n * spec.nb * 256 * torch.finfo(dtype).eps * parts).all(), err.max()


def _check_fp64(spec, u, sph, w, theta):
    """Against the distances of the samples that cr_fk gives. The two kernels round the bends (together at most
    theta) in their own order: 8 roundings of each shift a sample by at most pos, a row by rho_c viol pos."""
    bb = _samples(spec, u)
    d = np.sqrt(((bb[:, None] - sph[None, :, :3, None]) ** 2).sum(2))        # [samples][n_o][B]
    v = np.maximum(sph[None, :, 3, None] + spec.body_radius + w.delta - d, 0.0)
    ref = 0.5 * w.rho_c * (v * v).sum((0, 1))
    assert (ref > 0).sum() > B // 4
    size = sum(spec.L) + np.abs(sph).max()
    pos = 8 * 2.0 ** -53 * (theta + 16) * size
    err = np.abs(_coll(spec, u, sph, w) - ref)
    assert (err <= w.rho_c * (pos * v.sum((0, 1)) + v.size * pos * pos) + 1e-13 * ref).all(), (err / ref).max()


@pytest.mark.parametrize("n", [2, 4, 6])
@pytest.mark.parametrize("turns", [1.0, 10.0, 1e3, 1e6])
def test_fp64_bends(n, turns):
    """A first segment bent far beyond the curvature limit, as an unbounded optimiser's line search visits it: what
    follows lies where its last fraction of a turn points."""
    spec = dataclasses.replace(synth.ROBOT_FAMILY, L=synth.ROBOT_FAMILY.L[:n])
    rng = np.random.default_rng(n)
    u = synth.hexagon_states(rng, B, n, spec.umax)
    u[:, :3] *= turns
    u = torch.as_tensor(u.T.copy(), dtype=torch.float64, device="cuda")
    _check_fp64(spec, u, _near(rng, _samples(spec, u), 40, 0.004, 0.002, 0.006), synth.WEIGHTS,
                (turns + n) * 2.0 / spec.rc * spec.umax)


@pytest.mark.parametrize("scale", [1e-25, 1e-12, 1e12, 1e22])
def test_fp64_sizes(scale):
    """Robots and scenes in any unit of length."""
    f = synth.ROBOT_FAMILY
    spec = dataclasses.replace(f, L=tuple(scale * l for l in f.L[:3]), rc=scale * f.rc, umax=scale * f.umax)
    w = dataclasses.replace(synth.WEIGHTS, delta=0.0)
    rng = np.random.default_rng(5)
    u = torch.as_tensor(synth.hexagon_states(rng, B, 3, spec.umax).T.copy(), dtype=torch.float64, device="cuda")
    sph = _near(rng, _samples(spec, u), 40, 0.004 * scale, 0.002 * scale, 0.006 * scale)
    _check_fp64(spec, u, sph, w, 3 * 2.0 / f.rc * f.umax)


@pytest.mark.parametrize("far", [1e17, 3e18, 2e19, 1e30, 1e200])
def test_fp64_spheres(far):
    """A sphere as large as far and as far away has the robot inside it; small ones as far away are out of reach."""
    spec = dataclasses.replace(synth.ROBOT_FAMILY, L=synth.ROBOT_FAMILY.L[:3])
    rng = np.random.default_rng(6)
    u = torch.as_tensor(synth.hexagon_states(rng, B, 3, spec.umax).T.copy(), dtype=torch.float64, device="cuda")
    near = _near(rng, _samples(spec, u), 40, 0.004, 0.002, 0.006)
    away = np.array([[far, 0.0, 0.0, 0.01], [0.0, -far, far, 1.0]])
    theta = 3 * 2.0 / spec.rc * spec.umax
    alone = _coll(spec, u, near)
    assert (alone > 0).any() and np.array_equal(_coll(spec, u, np.concatenate([away, near])), alone)
    if far < 1e100:                                           # its square fits
        _check_fp64(spec, u, np.concatenate([near, [[far, 0.0, 0.0, 1.5 * far]]]), synth.WEIGHTS, theta)


@pytest.mark.parametrize("far", [2e19, 1e30])
def test_ik_inside_a_sphere(far):
    """The FP64 acceptance of the warp refine (each problem its own spheres, fewer than 8 candidates) finds a robot
    inside a sphere whose square FP32 does not hold."""
    spec = dataclasses.replace(synth.ROBOT_FAMILY, L=synth.ROBOT_FAMILY.L[:3])
    u = synth.hexagon_states(np.random.default_rng(7), B, 3, spec.umax)
    T = api.fk(api.robot_struct(spec), torch.as_tensor(u.T.copy(), device="cuda"))[0].cpu().numpy().T
    tg = targets_dev(synth.pose_targets(T, "pose"))
    ik = dataclasses.replace(synth.IK_GOAL, n_final=4)

    def success(row):
        s = api.IkSolver(spec, ik, synth.WEIGHTS, lib.CR_TASK_IK6, B, api.Scene(np.tile(row, (B, 1, 1)), per_problem=True))
        return s.solve(tg).success.cpu().numpy()

    assert (success([[far, 0.0, 0.0, 0.01]]) != 0).sum() > B // 2
    assert (success([[far, 0.0, 0.0, 1.5 * far]]) == 0).all()
