"""What a user of the solver library has it do, as measurable cases: kinematics queries, cost
gradients behind autograd, calibration, roadmaps and the whole solvers, from one state per control
tick to batches that fill the GPU. Robots, settings and sizes are those of the package's own
workloads (`synth`) or spread around them.

`prepare` makes what a program holds before the call (inputs, scene, solver objects with their
workspaces), `run` is one call, `exact` the same result from plain 64-bit torch for the pieces that
have a closed form (kinematics, costs and their gradients, the calibration's optimum). The iterative
solvers have no such value: their result is the iterate that the method reaches.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2607_11340_gb300 import api, lib, synth

DEV = "cuda"
W = synth.WEIGHTS
LENGTHS = {1: (0.10,), 2: (0.12, 0.10), 3: (0.12, 0.10, 0.08), 4: (0.10,) * 4, 5: (0.10,) * 5, 6: (0.10,) * 6}


def listed():
    return [
        # a controller asks for the tip pose and Jacobian of the one state it is in, every tick
        dict(name="control tick", kind="kinematics", n=3, B=1, bits=32, backbone=False),
        # workspace sampling / learning data: poses, backbones and Jacobians of many states at once
        dict(name="workspace sampling", kind="kinematics", n=4, B=200003, bits=32, backbone=True),
        # gradients of the pose cost for states and for the robot's lengths and radii (a training step
        # of a policy or of the robot's parameters), free space
        dict(name="pose gradients", kind="gradient", n=3, B=262144, S=256, n_o=0, bits=32),
        # the same among obstacles, an odd number of states
        dict(name="obstacle gradients", kind="gradient", n=4, B=60001, S=1, n_o=32, bits=32),
        # double precision, as for fits and gradient checks
        dict(name="double gradients", kind="gradient", n=3, B=5000, S=4, n_o=12, bits=64),
        # one gradient step of a user's own trajectory optimiser: 256 problems of 32 states, each with
        # its own 64 spheres
        dict(name="trajectory gradients", kind="trajectory", n=3, P=256, T=32, n_o=64, bits=32),
        # a kinematic calibration from logged measurements, double precision
        dict(name="calibration", kind="calibration", n=3, K=1024, bits=64),
        # new scenes: one roadmap for each, then a query on each
        dict(name="roadmaps", kind="roadmap", n=3, R=256, N=256, k=8, n_o=64, T=32),
        # the largest everyday call: beam-search IK for thousands of poses
        dict(name="batched ik", kind="ik", n=3, P=4096, S=256, k_init=64, n_final=8, n_o=0),
        # trajectory planning to pose goals among obstacles (goal IK, initialisation, refinement)
        dict(name="trajectory planning", kind="plan", n=3, P=256, T=32, n_o=64),
        # path following: waypoint sweep and joint refinement among obstacles
        dict(name="path following", kind="path", n=4, P=512, H=64, n_o=32),
        # a server's mixed batch of IK and path requests of all sizes
        dict(name="mixed requests", kind="batch", N=192, mix=7),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["kinematics", "gradient", "trajectory", "calibration", "roadmap", "ik", "plan", "path", "batch"])
    if kind == "kinematics":
        return dict(kind=kind, n=rng.randint(1, 6), B=_log(rng, 1, 150000), bits=rng.choice([32, 32, 64]),
                    backbone=rng.random() < 0.5)
    if kind == "gradient":
        bits = rng.choice([32, 32, 64])
        return dict(kind=kind, n=rng.randint(1, 6), B=_log(rng, 16, 250000 if bits == 32 else 10000),
                    S=rng.choice([1, 4, 32, 256]), n_o=rng.choice([0, 0, 1, 12, 32, 64, 100]), bits=bits)
    if kind == "trajectory":
        bits = rng.choice([32, 32, 64])
        return dict(kind=kind, n=rng.randint(2, 5), P=_log(rng, 1, 700 if bits == 32 else 60), T=rng.randint(3, 64),
                    n_o=rng.choice([0, 8, 33, 64]), bits=bits)
    if kind == "calibration":
        return dict(kind=kind, n=rng.randint(2, 4), K=_log(rng, 64, 20000), bits=64)
    if kind == "roadmap":
        N = _log(rng, 50, 400)
        return dict(kind=kind, n=rng.randint(2, 4), R=_log(rng, 1, 200), N=N, k=rng.randint(4, 12),
                    n_o=rng.choice([0, 8, 33, 64]), T=rng.randint(8, 64))
    if kind == "ik":
        return dict(kind=kind, n=rng.randint(2, 4), P=_log(rng, 1, 1500), S=rng.choice([32, 64, 100, 256]),
                    k_init=rng.choice([16, 32, 64]), n_final=rng.choice([4, 8]), n_o=rng.choice([0, 0, 8, 32]))
    if kind == "plan":
        return dict(kind=kind, n=rng.randint(2, 4), P=_log(rng, 1, 200), T=rng.randint(8, 48),
                    n_o=rng.choice([0, 16, 64]))
    if kind == "path":
        return dict(kind=kind, n=rng.randint(2, 5), P=_log(rng, 1, 300), H=rng.randint(2, 64), n_o=rng.choice([0, 16, 32]))
    return dict(kind="batch", N=_log(rng, 16, 180), mix=rng.randint(0, 1 << 20))


# --------------------------------------------------------------------------------------------------
# The kinematics and cost in plain 64-bit torch (targets and scenes of the inputs; the exact values)
# --------------------------------------------------------------------------------------------------
def _spec(n):
    return synth.RobotSpec(L=LENGTHS[n], rc=0.005, umax=0.010)



def _chain(u, L, rc):
    """u [B, n, 3]; L, rc [n]. Base frames (R, p) of every segment, bends, tip frame."""
    B, n, _ = u.shape
    R = torch.eye(3, dtype=u.dtype, device=u.device).expand(B, 3, 3)
    p = torch.zeros(B, 3, dtype=u.dtype, device=u.device)
    segs = []
    for i in range(n):
        K = -2.0 / (3.0 * rc[i])
        ax = K * (u[:, i, 0] - 0.5 * (u[:, i, 1] + u[:, i, 2]))
        ay = K * (math.sqrt(0.75) * (u[:, i, 1] - u[:, i, 2]))
        segs.append((R, p, ax, ay, L[i]))
        q, Ri = _arc(ax, ay, L[i])
        p = p + (R @ q.unsqueeze(-1)).squeeze(-1)
        R = R @ Ri
    return segs, R, p


def _arc(ax, ay, L):
    """End point and rotation of a constant-curvature arc of length L that bends by (ax, ay)."""
    t = torch.sqrt(ax * ax + ay * ay + 1e-300)
    s = torch.sin(t) / t
    c = 0.5 * (torch.sin(0.5 * t) / (0.5 * t)) ** 2
    q = torch.stack([L * c * ax, L * c * ay, L * s], -1)
    R = torch.stack([1 - c * ax * ax, -c * ax * ay, s * ax, -c * ax * ay, 1 - c * ay * ay, s * ay,
                     -s * ax, -s * ay, 1 - c * (ax * ax + ay * ay)], -1).reshape(-1, 3, 3)
    return q, R


def _points(segs, nb):
    """Backbone samples [B, n, nb, 3]: the ends of the sub-arcs of fractions k / nb."""
    out = []
    for R, p, ax, ay, L in segs:
        for k in range(1, nb + 1):
            f = k / nb
            q, _ = _arc(f * ax, f * ay, f * L)
            out.append(p + (R @ q.unsqueeze(-1)).squeeze(-1))
    return torch.stack(out, 1).reshape(out[0].shape[0], len(segs), nb, 3)


def _quat(R):
    """Rotations [B, 3, 3] to unit quaternions (w, x, y, z), largest component first found."""
    t = R[:, 0, 0] + R[:, 1, 1] + R[:, 2, 2]
    cand = torch.stack([t, R[:, 0, 0], R[:, 1, 1], R[:, 2, 2]], 1)
    k = cand.argmax(1)
    a, b, c = R[:, 2, 1], R[:, 0, 2], R[:, 1, 0]
    d, e, f = R[:, 1, 2], R[:, 2, 0], R[:, 0, 1]
    q0 = torch.stack([1 + t, a - d, b - e, c - f], 1)
    q1 = torch.stack([a - d, 1 + 2 * R[:, 0, 0] - t, f + c, b + e], 1)
    q2 = torch.stack([b - e, f + c, 1 + 2 * R[:, 1, 1] - t, a + d], 1)
    q3 = torch.stack([c - f, b + e, a + d, 1 + 2 * R[:, 2, 2] - t], 1)
    q = torch.stack([q0, q1, q2, q3], 1)[torch.arange(len(k), device=R.device), k]
    return q / q.norm(dim=1, keepdim=True)


def _rot_of(q):
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).reshape(-1, 3, 3)


def _log3(E):
    v = 0.5 * torch.stack([E[:, 2, 1] - E[:, 1, 2], E[:, 0, 2] - E[:, 2, 0], E[:, 1, 0] - E[:, 0, 1]], 1)
    cs = 0.5 * (E[:, 0, 0] + E[:, 1, 1] + E[:, 2, 2] - 1)
    s2 = (v * v).sum(1)
    sn = torch.sqrt(s2 + 1e-300)
    f = torch.where(s2 < 1e-12, 1 + s2 / 6, torch.atan2(sn, cs) / sn)
    return f.unsqueeze(1) * v


def _pose_cost(R, p, tg):
    """tg [B, 7]."""
    r = W.wp * (p - tg[:, :3])
    e = W.wR * _log3(_rot_of(tg[:, 3:]).transpose(1, 2) @ R)
    return 0.5 * (r * r).sum(1) + 0.5 * (e * e).sum(1)


def _state_cost(u, segs, spec, sph):
    """Penalty rows of the states u [B, n, 3]; sph [S, 4] shared or [B, S, 4], or None."""
    F = 0.5 * W.rho_eq * (u.sum(2) ** 2).sum(1)
    F = F + 0.5 * W.rho_b * (torch.relu(u.abs() - spec.umax) ** 2).sum((1, 2))
    for _, _, ax, ay, _ in segs:
        F = F + 0.5 * W.rho_k * torch.relu(torch.sqrt(ax * ax + ay * ay + 1e-300) - spec.thmax) ** 2
    if sph is not None and sph.shape[-2]:
        x = _points(segs, spec.nb)
        reach = sph[..., 3] + spec.body_radius + W.delta
        for j in range(sph.shape[-2]):
            c = sph[..., j, :3].reshape(-1, 1, 1, 3)
            d = torch.sqrt(((x - c) ** 2).sum(-1))
            v = torch.relu(reach[..., j].reshape(-1, 1, 1) - d)
            F = F + 0.5 * W.rho_c * (v * v).sum((1, 2))
    return F


# --------------------------------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 2654435761 % (1 << 62))


def _rand(g, *shape):
    return torch.rand(*shape, dtype=torch.float64, device=DEV, generator=g)


def _hexagon(g, count, n, umax):
    """In-bound states [count, n, 3], uniform on each segment's hexagon."""
    a = (2 * _rand(g, count, n, 8, 2) - 1) * umax
    ok = a.sum(-1).abs() <= umax
    ok[..., 7] = True
    a[:, :, 7] *= 0.5
    first = ok.to(torch.uint8).argmax(2)
    a = torch.gather(a, 2, first[..., None, None].expand(-1, -1, 1, 2)).squeeze(2)
    return torch.cat([a, -a.sum(2, keepdim=True)], 2)


def _bezier(g, P, H, n, umax):
    """[P, H, n, 3]: smooth curves in state space through four in-bound states."""
    c = _hexagon(g, 4 * P, n, umax).reshape(P, 4, n, 3)
    s = torch.linspace(0, 1, H, dtype=torch.float64, device=DEV)
    w = torch.stack([(1 - s) ** 3, 3 * s * (1 - s) ** 2, 3 * s * s * (1 - s), s ** 3], 1)
    return torch.einsum("hk,pknj->phnj", w, c)


def _robot_rows(spec):
    L = torch.tensor(spec.L, dtype=torch.float64, device=DEV)
    return L, torch.full_like(L, spec.rc)


def _fk(spec, u):
    segs, R, p = _chain(u, *_robot_rows(spec))
    return segs, R, p


def _poses(spec, u):
    _, R, p = _fk(spec, u)
    return torch.cat([p, _quat(R)], 1)


def _spheres(g, pts, count, margin, clearance, r_lo=0.005, r_hi=0.015):
    """[P, count, 4] spheres uniform in the dilated bounding box of pts [P, M, 3], none closer than
    `clearance` to a point of its problem."""
    P = pts.shape[0]
    lo, hi = pts.amin(1) - margin, pts.amax(1) + margin
    m = 8 * count + 16
    c = lo[:, None] + _rand(g, P, m, 3) * (hi - lo)[:, None]
    r = r_lo + (r_hi - r_lo) * _rand(g, P, m)
    d = torch.empty(P, m, dtype=torch.float64, device=DEV)
    step = max(1, (1 << 26) // (m * pts.shape[1]))
    for i in range(0, P, step):
        d[i:i + step] = torch.cdist(c[i:i + step], pts[i:i + step],
                                    compute_mode="donot_use_mm_for_euclid_dist").amin(2)
    bad = d < r + clearance
    order = torch.argsort(bad.to(torch.uint8), dim=1, stable=True)[:, :count]
    c = torch.where(bad[..., None], c + 1.0, c)  # what did not fit anywhere stands out of reach
    return torch.cat([torch.gather(c, 1, order[..., None].expand(-1, -1, 3)), torch.gather(r, 1, order)[..., None]], 2)


def _clear(spec):
    return spec.body_radius + W.delta


def _soa(x, dtype=torch.float64):
    """[B, ...] to [components, B]."""
    return x.reshape(x.shape[0], -1).T.contiguous().to(dtype)


def _type(case):
    return torch.float32 if case["bits"] == 32 else torch.float64


def _kin_inputs(case, seed):
    spec = _spec(case["n"])
    return spec, _hexagon(_gen(seed), case["B"], case["n"], spec.umax).to(_type(case))


def _gradient_inputs(case, seed):
    """States around those of their targets (a descent under way), an upstream gradient, a scene that
    they touch here and there, and robot parameters a little off the nominal ones."""
    g, spec, dt = _gen(seed), _spec(case["n"]), _type(case)
    B, n = case["B"], case["n"]
    P = -(-B // case["S"])
    ut = _hexagon(g, P, n, spec.umax)
    tg = _poses(spec, ut)
    u = ut.repeat_interleave(case["S"], 0)[:B] * 0.9 + 0.1 * _hexagon(g, B, n, spec.umax)
    u = (u + 2e-4 * (2 * _rand(g, B, n, 3) - 1)).to(dt)
    up = (0.5 + _rand(g, B)).to(dt)
    sph = None
    if case["n_o"]:
        segs, _, _ = _fk(spec, _hexagon(g, 64, n, spec.umax))
        x = _points(segs, spec.nb).reshape(1, -1, 3)
        sph = _spheres(g, x, case["n_o"], 0.03, 0.0)[0]
    L, rc = _robot_rows(spec)
    L, rc = (v.cpu() * (1 + 0.02 * (2 * _rand(g, n).cpu() - 1)) for v in (L, rc))
    return spec, u, up, tg, sph, L.to(dt), rc.to(dt)


def _trajectory_inputs(case, seed):
    g, spec, dt = _gen(seed), _spec(case["n"]), _type(case)
    P, T, n = case["P"], case["T"], case["n"]
    us, ug = _hexagon(g, P, n, spec.umax), _hexagon(g, P, n, spec.umax)
    goal = _poses(spec, ug)
    sph = None
    if case["n_o"]:
        segs, _, _ = _fk(spec, torch.cat([us, ug]))
        x = _points(segs, spec.nb).reshape(2, P, -1, 3)
        sph = _spheres(g, torch.cat([x[0], x[1]], 1), case["n_o"], 0.03, _clear(spec))
    f = (torch.arange(1, T, dtype=torch.float64, device=DEV) / (T - 1))[None, :, None, None]
    x = us[:, None] + f * (ug - us)[:, None]
    x = (x + 3e-4 * (2 * _rand(g, P, T - 1, n, 3) - 1)).reshape(P * (T - 1), n, 3).to(dt)
    up = (0.5 + _rand(g, P)).to(dt)
    return spec, us, goal, sph, x, up


def _calibration_inputs(case, seed):
    g, spec = _gen(seed), _spec(case["n"])
    U = _hexagon(g, case["K"], case["n"], spec.umax).to(_type(case))
    L, rc = _robot_rows(spec)
    nominal = torch.cat([L, rc])
    true = nominal * (1 + synth.PERTURB_CALIB * (2 * _rand(g, len(nominal)) - 1))
    _, _, p = _chain(U.double(), true[:case["n"]], true[case["n"]:])
    noise = torch.randn(p.shape, dtype=torch.float64, device=DEV, generator=g)
    return spec, U, p + synth.SIGMA_CALIB * noise, nominal


# --------------------------------------------------------------------------------------------------
# States and passes
# --------------------------------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    s = dict(kind=kind)
    if kind == "kinematics":
        spec, u = _kin_inputs(case, seed)
        s.update(robot=api.robot_struct(spec), u=_soa(u, u.dtype), backbone=case["backbone"])
    elif kind == "gradient":
        spec, u, up, tg, sph, L, rc = _gradient_inputs(case, seed)
        kept = api.Scene(sph) if sph is not None else api.Scene(None)
        task = api.task_struct(lib.CR_TASK_IK6, _soa(tg), case["S"], W)
        s.update(u=_soa(u, u.dtype).requires_grad_(), up=up, L=L.requires_grad_(), rc=rc.requires_grad_(),
                 ctx=(spec, kept, task))
    elif kind == "trajectory":
        spec, us, goal, sph, x, up = _trajectory_inputs(case, seed)
        kept = api.Scene(sph, per_problem=True) if sph is not None else api.Scene(None)
        task = api.traj_task_struct(_soa(us), _soa(goal), case["T"], W)
        s.update(x=_soa(x, x.dtype).requires_grad_(), up=up, ctx=(api.robot_struct(spec), kept, task))
    elif kind == "calibration":
        spec, U, p, nominal = _calibration_inputs(case, seed)
        s.update(spec=spec, U=_soa(U, U.dtype), p=_soa(p), nominal=nominal)
    elif kind == "roadmap":
        g, spec = _gen(seed), _spec(case["n"])
        R = case["R"]
        us, ug = _hexagon(g, R, case["n"], spec.umax), _hexagon(g, R, case["n"], spec.umax)
        kept = api.Scene(None)
        if case["n_o"]:
            segs, _, _ = _fk(spec, torch.cat([us, ug]))
            x = _points(segs, spec.nb).reshape(2, R, -1, 3)
            kept = api.Scene(_spheres(g, torch.cat([x[0], x[1]], 1), case["n_o"], 0.03, _clear(spec)), per_problem=True)
        prm = synth.PrmSpec(N=case["N"], k=case["k"], seed=int(seed) & 0x7fffffff)
        m = api.Roadmap(spec, prm, R)
        for t in (m.nodes, m.node_ok, m.nbr, m.row, m.col, m.wt):
            t.zero_()
        s.update(map=m, scene=kept, us=_soa(us), ug=_soa(ug), T=case["T"])
    elif kind == "ik":
        g, spec = _gen(seed), _spec(case["n"])
        ut = _hexagon(g, case["P"], case["n"], spec.umax)
        kept = api.Scene(None)
        if case["n_o"]:
            segs, _, _ = _fk(spec, ut[:256])
            x = _points(segs, spec.nb).reshape(1, -1, 3)
            kept = api.Scene(_spheres(g, x, case["n_o"], 0.03, 0.0)[0])
        ik = synth.IkSpec(S=case["S"], n_final=case["n_final"], k_init=case["k_init"], k_final=30, seed=int(seed) & 0xffff)
        s.update(solver=api.IkSolver(spec, ik, W, lib.CR_TASK_IK6, case["P"], kept), targets=_soa(_poses(spec, ut)))
    elif kind == "plan":
        g, spec = _gen(seed), _spec(case["n"])
        P = case["P"]
        us, ug = _hexagon(g, P, case["n"], spec.umax), _hexagon(g, P, case["n"], spec.umax)
        kept = api.Scene(None)
        if case["n_o"]:
            segs, _, _ = _fk(spec, torch.cat([us, ug]))
            x = _points(segs, spec.nb).reshape(2, P, -1, 3)
            kept = api.Scene(_spheres(g, torch.cat([x[0], x[1]], 1), case["n_o"], 0.03, _clear(spec)), per_problem=True)
        s.update(solver=api.TrajSolver(spec, synth.IK_GOAL, W, P, case["T"], kept), us=_soa(us), goal=_soa(_poses(spec, ug)))
    elif kind == "path":
        g, spec = _gen(seed), _spec(case["n"])
        P, H = case["P"], case["H"]
        u = _bezier(g, P, H, case["n"], spec.umax).reshape(P * H, case["n"], 3)
        kept = api.Scene(None)
        if case["n_o"]:
            segs, _, _ = _fk(spec, u)
            x = _points(segs, spec.nb).reshape(P, -1, 3)
            kept = api.Scene(_spheres(g, x, case["n_o"], 0.02, _clear(spec)), per_problem=True)
        s.update(solver=api.PathSolver(spec, synth.IK_PATH0, W, P, H, kept), wp=_soa(_poses(spec, u)))
    else:
        g = _gen(seed)
        items = synth.ragged_items(np.random.default_rng(case["mix"]), case["N"])
        targets, spheres = [], []
        for _, n, H, _, no in items.tolist():
            spec = _family(n)
            u = _bezier(g, 1, H, n, spec.umax)[0] if H > 1 else _hexagon(g, 1, n, spec.umax)
            segs, R, p = _fk(spec, u)
            targets.append(torch.cat([p, _quat(R)], 1))
            if no:
                spheres.append(_spheres(g, _points(segs, spec.nb).reshape(1, -1, 3), no, 0.02, _clear(spec))[0])
        # a server that has settled its plan's two choices
        b = api.BatchSolver(synth.ROBOT_FAMILY, items, synth.IK_RAGGED, W, seeds_per_unit=32, seed_regs=1)
        b.set_inputs(torch.cat(targets), torch.cat(spheres) if spheres else None)
        for t in (b.u, b.cost, b.pos, b.rot, b.flags):
            t.zero_()
        b.plan()
        s.update(solver=b)
    return s


def _family(n):
    f = synth.ROBOT_FAMILY
    return synth.RobotSpec(L=f.L[:n], rc=f.rc, umax=f.umax, nb=f.nb)


def run(s):
    kind = s["kind"]
    if kind == "kinematics":
        T, bb = api.fk(s["robot"], s["u"], s["backbone"])
        return dict(T=T, backbone=bb, J=api.fk_jac(s["robot"], s["u"]))
    if kind == "gradient":
        F = api.IkCost.apply(s["u"], s["L"], s["rc"], s["ctx"])
        gu, gL, gr = torch.autograd.grad(F, (s["u"], s["L"], s["rc"]), s["up"])
        return dict(cost=F.detach(), u=gu, L=gL, rc=gr)
    if kind == "trajectory":
        F = api.TrajCost.apply(s["x"], s["ctx"])
        (gx,) = torch.autograd.grad(F, (s["x"],), s["up"])
        return dict(cost=F.detach(), x=gx)
    if kind == "calibration":
        theta, F, _ = api.calibrate(s["spec"], s["U"], s["p"], s["nominal"])
        return dict(theta=theta, F=F)
    if kind == "roadmap":
        m = s["map"].build(s["scene"], W)
        X, length, hops = m.query(s["scene"], W, s["us"], s["ug"], s["T"])
        return dict(nodes=m.nodes, ok=m.node_ok, nbr=m.nbr, row=m.row, col=m.col, wt=m.wt, X=X, length=length, hops=hops)
    if kind == "ik":
        r = s["solver"].solve(s["targets"])
        return dict(u=r.u, cost=r.cost, pos=r.pos_err, rot=r.rot_err, success=r.success)
    if kind == "plan":
        r = s["solver"].solve(s["us"], s["goal"])
        return dict(X=r.X, cost=r.cost, pos=r.goal_pos, rot=r.goal_rot, speed=r.speed, accel=r.accel, lim=r.lim_ok, col=r.col_ok)
    if kind == "path":
        r = s["solver"].solve(s["wp"])
        return dict(X=r.X, cost=r.cost, pos=r.pos, rot=r.rot, lim=r.lim_ok, col=r.col_ok)
    r = s["solver"].run()
    return dict(u=r.u, cost=r.cost, pos=r.pos, rot=r.rot, flags=r.flags)


def exact(case, seed):
    kind = case["kind"]
    if kind == "kinematics":
        spec, u = _kin_inputs(case, seed)
        u = u.double().requires_grad_()
        segs, R, p = _chain(u, *_robot_rows(spec))
        Rd = R.detach()
        # d(rotation) R^T is skew: its three entries are the world angular velocity
        turn = [(R[:, 2] * Rd[:, 1]).sum(), (R[:, 0] * Rd[:, 2]).sum(), (R[:, 1] * Rd[:, 0]).sum()]
        rows = [torch.autograd.grad(f, u, retain_graph=True)[0] for f in [p[:, a].sum() for a in range(3)] + turn]
        with torch.no_grad():
            J = torch.stack([_soa(r) for r in rows])
            T = torch.cat([_soa(R), _soa(p)])
            bb = None
            if case["backbone"]:
                x = _points(segs, spec.nb)
                bb = x.reshape(x.shape[0], -1, 3).permute(1, 2, 0).contiguous()
        return dict(T=T, backbone=bb, J=J)
    if kind == "gradient":
        spec, u, up, tg, sph, L, rc = _gradient_inputs(case, seed)
        u, L, rc = u.double().requires_grad_(), L.double().to(DEV).requires_grad_(), rc.double().to(DEV).requires_grad_()
        tg = tg.repeat_interleave(case["S"], 0)[:case["B"]]
        costs, gu, gL, gr = [], [], 0, 0
        for i in range(0, case["B"], 8192):
            ui = u[i:i + 8192]
            segs, R, p = _chain(ui, L, rc)
            F = _state_cost(ui, segs, spec, sph) + _pose_cost(R, p, tg[i:i + 8192])
            g = torch.autograd.grad(F, (ui, L, rc), up[i:i + 8192].double())
            costs.append(F.detach())
            gu.append(g[0])
            gL, gr = gL + g[1], gr + g[2]
        return dict(cost=torch.cat(costs), u=_soa(torch.cat(gu)), L=gL, rc=gr)
    if kind == "trajectory":
        spec, us, goal, sph, x, up = _trajectory_inputs(case, seed)
        P, T, n = case["P"], case["T"], case["n"]
        x = x.double().requires_grad_()
        costs, grads = [], []
        for i in range(0, P, 64):  # a share of the problems at a time
            k = min(64, P - i)
            xi = x[i * (T - 1):(i + k) * (T - 1)]
            segs, R, p = _chain(xi, *_robot_rows(spec))
            own = sph[i:i + k].repeat_interleave(T - 1, 0) if sph is not None else None
            F = _state_cost(xi, segs, spec, own).reshape(k, T - 1).sum(1)
            F = F + _pose_cost(R.reshape(k, T - 1, 3, 3)[:, -1], p.reshape(k, T - 1, 3)[:, -1], goal[i:i + k])
            _, _, p0 = _fk(spec, us[i:i + k])
            tips = torch.cat([p0[:, None], p.reshape(k, T - 1, 3)], 1)
            F = F + 0.5 * W.w_len * (tips.diff(dim=1) ** 2).sum((1, 2))
            q = torch.cat([us[i:i + k][:, None], xi.reshape(k, T - 1, n, 3)], 1)
            v = q.diff(dim=1) / W.dt
            F = F + 0.5 * W.rho_v * (torch.relu(v.abs() - W.vmax) ** 2).sum((1, 2, 3))
            a = q.diff(n=2, dim=1) / W.dt ** 2
            F = F + 0.5 * W.rho_a * (torch.relu(a.abs() - W.amax) ** 2).sum((1, 2, 3))
            grads.append(torch.autograd.grad(F, xi, up[i:i + k].double())[0])
            costs.append(F.detach())
        return dict(cost=torch.cat(costs), x=_soa(torch.cat(grads)))
    if kind == "calibration":
        spec, U, pm, theta = _calibration_inputs(case, seed)
        n = case["n"]
        U = U.double()

        def residual(t):
            return (_chain(U, t[:n], t[n:])[2] - pm).reshape(-1)

        for _ in range(12):  # Gauss-Newton to the optimum
            J = torch.func.jacfwd(residual)(theta)
            theta = theta - torch.linalg.lstsq(J, residual(theta)[:, None]).solution[:, 0]
        return dict(theta=theta, F=0.5 * (residual(theta) ** 2).sum()[None])
    return None


# --------------------------------------------------------------------------------------------------
# The work that no implementation can leave out: inputs read and outputs written once; arithmetic of
# the method (about 150 n flops for one cost of n segments, 380 n with its gradient; for every sample
# near a sphere the distance rows)
# --------------------------------------------------------------------------------------------------
def _eval(n, n_o, grad):
    return (380 if grad else 150) * n + 10 * n * n_o


def _ik_flops(n, P, S, k_init, K, k_final, n_o):
    d = 3 * n
    lm = 2 * _eval(n, n_o, False) + 230 * n + 10 * d * d + d ** 3 / 3
    return P * (S * (k_init + 1) * _eval(n, n_o, True) + K * k_final * lm)


def work(case):
    kind, n = case["kind"], case.get("n", 0)
    d, es = 3 * n, case.get("bits", 64) // 8
    if kind == "kinematics":
        per = d + 12 + 6 * d + (n * 16 * 3 if case["backbone"] else 0)
        return dict(bytes=case["B"] * per * es, flops=case["B"] * (350 * n + (n * 16 * 50 if case["backbone"] else 0)))
    if kind == "gradient":
        B = case["B"]
        return dict(bytes=B * (2 * d + 2) * es + 56 * (B // case["S"] + 1) + 32 * case["n_o"],
                    flops=B * (_eval(n, case["n_o"], False) + _eval(n, case["n_o"], True)))
    if kind == "trajectory":
        B = case["P"] * (case["T"] - 1)
        return dict(bytes=2 * B * d * es + case["P"] * (8 * d + 56 + 32 * case["n_o"]),
                    flops=B * (_eval(n, case["n_o"], False) + _eval(n, case["n_o"], True) + 20 * d))
    if kind == "calibration":
        K = case["K"]
        return dict(bytes=K * (d * es + 24), flops=20 * K * (350 * n + 150 * n + 3 * (2 * n) * (2 * n + 1)))
    if kind == "roadmap":
        R, N, k = case["R"], case["N"], case["k"]
        return dict(bytes=R * (32 * case["n_o"] + N * (8 * d + 1 + 4 * k + 4) + 12 * N * k + 8 * d * case["T"]),
                    flops=R * (N * N * 3 * d + N * (k * 8 * 0.6 + 1.5) * _eval(n, case["n_o"], False)))
    if kind == "ik":
        P = case["P"]
        return dict(bytes=P * (56 + 8 * d + 25),
                    flops=_ik_flops(n, P, case["S"], case["k_init"], case["n_final"], 30, case["n_o"]))
    if kind == "plan":
        P, T = case["P"], case["T"]
        return dict(bytes=P * (8 * d + 56 + 32 * case["n_o"] + 8 * d * T + 42),
                    flops=_ik_flops(n, P, 64, 32, 4, 30, case["n_o"])
                    + P * T * (synth.K_TRAJ + 1) * (_eval(n, case["n_o"], True) + 20 * d))
    if kind == "path":
        P, H = case["P"], case["H"]
        lm = 2 * _eval(n, case["n_o"], False) + 230 * n + 7 * d * d + d ** 3
        return dict(bytes=P * (56 * H + 32 * case["n_o"] + 8 * d * H + 16 * H + 10),
                    flops=_ik_flops(n, P, 64, 32, 8, 30, case["n_o"])
                    + P * H * lm * (synth.K_WARM + synth.K_JOINT))
    flops = size = 0
    for path, n, H, S, no in synth.ragged_items(np.random.default_rng(case["mix"]), case["N"]).tolist():
        d = 3 * n
        lm = 2 * _eval(n, no, False) + 230 * n + 7 * d * d + d ** 3
        flops += _ik_flops(n, 1, S, 64, 8, 30, no) + (H * lm * (synth.K_WARM + synth.K_JOINT) if path else 0)
        size += 56 * H + 32 * no + 8 * d * H + 16 * H + 9
    return dict(bytes=size, flops=flops)
