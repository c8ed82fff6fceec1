"""The warp's LM steps keep the normal equations of an accepted trial and stop where the damping leaves no change. Both
leave the result as it is: the states equal, bit for bit, those of steps that form everything anew and run on to the
last iteration. Targets within and out of reach, states at and near zero, spheres that the robot touches."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest
import torch

import oracle as O
from gpu_util import orc_robot, targets_dev
from paper_2607_11340_gb300 import api, build_lib, synth

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "cr_host.h"
#include "cr_warp.cuh"
using namespace crk;
template <typename V>
__global__ void k_run(RobotK<float> rb, WeightsK<float> w, const double* targets, int64_t P, const Sphere4<float>* sph,
                      int no, int iters, int plain, float* u_io, int* steps) {
  constexpr int N = 3, D = 3 * N;
  __shared__ V scr[4 * 32];
  const int64_t p = blockIdx.x;
  const int lane = threadIdx.x;
  float u[D];
  for (int q = 0; q < D; ++q) u[q] = u_io[q * P + p];
  const TargetK<float> tg = load_target<float>(targets, P, p, CR_TASK_IK6);
  const AugSlots<D> sl = aug_slots<D>(lane);
  V lam = V(1e-3), nu = V(2);
  WarpNormal<float, D> nm;
  nm.held = false;
  int it = 0;
  for (; it < iters; ++it) {
    if (plain) nm.held = nm.solved = false;
    if (!warp_lm_step<float, N, true, V>(rb, w, tg, sph, no, u, sl, lam, nu, scr, scr + 32, scr + 64, scr + 96, nm)) break;
  }
  for (int q = 0; q < D; ++q)
    if (q == lane) u_io[q * P + p] = u[q];
  if (lane == 0) steps[p] = it;
}
extern "C" __attribute__((visibility("default"))) int run(const cr_robot* r, const cr_weights* w, const double* targets,
    int64_t P, const void* sph, int no, int iters, int plain, int wide, float* u, int* steps) {
  const RobotK<float> rb = crh::robot_k<float>(*r);
  const WeightsK<float> wk = crh::weights_k<float>(*w);
  const Sphere4<float>* s = (const Sphere4<float>*)sph;
  if (wide) k_run<double><<<(unsigned)P, 32>>>(rb, wk, targets, P, s, no, iters, plain, u, steps);
  else k_run<float><<<(unsigned)P, 32>>>(rb, wk, targets, P, s, no, iters, plain, u, steps);
  cudaError_t e = cudaGetLastError();
  return (int)(e == cudaSuccess ? cudaDeviceSynchronize() : e);
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("warp_lm")
    src, so = str(d / "warp_lm.cu"), str(d / "warp_lm.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([build_lib.nvcc()] + build_lib.NVCC_FLAGS + build_lib.ARCH + ["-shared", "-cudart", "shared", src,
                                                                                 "-o", so], check=True)
    fn = C.CDLL(so).run
    P = C.c_void_p
    fn.argtypes = [P, P, P, C.c_int64, P, C.c_int, C.c_int, C.c_int, C.c_int, P, P]
    return fn


@pytest.mark.parametrize("n_o", [0, 24])
@pytest.mark.parametrize("wide", [0, 1])
def test_same_as_plain_steps(run, wide, n_o):
    spec, w, P, iters = synth.ROBOT_FAMILY, synth.WEIGHTS, 512, 60
    spec = type(spec)(L=spec.L[:3], rc=spec.rc, umax=spec.umax, nb=spec.nb)
    rng = np.random.default_rng(10 + n_o)
    U = synth.hexagon_states(rng, P, 3, spec.umax)
    tg = synth.pose_targets(O.fk(orc_robot(spec), U)[0], "pose")
    tg[::7, :3] *= 5.0                                        # out of reach
    start = U + 0.2 * spec.umax * rng.normal(size=U.shape)
    start[::5] = U[::5]                                       # at the solution
    start[1::11] = 0.0
    start[2::11, :4] *= 1e-12
    bb = O.fk(orc_robot(spec), U, backbone=True)[1].reshape(-1, 3)
    sph = np.concatenate([bb[rng.integers(0, len(bb), n_o)] + rng.normal(0, 0.02, (n_o, 3)),
                          np.full((n_o, 1), 0.01) + spec.body_radius + w.delta], axis=1)
    r, wt, tgd = api.robot_struct(spec), api.weights_struct(w), targets_dev(tg)
    sd = torch.as_tensor(np.concatenate([sph, np.zeros((1, 4))]), dtype=torch.float32, device="cuda")

    def solve(plain):
        u = torch.as_tensor(start.T.copy(), dtype=torch.float32, device="cuda")
        steps = torch.zeros(P, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        assert run(C.addressof(r), C.addressof(wt), tgd.data_ptr(), P, sd.data_ptr(), n_o, iters, plain, wide,
                   u.data_ptr(), steps.data_ptr()) == 0
        return u, steps

    (u, steps), (up, sp) = solve(0), solve(1)
    assert bool((sp == iters).all()) and float((steps < iters).float().mean()) > 0.25
    assert bool(torch.isfinite(u).all())
    assert torch.equal(u, up)
