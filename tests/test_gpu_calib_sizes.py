"""Calibration at the sizes where its tiles of 32 poses, blocks of 4 tiles and the cap on blocks begin and end."""
import numpy as np
import pytest
import torch

import oracle as O
from gpu_util import dev_soa, orc_robot
from paper_2607_11340_gb300 import api, lib, synth

pytestmark = pytest.mark.gpu


def _spec(n):
    return synth.RobotSpec(L=(0.12, 0.10, 0.08, 0.1, 0.09, 0.11)[:n], rc=0.005, umax=0.01)


def _poses(spec, K, seed):
    rng = np.random.default_rng(seed)
    U = synth.hexagon_states(rng, K, spec.n, spec.umax)
    nom = np.concatenate([spec.L, np.full(spec.n, spec.rc)])
    true = nom * (1 + rng.uniform(-0.05, 0.05, nom.shape))
    P = O.fk(O.make_robot(list(true[:spec.n]), list(true[spec.n:]), spec.umax, nb=spec.nb), U)[0][:, 9:12]
    return U, P + rng.normal(0, 5e-4, P.shape), nom


@pytest.mark.parametrize("n", [1, 3, 6])
@pytest.mark.parametrize("K", [1, 31, 33, 129])
def test_iterates_against_the_oracle(n, K):
    """Three iterations: rounding 1e-15 times the damped system's condition, at most 12 / (1e-3 / 27) = 3e5,
    with a margin of 30."""
    spec = _spec(n)
    U, P, nom = _poses(spec, K, 10 * n + K)
    ref = O.calibrate(orc_robot(spec), U, P, nom, 3, history=True)
    th, F, hist = api.calibrate(spec, dev_soa(U, torch.float64), dev_soa(P, torch.float64), nom, iters=3, history=True)
    np.testing.assert_allclose(hist.cpu().numpy(), ref["hist"], rtol=1e-8)
    assert torch.equal(th, hist[-1])


@pytest.mark.parametrize("K", [304 * 128 - 1, 304 * 128 + 33])
def test_sums_over_more_tiles_than_blocks(K):
    """The sums of all poses equal those of two shares added: K products added in FP64 in two orders."""
    spec = _spec(3)
    U, P, nom = _poses(spec, K, 3)
    Ud, Pd = dev_soa(U, torch.float64), dev_soa(P, torch.float64)
    theta = torch.as_tensor(nom, dtype=torch.float64, device="cuda")
    whole = api.CalibShard(spec, Ud, Pd)
    cut = 5000
    a = api.CalibShard(spec, Ud[:, :cut].contiguous(), Pd[:, :cut].contiguous())
    b = api.CalibShard(spec, Ud[:, cut:].contiguous(), Pd[:, cut:].contiguous())
    s, t = whole.sums(theta), a.sums(theta) + b.sums(theta)
    NP = 2 * spec.n
    d = torch.stack([s[i * (i + 3) // 2] for i in range(NP)] + [2 * s[-1]]).sqrt()  # column norms, |r| last
    rows = [(i, j) for i in range(NP) for j in range(i + 1)] + [(i, NP) for i in range(NP)] + [(NP, NP)]
    size = torch.stack([d[i] * d[j] for i, j in rows])  # a sum of products is at most this
    assert torch.all((s - t).abs() <= 2 * K * 2.0 ** -53 * size)
    assert torch.equal(whole.cost(theta)[0], s[-1])  # the cost piece adds in the same order
