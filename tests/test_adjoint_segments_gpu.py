"""The adjoint over the segment layouts and tile edges of its kernels, FP32 and FP64, against the
FP64 oracle's adjoint within the stated gradient bars (1e-4 and 1e-8 of each family's largest):
snapshots at 0, inside segments and on their boundaries, segments longer than the run and of one step;
sides around the 64 x 32 tiles of the weights' gradient, with rows that are and are not whole
16-byte groups; off-diagonal D (its dOmega/dD is still an outer product); BGK."""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import lbm_oracle as O
from paper_1706_09161_gb300 import workloads as W
from test_adjoint_gpu import L, check, observations  # noqa: F401

pytestmark = pytest.mark.gpu


def full_D_reference(pb, C0, snaps, obs):
    """The oracle's loss and gradient with the whole tensor D (its loss_and_grad keeps the diagonal)."""
    leaf = [torch.tensor(v, dtype=torch.float64, requires_grad=True) for v in (pb.alpha, pb.p, pb.D, pb.u)]
    ops = O.Operators(pb, alpha=leaf[0], p=leaf[1], D=leaf[2], u=leaf[3])
    f = O.init_populations(ops, torch.tensor(C0))
    loss, t = torch.zeros((), dtype=torch.float64), 0
    for k, ts in enumerate(snaps):
        while t < ts:
            f = O.step(ops, f)
            t += 1
        loss = loss + (O.concentration(f) - obs[k]).square().sum()
    ga, gp, gD, gu = torch.autograd.grad(loss, leaf)
    return float(loss.detach()), torch.cat([ga, gp, torch.diagonal(gD), gu])


@pytest.mark.parametrize("precision,rtol", [("fp32", 1e-4), ("fp64", 1e-8)])
@pytest.mark.parametrize("grid,snaps,ckpt,collision", [
    ((64, 33), [0, 8, 16, 17], 8, "mrt"), ((65, 32), [5, 12], 50, "bgk"), ((68, 67), [2, 30], 1, "mrt"),
    ((35, 130), [7, 9], 4, "mrt"), ((20, 17, 12), [4, 8], 4, "mrt")])
def test_segments_and_tiles(L, monkeypatch, precision, rtol, grid, snaps, ckpt, collision):  # noqa: F811
    rng = np.random.default_rng(7 * sum(grid))
    pb = W.random_problem(rng, len(grid), collision, grid, spherical=collision == "bgk")
    if collision == "mrt" and len(grid) == 2:
        D = [list(r) for r in pb.D]
        D[0][1] = D[1][0] = 0.3 * min(D[0][0], D[1][1])
        pb = dataclasses.replace(pb, D=tuple(tuple(r) for r in D))
        monkeypatch.setattr(O, "loss_and_grad", full_D_reference)
    check(L, pb, W.random_field(rng, grid), snaps, ckpt, precision, rtol)


def test_only_the_initial_state_observed(L):  # noqa: F811
    rng = np.random.default_rng(3)
    pb = W.random_problem(rng, 2, "mrt", (24, 20))
    C0 = W.random_field(rng, pb.grid)
    obs = observations(pb, C0, [0], seed=1)
    with L.Lattice(pb, C0, "fp64") as lat:
        loss, grad = lat.grad([0], obs, 10)
    # the scheme conserves C in feq: the initial state does not depend on any parameter
    assert loss == pytest.approx(float(np.square(C0 - obs[0]).sum()), rel=1e-9)
    assert np.max(np.abs(grad)) < 1e-12
