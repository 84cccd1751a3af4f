"""The D part of the FP32 gradient is summed over a node's populations to FP64's precision.

Two steps of a compact pulse whose amplitude is far below the FP32 spacing of the observations: the
adjoint of the last step is then 2 (C - obs) = -2 obs exactly, and what dL/dD sees of it are
differences of 2^-17 to 2^-14 between neighbours beside a common 14.6.  A sum of the populations'
terms in FP32 rounds at 2^-22 (the product of 14.6 and an off-diagonal rate), a percent of them; to
FP64's precision what is left is the rounding of the forward state (2^-24 of each of a few terms),
within the stated gradient bar of 1e-4."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_1706_09161_gb300 import workloads as W
from test_adjoint_gpu import L  # noqa: F401
from test_adjoint_segments_gpu import full_D_reference

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_D_gradient_beside_a_common_residual(L, seed):  # noqa: F811
    rng = np.random.default_rng(seed)
    grid = (24, 20)
    pb = W.random_problem(rng, 2, "mrt", grid)
    pb = dataclasses.replace(pb, alpha=(2.0, 2.0), D=((0.2, 0.1), (0.1, 0.25)), u=(0.02, -0.03), g=(1.0, 1.0))
    C0 = np.zeros(pb.shape)
    C0[8:12, 10:15] = 1e-12 * (1.0 + rng.random((4, 5)))
    obs = (-7.3125 + rng.integers(-8, 9, size=(1,) + pb.shape) * 2.0 ** -18).astype(np.float64)
    assert np.array_equal(obs, obs.astype(np.float32))
    _, ref = full_D_reference(pb, C0, [2], torch.tensor(obs))
    ref = ref.numpy()[4:6]
    with L.Lattice(pb, C0, "fp32") as lat:
        _, grad = lat.grad([2], obs, 10)
    assert np.all(np.abs(grad[4:6] - ref) <= 1e-4 * np.abs(ref).max()), (grad[4:6], ref)
