"""The built-in operator plan of grids of one to two 128-column tiles per SM accumulates in as many
TMEM regions as the per-tile plan: F and the steps are equal bit for bit."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_1706_09161_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.fail("CUDA GPU required for -m gpu tests")
    from paper_1706_09161_gb300 import lbm
    return lbm


# 162 to 300 tiles on 152 SMs: two-dimensional lines of several contraction blocks, aligned and ragged
# rows, three-dimensional ones of one or two; partial last tiles
@pytest.mark.parametrize("grid,kinds", [((1100, 1050), ["bf16split", "bf16x6split", "tf32split"]),
                                        ((1101, 1030), ["bf16x6split", "tf32split"]),
                                        ((64, 64, 64), ["bf16x6split"]), ((72, 30, 100), ["bf16x5split", "bf16x6split"]),
                                        ((75, 75, 75), ["bf16x6split"])])
def test_persistent_plan_sums_as_the_per_tile_plan(L, grid, kinds):
    rng = np.random.default_rng(1901 + sum(grid))
    pb = W.random_problem(rng, len(grid), "mrt", grid)
    pb = dataclasses.replace(pb, alpha=tuple(1.5 + 0.5 * (a - 1.2) / 0.8 for a in pb.alpha))
    C0 = W.random_field(rng, grid)
    for kind in kinds:
        with L.Lattice(pb, C0, kind) as a, L.Lattice(pb, C0, kind) as b:
            b.configure(128, 1, 0, 0, 0)
            b.reset()
            for mu in range(len(grid)):
                assert np.array_equal(a.F(mu), b.F(mu)), (kind, mu)
            a.step(3)
            b.step(3)
            assert np.array_equal(a.f(), b.f()), kind
