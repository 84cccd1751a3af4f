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


# clusters of eight CTAs fill fewer SMs than there are, and 18 tiles would take two waves of them: the
# built-in plan of ragged rows, and of varying coefficients on aligned ones, is 64 columns split four ways
@pytest.mark.parametrize("grid,fields", [((301, 300), False), ((300, 301), True)])
def test_built_in_clusters_are_resident(L, grid, fields):
    rng = np.random.default_rng(2201)
    pb = W.random_problem(rng, 2, "mrt", grid)
    C0 = W.random_field(rng, grid)
    coeff = W.smooth_fields(np.random.default_rng(5), grid, "mrt", D0=0.03, g_amp=0.2, u_amp=0.03)
    with L.Lattice(pb, C0, "tf32split") as a, L.Lattice(pb, C0, "tf32split") as b:
        b.configure(64, 4, 0, 0, 0)
        for lat in (a, b):
            if fields:
                lat.set_fields(**coeff)
            lat.reset()
        for mu in range(2):
            assert np.array_equal(a.F(mu), b.F(mu)), mu
        a.set_fields()  # (constant coefficients again: the plan of a new handle)
        with L.Lattice(pb, C0, "tf32split") as new:
            assert np.array_equal(a.F(0), new.F(0))
