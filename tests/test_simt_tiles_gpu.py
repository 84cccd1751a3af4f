"""The CUDA-core operator and the FP64 march over the sizes that select each of their tiles,
with remainders on every side, against the FP64 oracle.

FP32 operator: a sum of N products, each operand and each accumulation rounded to FP32, errs by
at most about (N + 2) 2^-24 of sum |K||C| per node; K and C are non-negative here, so that is
the same fraction of F itself, node by node (N = 520: 3.1e-5; rounding errors of both signs
leave about sqrt(N) of it, which the relative L2 bound of 1e-6 holds to).  FP64: the same with
2^-53 (1e-13 per node), and 1e-12 for the concentration after a few steps.
"""
import numpy as np
import pytest
import torch

from oracle import lbm_oracle as O
from paper_1706_09161_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1706_09161_gb300 import lbm
    return lbm


def _case(grid, seed, collision="mrt"):
    rng = np.random.default_rng(seed)
    pb = W.random_problem(rng, len(grid), collision, grid, spherical=collision == "bgk")
    return pb, W.random_field(rng, grid)


# 32 x 32 tiles; 64 x 64 (M = 300 pads less in 64s); 128 x 64; rows that are no multiple of 16 bytes
@pytest.mark.parametrize("grid", [(33, 31), (130, 70), (300, 300), (304, 299), (301, 300), (520, 500), (35, 70, 34),
                                  (68, 66, 65)])
def test_fp32_operator_tiles(L, grid):
    pb, C0 = _case(grid, 41 + sum(grid))
    with L.Lattice(pb, C0, "fp32") as lat:
        C = lat.C()
        F = O.fractional_terms(O.Operators(pb), torch.tensor(C))
        for mu in range(len(grid)):
            ref = F[mu].numpy()
            got = lat.F(mu)
            assert np.linalg.norm(got - ref) < 1e-6 * np.linalg.norm(ref), mu
            assert np.all(np.abs(got - ref) <= (grid[mu] + 2) * 2.0 ** -24 * np.abs(ref) + 1e-38), mu


# operator tiles of 8 (17 x 13, 64 x 60), 16 (130 x 90, 3-D) and 32 (200 x 198); march tiles of
# 8 x 4, 16 x 16 and 32 x 16 with partial tiles and several z chunks
@pytest.mark.parametrize("grid", [(3, 3), (17, 13), (64, 60), (130, 90), (200, 198), (333, 400), (19, 18, 5),
                                  (34, 33, 40), (49, 48, 47)])
@pytest.mark.parametrize("collision", ["bgk", "mrt"])
def test_fp64_tiles(L, grid, collision):
    pb, C0 = _case(grid, 83 + sum(grid), collision)
    n = 4
    with L.Lattice(pb, C0, "fp64") as lat:
        F = O.fractional_terms(O.Operators(pb), torch.tensor(lat.C()))
        for mu in range(len(grid)):
            ref = F[mu].numpy()
            assert np.max(np.abs(lat.F(mu) - ref)) <= 1e-13 * np.max(np.abs(ref)), mu
        lat.step(n)
        C, C_ref = lat.C(), O.run_C(pb, C0, n).numpy()
        assert np.max(np.abs(C - C_ref)) <= 1e-12 * np.max(np.abs(C_ref))
        assert abs(lat.mass() - C.sum()) <= 1e-12 * np.abs(C).sum()
