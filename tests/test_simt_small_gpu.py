"""The unsplit FP32 operator at the sizes that select its kernels (256 threads up to two 32 x 32 tiles
per SM, else 64 threads; one chain or two), with remainders on every side, against the oracle: N
products and additions rounded to FP32, all terms non-negative, so at most (N + 2) 2^-24 of F per
node.  A batch member is summed as the unsplit operator of one problem is, bit for bit."""
import numpy as np
import pytest
import torch

from oracle import lbm_oracle as O
from paper_1706_09161_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.fail("CUDA GPU required for -m gpu tests")
    from paper_1706_09161_gb300 import lbm
    return lbm


def _case(grid, seed):
    rng = np.random.default_rng(seed)
    return W.random_problem(rng, len(grid), "mrt", grid), W.random_field(rng, grid)


@pytest.mark.parametrize("ks", [0, 1])  # the built-in split, and none
@pytest.mark.parametrize("grid", [(3, 3), (33, 31), (64, 64), (50, 61), (65, 40), (390, 383), (401, 399), (16, 16, 16),
                                  (33, 34, 35), (100, 30, 20)])
def test_unsplit_operator(L, grid, ks):
    pb, C0 = _case(grid, 2001 + sum(grid))
    with L.Lattice(pb, C0, "fp32") as lat:
        lat.configure(0, ks)
        F = O.fractional_terms(O.Operators(pb), torch.tensor(lat.C()))
        for mu, n in enumerate(grid):
            ref = F[mu].numpy()
            assert np.all(np.abs(lat.F(mu) - ref) <= (n + 2) * 2.0 ** -24 * np.abs(ref) + 1e-38), mu


@pytest.mark.parametrize("sizes", [[(48, 48), (64, 50), (130, 97), (390, 383), (401, 399)],
                                   [(33, 34, 35), (64, 64, 64), (20, 30, 12)]])
def test_batch_members_are_summed_as_one_problem_is(L, sizes):
    cases = [_case(g, 2101 + sum(g)) for g in sizes]
    with L.Batch([p for p, _ in cases], [c for _, c in cases], "fp32") as b:
        b.step(3)
        for i, (pb, C0) in enumerate(cases):
            with L.Lattice(pb, C0, "fp32") as lat:
                lat.configure(0, 1)
                lat.reset()
                lat.step(3)
                assert np.array_equal(b.C(i), lat.C()), sizes[i]
