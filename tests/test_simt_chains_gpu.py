"""Accumulation chains of the FP32 CUDA-core operator, bit for bit: the products of a chain are added
in contraction order by fused multiply-adds, a slice's chains in order, then the slices in order.
The reference does the same on the host in extended precision, rounded to FP32 after every
operation (a product of two FP32 numbers has 48 bits)."""
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


def chained(K, C, slices, chains):
    """sum_l K[n, l] C[:, l] for every n: `slices` x `chains` chains over whole blocks of 32."""
    wide = np.longdouble
    nkb = -(-K.shape[0] // 32)
    total = None
    for r in range(slices):
        part = None
        for j in range(r * chains, (r + 1) * chains):
            lo, hi = (32 * (i * nkb // (slices * chains)) for i in (j, j + 1))
            acc = np.zeros((C.shape[0], K.shape[0]), dtype=np.float32)
            for l in range(lo, min(hi, K.shape[0])):
                acc = (C[:, l, None].astype(wide) * K[None, :, l].astype(wide) + acc.astype(wide)).astype(np.float32)
            part = acc if part is None else part + acc
        total = part if total is None else total + part
    return total


# grids whose built-in split has as many slices as chains (100^2, 512^2) and fewer
@pytest.mark.parametrize("grid,slices,chains", [((100, 100), 4, 1), ((512, 512), 4, 1), ((300, 300), 4, 2),
                                                ((230, 518), 2, 4), ((64, 64, 64), 1, 2), ((98, 49, 58), 1, 2)])
def test_chains_of_the_built_in_split(L, grid, slices, chains):
    if np.finfo(np.longdouble).nmant < 100:
        pytest.skip("needs a long double of at least 100 bits")
    rng = np.random.default_rng(1801 + sum(grid))
    pb = W.random_problem(rng, len(grid), "mrt", grid)
    with L.Lattice(pb, W.random_field(rng, grid), "fp32") as lat:
        C = lat.C().astype(np.float32)
        for mu, n in enumerate(grid):
            K = L.lbm_frac_matrix(L.params_from_problem(pb), mu).astype(np.float32)
            lines = np.moveaxis(C, len(grid) - 1 - mu, -1).reshape(-1, n)
            F = np.moveaxis(lat.F(mu), len(grid) - 1 - mu, -1).reshape(-1, n)
            rows = rng.choice(lines.shape[0], size=4, replace=False)
            assert np.array_equal(F[rows], chained(K, lines[rows], slices, chains).astype(np.float64)), mu
