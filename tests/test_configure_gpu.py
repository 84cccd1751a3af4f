"""Launch configurations that a caller sets: which values are taken, what they mean after the
kind of march changes, and what a refused one leaves behind.  A configuration changes the schedule
of a step, never its result: populations are equal bit for bit."""
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


def _case(grid, seed, collision="mrt"):
    rng = np.random.default_rng(seed)
    return W.random_problem(rng, len(grid), collision, grid, spherical=collision == "bgk"), W.random_field(rng, grid)


# rows per warp are two per unit of the chunk: values whose double does not fit in 32 bits
@pytest.mark.parametrize("chunk", [2 ** 30 - 1, 2 ** 30, 2 ** 31 - 1])
@pytest.mark.parametrize("kind", ["fp32", "bf16split"])
def test_any_positive_chunk_is_taken(L, kind, chunk):
    cases = [_case(g, 1201 + sum(g)) for g in [(37, 20), (64, 64), (130, 33)]]
    with L.Batch([p for p, _ in cases], [c for _, c in cases], kind) as b:
        b.step(5)
        ref = [b.C(i) for i in range(len(cases))]
        L.lbm_configure(b.h, 0, 0, 0, chunk, 0)
        b.reset()
        b.step(5)
        for i in range(len(cases)):
            assert np.array_equal(b.C(i), ref[i]), i
    pb, C0 = _case((66, 50), 1301)
    fields = W.smooth_fields(np.random.default_rng(5), pb.grid, "mrt", D0=0.03, g_amp=0.2, u_amp=0.03)
    for f in ({}, fields):
        with L.Lattice(pb, C0, kind) as lat:
            lat.set_fields(**f)
            lat.configure(0, 0, 0, 40, 0)
            lat.reset()
            lat.step(5)
            ref = lat.f()
            lat.configure(0, 0, 0, chunk, 0)
            lat.reset()
            lat.step(5)
            assert np.array_equal(lat.f(), ref), bool(f)
