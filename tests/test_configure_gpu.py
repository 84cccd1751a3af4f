"""Launch configurations that a caller sets: which values are taken, what they mean after the
kind of march changes, and what a refused one leaves behind.  A configuration changes the schedule
of a step, never its result: populations are equal bit for bit."""
import dataclasses
import re

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
    pb = W.random_problem(rng, len(grid), collision, grid, spherical=collision == "bgk")
    pb = dataclasses.replace(pb, alpha=tuple(1.5 + 0.5 * (a - 1.2) / 0.8 for a in pb.alpha))  # stable over the runs here
    return pb, W.random_field(rng, grid)


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


class Hooks:
    """Device memory from PyTorch's allocator, refused while `refuse` is set."""

    def __init__(self, L):
        self.L, self.refuse = L, False

    def __enter__(self):
        def alloc(nbytes, stream, ctx):
            if self.refuse:
                return None
            return torch.cuda.caching_allocator_alloc(int(nbytes), torch.cuda.current_device(), int(stream or 0))

        self.L.lbm_set_allocator(alloc, lambda ptr, ctx: torch.cuda.caching_allocator_delete(int(ptr)))
        return self

    def __exit__(self, *exc):
        self.L.lbm_set_allocator(None, None)


# a plan whose larger F is refused, or whose fused form is not there after F has grown: the handle
# goes on with the plan, the buffers and the captured graph that it had
@pytest.mark.parametrize("fused", [0, 1])
@pytest.mark.parametrize("kind", ["bf16split", "tf32split"])
def test_a_refused_plan_leaves_the_old_one(L, kind, fused):
    pb, C0 = _case((520, 520), 1409)
    with Hooks(L) as mem, L.Lattice(pb, C0, kind) as a, L.Lattice(pb, C0, kind) as b:
        a.step(130)  # a captured graph of 128 steps and two single ones
        mem.refuse = not fused
        with pytest.raises(L.LBMError):
            a.configure(128, 8, 0, 3, fused)
        mem.refuse = False
        a.step(130)
        b.step(260)
        assert np.array_equal(a.f(), b.f())
        a.configure(128, 8, 0, 3, 0)
        b.configure(128, 8, 0, 3, 0)
        a.step(3)
        b.step(3)
        assert np.array_equal(a.f(), b.f())


def test_a_refused_batch_configuration_leaves_the_old_one(L):
    cases = [_case(g, 1511 + sum(g)) for g in [(37, 20), (64, 64)]]
    args = ([p for p, _ in cases], [c for _, c in cases], "bf16split")
    with Hooks(L) as mem, L.Batch(*args) as a, L.Batch(*args) as b:
        a.step(40)
        mem.refuse = True
        with pytest.raises(L.LBMError):
            L.lbm_configure(a.h, 0, 0, 0, 16, 0)
        mem.refuse = False
        a.step(40)
        b.step(80)
        for i in range(len(cases)):
            assert np.array_equal(a.C(i), b.C(i)), i
            assert a.mass(i) == b.mass(i), i


# with varying coefficients a split needs no larger F; constant ones again would take slots of it
# and go without where they are refused
def test_constant_coefficients_again_without_memory(L):
    pb, C0 = _case((520, 520), 1409)
    one = np.ones(pb.shape)
    with Hooks(L) as mem, L.Lattice(pb, C0, "bf16split") as a, L.Lattice(pb, C0, "bf16split") as b:
        a.set_fields(u=np.stack([pb.u[0] * one, pb.u[1] * one]), g=np.stack([pb.g[0] * one, pb.g[1] * one]))
        for lat in (a, b):
            lat.configure(128, 8, 0, 0, 0)
        mem.refuse = True
        a.set_fields()
        mem.refuse = False
        b.reset()
        a.step(130)
        b.step(130)
        assert np.array_equal(a.f(), b.f())


# the mass is added up in the order of the march's blocks, so that its last bits tell the marches
# and their chunks apart; the populations don't depend on them
def test_the_built_in_chunk_comes_back(L):
    pb, C0 = _case((300, 300), 1703)
    fields = W.smooth_fields(np.random.default_rng(5), pb.grid, "mrt", D0=0.03, g_amp=0.2, u_amp=0.03)

    def mass(lat):
        lat.reset()
        lat.step(5)
        return lat.mass()

    with L.Lattice(pb, C0, "bf16x6split") as a, L.Lattice(pb, C0, "bf16x6split") as b:
        a.set_fields(**fields)
        b.set_fields(**fields)
        built_in = mass(a)
        b.configure(0, 0, 0, 40, 0)
        assert mass(b) != built_in  # (what this test can tell apart)
        b.configure(0, 0, 0, 0, 0)
        assert mass(b) == built_in


@pytest.mark.parametrize("kind", ["fp32", "bf16x6split"])
def test_a_chunk_belongs_to_its_march(L, kind):
    pb, C0 = _case((300, 300), 1703)
    fields = W.smooth_fields(np.random.default_rng(5), pb.grid, "mrt", D0=0.03, g_amp=0.2, u_amp=0.03)

    def run(lat):
        lat.reset()
        lat.step(5)
        return lat.f(), lat.mass()

    def same(x, y):
        return np.array_equal(x[0], y[0]) and x[1] == y[1]

    with L.Lattice(pb, C0, kind) as a, L.Lattice(pb, C0, kind) as b:
        b.configure(0, 0, 0, 3, 0)  # tile rows of the march of constant coefficients
        const = run(b)
        for lat in (a, b):
            lat.set_fields(**fields)
        assert same(run(a), run(b))
        a.configure(0, 0, 0, 7, 0)  # strip rows of the march of varying ones
        varying = run(a)
        a.set_fields()
        b.set_fields()
        assert same(run(b), const)
        a.set_fields(**fields)
        assert same(run(a), varying)
        a.set_fields()
        with L.Lattice(pb, C0, kind) as fresh:
            assert same(run(a), run(fresh))


# what lbm_autotune reports can be passed back: also the built-in split of an elongated grid, above what
# lbm_configure takes as a number, and the built-in persistent plan of one to two tiles per SM
@pytest.mark.parametrize("kind,grid", [("fp32", (400, 33)), ("fp32", (300, 300)), ("bf16x6split", (75, 75, 75)),
                                       ("tf32split", (260, 130))])
def test_a_tuned_configuration_can_be_set_again(L, kind, grid):
    pb, C0 = _case(grid, 1801)
    with L.Lattice(pb, C0, kind) as a, L.Lattice(pb, C0, kind) as b:
        desc = a.autotune(128)
        ks, chunk = (int(re.search(key + r"=(\d+)", desc).group(1)) for key in ("ks", "chunk"))
        bn = int(re.search(r"bn=(\d+)", desc).group(1)) if "bn=" in desc else 0
        b.configure(bn, ks, int("persistent" in desc), chunk, 0)
        for lat in (a, b):
            lat.reset()
            lat.step(5)
        assert np.array_equal(a.f(), b.f()), desc
