"""Collide-stream kernels and the per-tile operator at the edges of their tiles, and the stores
that a call of several steps leaves out, against the FP64 oracle.

Concentrations: 6x the error that the form's own arithmetic makes when re-run on the CPU
(``arith_bounds.bounds``, never below 1e-5), in relative L2 and node by node.  The mass is the
sum of the C that the kernel stores: rel 1e-6 of sum |C|, FP32 rounding of each term counted.
Operator: the split's rounding plus 2 sqrt(N) roundings of 2^-23 of FP32 accumulation, as a
relative L2 (all terms are non-negative).  Where only the schedule differs, results are equal bit
for bit.
"""
import dataclasses

import numpy as np
import pytest
import torch

import arith_bounds
from oracle import lbm_oracle as O
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
    pb = dataclasses.replace(pb, alpha=tuple(1.5 + 0.5 * (a - 1.2) / 0.8 for a in pb.alpha))
    return pb, W.random_field(rng, grid)


# strips of 64 (even rows) or 32 nodes (odd rows): below, at and above one strip; rows below, at
# and above a ring block (16) and a chunk (8), the last chunk of one row
@pytest.mark.parametrize("precision", ["fp32", "bf16split", "bf16x6split"])
@pytest.mark.parametrize("collision", ["bgk", "mrt"])
def test_batch_strips(L, precision, collision):
    sizes = [(3, 3), (31, 9), (33, 16), (63, 17), (64, 8), (65, 33), (66, 25), (128, 7), (130, 70), (191, 41)]
    cases = [_case(g, 211 + sum(g), collision) for g in sizes]
    n = 6
    with L.Batch([p for p, _ in cases], [c for _, c in cases], precision) as b:
        b.step(n)
        for i, (pb, C0) in enumerate(cases):
            C = b.C(i)
            arith_bounds.check_form(C, pb, C0, n, precision, f"{sizes[i]}")
            assert abs(b.mass(i) - C.sum()) <= 1e-6 * np.abs(C).sum(), sizes[i]


# tiles of 32 x 16 nodes with and without remainders, one to several z chunks, the shortest box
@pytest.mark.parametrize("precision", ["fp32", "bf16split", "bf16x6split", "tf32split"])
@pytest.mark.parametrize("grid", [(4, 3, 3), (32, 16, 17), (36, 17, 33), (64, 15, 16), (28, 33, 50)])
def test_3d_march_chunks(L, precision, grid):
    pb, C0 = _case(grid, 307 + sum(grid))
    n = 5
    f = []
    for chunk in (0, 1, 2, grid[2]):
        with L.Lattice(pb, C0, precision) as lat:
            lat.configure(0 if precision == "fp32" else 128, 1, 0, chunk, 0)
            lat.reset()
            lat.step(n)
            f.append(lat.f())
            C, mass = lat.C(), lat.mass()
        assert np.array_equal(f[0], f[-1]), chunk
        assert abs(mass - C.sum()) <= 1e-6 * np.abs(C).sum(), chunk
    arith_bounds.check_form(C, pb, C0, n, precision, f"{grid}")


# rows that TMA cannot store, where the CTAs of a tile add their partial tiles themselves, and
# grids small enough for 64-column tiles; sides below, at and above a tile
@pytest.mark.parametrize("kind", ["bf16split", "bf16x5split", "bf16x6split", "tf32split"])
@pytest.mark.parametrize("grid", [(301, 203), (129, 257), (63, 300), (256, 255), (67, 65, 30), (48, 48, 48)])
def test_operator_built_in_plan(L, kind, grid):
    split = {"bf16split": 4e-5, "bf16x5split": 2e-5, "bf16x6split": 2e-6, "tf32split": 2e-6}[kind]
    pb, C0 = _case(grid, 401 + sum(grid))
    with L.Lattice(pb, C0, kind) as lat:
        F = O.fractional_terms(O.Operators(pb), torch.tensor(lat.C()))
        for mu, N in enumerate(grid):
            tol = max(split, 2.0 * np.sqrt(N) * 2.0 ** -23)
            assert arith_bounds.rel_l2(lat.F(mu), F[mu].numpy()) < tol, mu


# C is stored by the last step of a call only (133 steps: a captured graph and single steps)
@pytest.mark.parametrize("kind", ["fp32", "bf16split", "bf16x5split", "bf16x6split", "tf32split"])
@pytest.mark.parametrize("grid,fields", [((68, 50), False), ((67, 50), False), ((36, 20, 18), False),
                                         ((35, 20, 18), False), ((68, 50), True), ((36, 20, 18), True)])
def test_one_call_equals_single_steps(L, kind, grid, fields):
    pb, C0 = _case(grid, 503 + sum(grid))
    n = 133
    with L.Lattice(pb, C0, kind) as a, L.Lattice(pb, C0, kind) as b:
        for lat in (a, b):
            if fields:
                x = np.linspace(0.0, 1.0, grid[0]) * np.ones(pb.shape)
                d = pb.d
                lat.set_fields(D=np.array(pb.D).reshape((d, d) + (1,) * d) * (1.0 + 0.3 * x),
                               g=np.stack([1.0 + 0.2 * x] * d), u=np.stack([0.02 * x] * d))
        a.step(n)
        for _ in range(n):
            b.step(1)
        assert np.array_equal(a.f(), b.f())
        assert np.array_equal(a.C(), b.C())


@pytest.mark.parametrize("kind", ["fp32", "bf16split", "bf16x6split"])
def test_one_batch_call_equals_single_steps(L, kind):
    cases = [_case(g, 601 + sum(g)) for g in [(37, 20), (64, 64), (130, 33)]]
    n = 133
    args = ([p for p, _ in cases], [c for _, c in cases], kind)
    with L.Batch(*args) as a, L.Batch(*args) as b:
        a.step(n)
        for _ in range(n):
            b.step(1)
        for i in range(len(cases)):
            assert np.array_equal(a.C(i), b.C(i)), i


# strips of 64 or 32 nodes at their edges, one to many rows per warp, coefficients per node
@pytest.mark.parametrize("kind", ["fp32", "bf16split", "bf16x6split", "tf32split"])
@pytest.mark.parametrize("collision", ["bgk", "mrt"])
@pytest.mark.parametrize("grid", [(3, 3), (31, 17), (33, 34), (64, 18), (66, 7), (130, 70)])
def test_fields_strips(L, kind, collision, grid):
    pb, C0 = _case(grid, 701 + sum(grid), collision)
    fields = W.smooth_fields(np.random.default_rng(5), grid, collision, D0=0.03, g_amp=0.2, u_amp=0.03)
    n = 6
    f = []
    with L.Lattice(pb, C0, kind) as lat:
        for with_fields in (True, False, True):  # back to constant coefficients and on again
            lat.set_fields(**(fields if with_fields else {}))
        for chunk in (1, 3, 40):
            lat.configure(0, 0, 0, chunk, 0)
            lat.reset()
            lat.step(n)
            f.append(lat.f())
            C, mass = lat.C(), lat.mass()
            assert np.array_equal(f[0], f[-1]), chunk
            assert abs(mass - C.sum()) <= 1e-6 * np.abs(C).sum(), chunk
    l2_tol, node_tol, ref = arith_bounds.bounds(pb, C0, n, kind, fields=fields)
    arith_bounds.assert_close(C, ref, l2_tol, node_tol, f"{grid} {collision} {kind}")


# a split contraction adds its partial tiles in the operator when coefficients vary, in the march
# when they don't, also after the coefficients are constant again
@pytest.mark.parametrize("kind", ["bf16split", "bf16x6split"])
def test_fields_with_a_split_contraction(L, kind):
    pb, C0 = _case((260, 200), 809)
    one = np.ones(pb.shape)
    with L.Lattice(pb, C0, kind) as a, L.Lattice(pb, C0, kind) as b:
        for lat in (a, b):
            lat.configure(128, 2, 0, 0, 0)
            lat.reset()
        b.set_fields(u=np.stack([pb.u[0] * one, pb.u[1] * one]))
        for mu in range(2):
            assert arith_bounds.rel_l2(b.F(mu), a.F(mu)) < {"bf16split": 4e-5, "bf16x6split": 2e-6}[kind], mu
        b.set_fields()
        a.step(4)
        b.step(4)
        assert np.array_equal(a.f(), b.f())


# elongated grids: more contraction slices than the short axis has blocks of 32 (some are empty)
@pytest.mark.parametrize("grid", [(400, 33), (35, 300), (257, 3)])
def test_fp32_split_of_elongated_grids(L, grid):
    pb, C0 = _case(grid, 1009 + sum(grid))
    with L.Lattice(pb, C0, "fp32") as lat:
        F = O.fractional_terms(O.Operators(pb), torch.tensor(lat.C()))
        for mu, N in enumerate(grid):
            ref = F[mu].numpy()
            assert np.all(np.abs(lat.F(mu) - ref) <= (N + 2) * 2.0 ** -24 * np.abs(ref) + 1e-38), mu
        lat.configure(0, 0, 0, 0, 0)  # the built-in split is accepted again
