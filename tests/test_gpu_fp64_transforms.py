"""The FP64 path's transforms at the sizes where their tiling and radix plans
change: longitude counts with every radix the fixed-point ring kernel uses
(8, 4, 2, 9, 3), odd numbers of latitudes and of northern latitudes, tile
remainders of the Legendre sums, the smallest plan and the largest longitude
count at a low truncation.

Tolerance 1e-12 (global, relative): the bar of the FP64 path.  Scaling by a
power of two commutes with every rounding of the path, so it is exact."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.rhs import Problem, project, rhs_separable, synthesize
from seeded_inputs import coefficients, random_packed

pytestmark = pytest.mark.gpu

SIZES = [(1, 6), (2, 8), (4, 16), (8, 36), (16, 54), (21, 72), (33, 108), (42, 128), (47, 144), (53, 162), (63, 256),
         (66, 216), (85, 288), (100, 324), (40, 486), (20, 1458), (15, 1536)]


def _plan(L, nlon, nu=1e-2, Om=1.0):
    from paper_1009_3308_gb300 import Plan
    return Plan(L, nlon // 2, nlon, nu, Om)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("L,nlon", SIZES)
def test_fp64_operations_match_oracle(L, nlon):
    prob, plan = Problem(L, nlon, 1e-2, 1.0), _plan(L, nlon)
    a = coefficients(L, 900 + L, 3.0 / L) * 3.0
    assert _rel(plan.rhs(_dev(a)).cpu().numpy(), rhs_separable(prob, a)) <= 1e-12
    got = plan.grid_fields(_dev(a))
    for g, r in zip(got, synthesize(prob, a)):
        assert _rel(g.cpu().numpy(), r) <= 1e-12
    rng = np.random.default_rng(L)
    v = rng.standard_normal((2, nlon // 2, nlon))
    assert _rel(plan.project(_dev(v[0]), _dev(v[1])).cpu().numpy(), project(prob, v[0], v[1])) <= 1e-12


@pytest.mark.parametrize("L,nlon", [(5, 18), (33, 108), (47, 144), (100, 324), (127, 384)])
def test_fp64_adjoint_is_the_transpose(L, nlon):
    # <J v, w> = <v, J^T w> with J v from the exact polarisation of the
    # quadratic F: J(a) v = (F(a + v) - F(a - v)) / 2
    plan = _plan(L, nlon)
    a, v, w = (coefficients(L, s, 3.0 / L) for s in (11, 12, 13))
    jv = 0.5 * (plan.rhs(_dev(a + v)) - plan.rhs(_dev(a - v))).cpu().numpy()
    jtw = plan.rhs_adjoint(_dev(a), _dev(w)).cpu().numpy()
    dot = lambda x, y: float(np.sum(x.real * y.real + x.imag * y.imag))
    scale = np.linalg.norm(jv) * np.linalg.norm(w)
    assert abs(dot(jv, w) - dot(v, jtw)) <= 1e-12 * scale


@pytest.mark.parametrize("L,nlon", [(33, 108), (63, 192), (100, 324)])
def test_fp64_power_of_two_scaling_is_exact(L, nlon):
    # without viscosity and rotation F is quadratic
    plan = _plan(L, nlon, nu=0.0, Om=0.0)
    a = _dev(coefficients(L, 31, 3.0 / L))
    ref = plan.rhs(a)
    for e in (-200, -30, 40, 200):
        assert torch.equal(plan.rhs(a * 2.0 ** e), ref * 2.0 ** (2 * e))
    assert bool((plan.rhs(a * 0.0) == 0).all())


def test_fp64_nonfinite_input_reaches_the_output():
    plan = _plan(33, 108)
    for bad in (float("nan"), float("inf")):
        a = coefficients(33, 3, 0.1)
        a[40] = bad
        assert not bool(torch.isfinite(torch.view_as_real(plan.rhs(_dev(a)))).any(dim=1).all())
        assert bool(torch.isnan(plan.grid_fields(_dev(a))[0]).any())
