"""The FP32 and BF16x3 paths' transforms at the sizes where their tiling and
radix plans change: every radix of the general ring kernel (8, 4, 2, 3) in
first and later stages, odd numbers of latitudes, remainders of the latitude
and row tiles, the largest longitude count at a low truncation.

Tolerance 3e-5 (global, relative): the bar of these paths."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.rhs import Problem, project, rhs_separable, synthesize
from seeded_inputs import coefficients

pytestmark = pytest.mark.gpu

SIZES = [(1, 6), (2, 8), (3, 12), (8, 36), (16, 54), (21, 72), (33, 108), (40, 128), (47, 144), (53, 162), (62, 192),
         (66, 216), (85, 288), (100, 324), (127, 432), (40, 486), (15, 1536)]


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("prec", ["fp32", "bf16x3"])
@pytest.mark.parametrize("L,nlon", SIZES)
def test_fp32_operations_match_oracle(L, nlon, prec):
    from paper_1009_3308_gb300 import Plan
    prob, plan = Problem(L, nlon, 1e-2, 1.0), Plan(L, nlon // 2, nlon, 1e-2, 1.0, precision=prec)
    a, w = (coefficients(L, s + L, 3.0 / L) * 3.0 for s in (900, 700))
    assert _rel(plan.rhs(_dev(a)).cpu().numpy(), rhs_separable(prob, a)) <= 3e-5
    for g, r in zip(plan.grid_fields(_dev(a)), synthesize(prob, a)):
        assert _rel(g.cpu().numpy(), r) <= 3e-5
    v = np.random.default_rng(L).standard_normal((2, nlon // 2, nlon))
    assert _rel(plan.project(_dev(v[0]), _dev(v[1])).cpu().numpy(), project(prob, v[0], v[1])) <= 3e-5
    got = plan.rhs_adjoint(_dev(a), _dev(w)).cpu().numpy()
    ref = Plan(L, nlon // 2, nlon, 1e-2, 1.0).rhs_adjoint(_dev(a), _dev(w)).cpu().numpy()
    assert _rel(got, ref) <= 3e-5
