"""Sums that kernels leave as one partial per block: the derivative in nu that
comes with J^T w, at coefficient counts around the block size and for the plans
whose blocks are orders, and the objective on a grid with far more latitudes
than coefficients.

Tolerance 1e-13 of the sum of magnitudes: at most 2e4 products in FP64 (2e4
times 1.1e-16 if every rounding had the same sign, 1e-14 at random)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from seeded_inputs import coefficients

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _degrees(L):
    return np.concatenate([np.arange(max(m, 1), L + 1) for m in range(L + 1)])


@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16x3"])
@pytest.mark.parametrize("L,nlon", [(1, 6), (21, 72), (22, 72), (31, 96), (53, 162), (100, 324), (127, 384)])
def test_adjoint_nu_derivative(L, nlon, prec):
    from paper_1009_3308_gb300 import Plan
    plan = Plan(L, nlon // 2, nlon, 1e-2, 1.0, precision=prec)
    a, w = (coefficients(L, s + L, 3.0 / L) for s in (5, 6))
    out, nu = plan.rhs_adjoint(_dev(a), _dev(w), want_nu=True)
    k = _degrees(L)
    terms = k * (k + 1.0) * (a.real * w.real + a.imag * w.imag)
    assert abs(nu + terms.sum()) <= 1e-13 * np.abs(terms).sum()
    assert torch.equal(out, plan.rhs_adjoint(_dev(a), _dev(w)))


def test_objective_with_more_latitudes_than_coefficients():
    from paper_1009_3308_gb300 import Plan
    plan = Plan(1, 768, 1536, 1e-2, 1.0)
    a = coefficients(1, 4, 1.0)
    J, _ = plan.objective(_dev(a), _dev(a), 0.0, float(np.pi))
    # the whole sphere: half of sum s_m |alpha|^2, s_0 = 1, s_m = 2
    m = np.array([0, 1])
    want = 0.5 * float(np.sum(np.where(m == 0, 1.0, 2.0) * np.abs(a) ** 2))
    assert abs(J - want) <= 1e-13 * want
