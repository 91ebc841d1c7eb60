"""Ends of the reverse step's linear solve that need no iteration: a zero right
side (mu = 0 whatever the next state holds) and one beyond the range of the
norms (refused, whatever the residual that follows it)."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from seeded_inputs import coefficients

pytestmark = pytest.mark.gpu

E_NONFINITE = -5


def _step(plan, alpha, abar):
    from paper_1009_3308_gb300 import _capi
    dbar = torch.zeros(7, plan.n_coeff, dtype=torch.complex128, device="cuda")
    nu = ctypes.c_double(0.0)
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    rc = _capi.lib().sphnse_adjoint_step_explicit(plan._h, 0.01, 1, 0.01, p(alpha), p(abar), p(dbar), ctypes.byref(nu))
    return rc, dbar


@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16x3"])
@pytest.mark.parametrize("L,nlon", [(31, 96), (100, 324)])
def test_zero_right_side(L, nlon, prec):
    from paper_1009_3308_gb300 import Plan
    plan = Plan(L, nlon // 2, nlon, 1e-3, 1.0, precision=prec)
    a = coefficients(L, 21, 3.0 / L)
    a[7] = np.nan
    abar = torch.zeros(plan.n_coeff, dtype=torch.complex128, device="cuda")
    rc, dbar = _step(plan, torch.from_numpy(a).cuda(), abar)
    assert rc == 0
    assert bool((abar == 0).all()) and bool((dbar == 0).all())


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("value", [float("nan"), float("inf"), 2.0e300])
def test_right_side_beyond_the_norms_is_refused(value, prec):
    from paper_1009_3308_gb300 import Plan
    L, nlon = 31, 96
    plan = Plan(L, nlon // 2, nlon, 0.0, 0.0, precision=prec)
    alpha = torch.zeros(plan.n_coeff, dtype=torch.complex128, device="cuda")
    b = torch.zeros_like(alpha)
    b[7] = complex(value, value)
    rc, _ = _step(plan, alpha, b)
    assert rc == E_NONFINITE
    b.fill_(1.0)
    assert _step(plan, alpha, b)[0] == 0   # nothing is left for the next call
