"""The linear solve of a reverse step, (I - c J(alpha)^T) mu = b: from zero
difference adjoints a first-order step turns the state's adjoint b into mu, so
that J^T mu from sphnse_rhs_adjoint (all five fields synthesised) checks the
iteration (which keeps the three fields of alpha) at sizes around the tiles of
the FP32 synthesis.

Tolerance: FP64 iterates to 1e-14 of |b|, bar 1e-12; FP32 and BF16x3 stop at the
rounding of their contractions, bar 3e-5 of |c J^T mu| as for J^T itself."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from seeded_inputs import coefficients

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16x3"])
@pytest.mark.parametrize("L,nlon", [(1, 6), (15, 54), (31, 96), (42, 128), (53, 162), (100, 324), (127, 384)])
def test_reverse_step_solves_its_linear_system(L, nlon, prec):
    from paper_1009_3308_gb300 import Plan, _capi
    plan = Plan(L, nlon // 2, nlon, 1e-3, 1.0, precision=prec)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    alpha, b = (dev(coefficients(L, s + L, 3.0 / L)) for s in (21, 22))
    abar, dbar = b.clone(), torch.zeros(7, plan.n_coeff, dtype=torch.complex128, device="cuda")
    h = 0.01
    c = h / 1.185            # 1 / ((1 - kappa_1) gamma_1), kappa_1 = -0.1850
    nu = ctypes.c_double(0.0)
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    rc = _capi.lib().sphnse_adjoint_step_explicit(plan._h, h, 1, h, p(alpha), p(abar), p(dbar), ctypes.byref(nu))
    assert rc == 0
    jt = c * plan.rhs_adjoint(alpha, abar)
    res = float((abar - jt - b).norm())
    assert res <= (1e-12 * float(b.norm()) if prec == "fp64" else 3e-5 * float(jt.norm()))
