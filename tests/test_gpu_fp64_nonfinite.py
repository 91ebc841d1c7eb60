"""Non-finite and overflowing values through the FP64 transforms, on plans of
the tensor-core sums (more than 40 northern latitudes) and of the small ones.

A non-finite coefficient reaches every latitude (its product with the table
does, also where the table underflows), and a plan gives the same results after
such a call as before it.  What overflows is infinite or NaN, never a finite
number that is wrong."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from seeded_inputs import coefficients

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _off(N, m):
    return 0 if m == 0 else N + (m - 1) * (N + 1) - (m - 1) * m // 2


def _plan(L, nlon, nu=1e-2, Om=1.0):
    from paper_1009_3308_gb300 import Plan
    return Plan(L, nlon // 2, nlon, nu, Om)


BAD = [(53, 162, 50, 53), (53, 162, 0, 1), (100, 324, 90, 95), (100, 324, 3, 4), (255, 768, 250, 255),
       (255, 768, 9, 40), (33, 108, 30, 33)]


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("L,nlon,m,l", BAD)
def test_nonfinite_coefficient_reaches_every_output(L, nlon, m, l, bad):
    plan = _plan(L, nlon)
    a, w = coefficients(L, 3, 3.0 / L), coefficients(L, 4, 3.0 / L)
    v = [_dev(np.random.default_rng(k).standard_normal((nlon // 2, nlon))) for k in (0, 1)]
    ops = [lambda a, w: plan.rhs(a), lambda a, w: torch.stack(plan.grid_fields(a)),
           lambda a, w: plan.rhs_adjoint(a, w), lambda a, w: plan.project(*v)]
    ref = [f(_dev(a), _dev(w)) for f in ops]
    i = _off(L, m) + l - max(m, 1)
    ab, wb = a.copy(), w.copy()
    ab[i] = wb[i] = bad
    fin = lambda t: torch.isfinite(torch.view_as_real(t) if t.is_complex() else t)
    assert not fin(plan.rhs(_dev(ab))).any()
    for k, g in enumerate(plan.grid_fields(_dev(ab))):
        # every latitude (u_theta of order 0 is zero times the coefficient)
        assert not fin(g).all(dim=1).any(), k
    assert not fin(plan.rhs_adjoint(_dev(ab), _dev(w))).any()
    assert not fin(plan.rhs_adjoint(_dev(a), _dev(wb))).any()
    vb = v[0].clone()
    vb[5, 7] = bad
    assert not fin(plan.project(vb, v[1])).all(dim=1).any()
    for f, r in zip(ops, ref):
        assert torch.equal(f(_dev(a), _dev(w)), r)


@pytest.mark.parametrize("size", [0.4, 1.0, 2.5, 20.0, 64.0])
@pytest.mark.parametrize("L,nlon", [(255, 768), (100, 324), (53, 162), (33, 108)])
def test_overflowing_vorticity(L, nlon, size):
    # one zonal mode, its vorticity coefficient about size 2^1023
    plan = _plan(L, nlon, 0.0, 0.0)
    a = np.zeros(plan.n_coeff, np.complex128)
    a[L - 1] = min(size / L, 1.9) * 2.0 ** 1023
    exact, got = plan.grid_fields(_dev(a * 2.0 ** -64)), plan.grid_fields(_dev(a))
    ok = torch.isfinite(got[0])
    big = exact[0] * 2.0 ** 64
    assert torch.equal(got[0][ok], big[ok])
    for k in (1, 2):   # the velocity is in range where the vorticity is not
        b = exact[k] * 2.0 ** 64
        assert bool(torch.isfinite(b).any()) and torch.equal(torch.isfinite(got[k]), torch.isfinite(b))
        assert torch.equal(got[k][torch.isfinite(b)], b[torch.isfinite(b)])
    if size <= 1.0:   # the coefficient is finite: so is what it gives away from overflowing latitudes
        assert torch.equal(ok.all(dim=1), torch.isfinite(big).all(dim=1))
    else:
        assert not bool(ok.all())


@pytest.mark.parametrize("L,nlon", [(100, 324), (53, 162), (33, 108)])
def test_overflowing_product(L, nlon):
    # without viscosity and rotation F is quadratic
    plan = _plan(L, nlon, 0.0, 0.0)
    a = coefficients(L, 31, 3.0 / L)
    ref = torch.view_as_real(plan.rhs(_dev(a)))
    for e in range(504, 524):
        got = torch.view_as_real(plan.rhs(_dev(a * 2.0 ** e)))
        ok = torch.isfinite(got)
        assert torch.equal(got[ok], (ref * 2.0 ** 500 * 2.0 ** (2 * e - 500))[ok]), e
    assert not bool(ok.any())
