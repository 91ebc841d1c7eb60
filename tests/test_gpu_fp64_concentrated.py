"""Rounding of the FP64 Legendre sums where the large terms of a state or field
meet small table entries of their row: one mode, or one order with a falling
spectrum, whose degrees lie well below those that are largest at the polar
latitudes, and a field on one polar ring.

The reference takes the plan's own table (the library's host routine on the
plan's nodes) and sums it in extended precision, so that what is left are the
roundings of the sums themselves: the coefficient sets (three), the products and
their sum (two, S the sum of magnitudes; the sums are exact up to 2^-57 S), the
hemispheres (one), the factors of 1/sin (three) and the longitude transform
(one): ten roundings of 2^-53 S at most, S the largest over the output."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

LD = np.longdouble
PI = LD("3.14159265358979323846264338327950288")
TOL = 10 * 2.0 ** -53


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _off(N, m):
    return 0 if m == 0 else N + (m - 1) * (N + 1) - (m - 1) * m // 2


def _eps(l, m):
    l, m = np.asarray(l, LD), LD(m)
    return np.sqrt(np.maximum(l * l - m * m, 0) / (4 * l * l - 1))


def _circle(m, M):
    """cos and sin of 2 pi m q / M, q = 0 .. M - 1."""
    ang = 2 * PI / M * (np.arange(M) * m % M)
    return np.cos(ang), np.sin(ang)


def _table(plan, m):
    """x, sin, w of every latitude and Pt_K^m, K = m .. L + 1, at all of them."""
    from paper_1009_3308_gb300 import _capi
    _, x, s, w = (t.numpy() for t in plan.nodes())
    nh, cnt = (plan.nlat + 1) // 2, plan.L + 2 - m
    out = np.zeros((cnt, nh))
    p = lambda a: a.ctypes.data_as(_capi.c_double_p)
    xn, sn = np.ascontiguousarray(x[:nh]), np.ascontiguousarray(s[:nh])
    assert _capi.lib().sphnse_host_legendre(plan.L + 1, m, nh, p(xn), p(sn), p(out)) == 0
    sign = (-1.0) ** np.arange(cnt)[:, None]
    south = (sign * out)[:, :plan.nlat // 2][:, ::-1]
    return x, s, w, np.concatenate([out, south], axis=1).astype(LD)


def _spectra(N, nlon, state):
    rng = np.random.default_rng(5)
    if isinstance(state, int):
        return {state: 1.0 + rng.random()}
    kind, p, m = state
    f = (lambda l: np.exp(-p * (l - m))) if kind == "exp" else (lambda l: float(l) ** -p)
    return {l: float(rng.standard_normal() * f(l)) for l in range(max(m, 1), N + 1)}


CASES = [(511, 1536, 8, 9), (511, 1536, 8, 13), (511, 1536, 12, 13), (511, 1536, 8, ("exp", 0.3, 8)),
         (511, 1536, 1, ("pow", 4, 1)), (511, 1536, 0, ("pow", 4, 0)), (511, 1536, 200, 200),
         (255, 768, 8, 8), (255, 768, 1, 1), (100, 324, 9, 9), (100, 324, 1, ("pow", 2, 1)), (85, 288, 3, 3),
         (53, 162, 2, 33), (20, 1458, 1, ("pow", 4, 1)), (31, 96, 8, 9)]


@pytest.mark.parametrize("L,nlon,m,state", CASES)
def test_fields_of_one_order(L, nlon, m, state):
    from paper_1009_3308_gb300 import Plan
    plan = Plan(L, nlon // 2, nlon, 0.0, 0.0)
    spec = _spectra(L, nlon, state)
    a = np.zeros(plan.n_coeff, np.complex128)
    for l, v in spec.items():
        a[_off(L, m) + l - max(m, 1)] = v
    _, s, _, T = _table(plan, m)
    lo, n = max(m, 1), L + 2 - m
    b = np.zeros((3, n), LD)     # coefficient sets of zeta, u_theta, u_phi per degree K = m + row
    S = np.zeros((3, n), LD)     # magnitudes
    for l, v in spec.items():
        lam = LD(l) * (l + 1)
        b[0, l - m] = np.sqrt(lam) * LD(v)
        b[1, l - m] = LD(v) / np.sqrt(lam)
        up, dn = l * _eps(l + 1, m) / np.sqrt(lam) * LD(v), -(l + 1) * _eps(l, m) / np.sqrt(lam) * LD(v)
        b[2, l + 1 - m] += up
        S[2, l + 1 - m] += abs(up)
        if l - 1 >= m:
            b[2, l - 1 - m] += dn
            S[2, l - 1 - m] += abs(dn)
    S[:2] = np.abs(b[:2])
    scale = [np.ones_like(s, LD), m / s.astype(LD), 1 / s.astype(LD)]
    c, sn = _circle(m, nlon)
    two = 1 if m == 0 else 2
    got = [g.cpu().numpy() for g in plan.grid_fields(_dev(a))]
    for f in range(3):
        g = (b[f] @ T) * scale[f]
        # zeta: g e^{i m phi}; u_theta: i g e^{i m phi}; u_phi: -g e^{i m phi}, real parts
        ref = two * (np.outer(g, c) if f == 0 else np.outer(g, -sn) if f == 1 else np.outer(-g, c))
        tol = TOL * two * float(((S[f] @ np.abs(T)) * scale[f]).max())
        err = float(np.abs(got[f].astype(LD) - ref).max())
        assert err <= tol, (f, err / tol)


@pytest.mark.parametrize("L,nlon,m,row", [(511, 1536, 5, 0), (255, 768, 5, 0), (100, 324, 5, 1), (255, 768, 0, 97),
                                          (100, 324, 3, 161), (53, 162, 4, 0), (31, 96, 5, 0)])
def test_projection_of_one_ring(L, nlon, m, row):
    from paper_1009_3308_gb300 import Plan
    plan = Plan(L, nlon // 2, nlon, 0.0, 0.0)
    phi = 2 * np.pi * np.arange(nlon) / nlon
    v = np.zeros((2, plan.nlat, nlon))
    v[0, row], v[1, row] = 1.3 * np.cos(m * phi), 0.7 * np.cos(m * phi)
    x, s, w, T = _table(plan, m)
    # the order's Fourier coefficients of the two rows
    c, sn = _circle(m, nlon)
    q = 2 * PI / nlon * LD(w[row]) / LD(s[row])
    Gt, Gp = (q * ((v[k, row] * c).sum() - 1j * (v[k, row] * sn).sum()) for k in (0, 1))
    lo = max(m, 1)
    l = np.arange(lo, L + 1)
    isl = 1 / np.sqrt(l.astype(LD) * (l + 1))
    P = T[:, row]
    up, dn = l * _eps(l + 1, m) * P[l + 1 - m], np.where(l > m, (l + 1) * _eps(l, m) * P[np.maximum(l - 1 - m, 0)], 0)
    ref = isl * (-1j * m * P[l - m] * Gt - (up - dn) * Gp)
    S = isl * (m * abs(P[l - m]) * abs(Gt) + (abs(up) + abs(dn)) * abs(Gp))
    out = plan.project(_dev(v[0]), _dev(v[1])).cpu().numpy()
    got = out[_off(L, m): _off(L, m) + l.size]
    assert float(np.abs(got - ref).max()) <= TOL * float(S.max())
