"""The Givens step of a Hessenberg column by a prefix sum with products of the
rotations, written out in numpy as the kernel forms it (per lane a range of
rotations, a scan over 32 lanes), against the rotations applied one by one.

Every term of the sum is at most |h| in magnitude and the products carry one
rounding per rotation, so the two agree within about 10 j rounding errors of
|h|: 10 * 200 * 1.1e-16 = 2e-13, taken as 1e-12; also while the residual
(the product of the |s_i|) falls to 1e-13."""
import numpy as np
import pytest


def _step(j, h, hn, cs, sn, pp, pq, ip):
    per = (j + 31) // 32
    L = np.zeros(32, complex)
    rng = [(min(j, l * per), min(j, min(j, l * per) + per)) for l in range(32)]
    for l, (b, e) in enumerate(rng):
        for i in range(b, e):
            L[l] += pq[i] * h[i + 1]
    d = 1
    while d < 32:
        L[d:] = L[d:] + L[:-d].copy()
        d *= 2
    r = np.zeros(j + 1, complex)
    a = pp[j] * (h[0] + L[31])
    for l, (b, e) in enumerate(rng):
        S = h[0] + (L[l - 1] if l else 0)
        for i in range(b, e):
            r[i] = cs[i] * pp[i] * S + sn[i] * h[i + 1]
            S = S + pq[i] * h[i + 1]
    n2a, d2 = abs(a) ** 2, abs(a) ** 2 + hn * hn
    f = 1 / np.sqrt(n2a) / np.sqrt(d2)
    c, s = n2a * f, a * hn * f
    r[j] = c * a + s * hn
    ipn = ip * -s * d2 / hn / hn
    return r, c, s, -np.conj(s) * pp[j], ipn


@pytest.mark.parametrize("m,fall", [(1, 0.5), (31, 0.6), (33, 0.4), (64, 0.63), (200, 0.86)])
def test_prefix_sum_of_products_equals_the_rotations(m, fall):
    rng = np.random.default_rng(m)
    cs, sn, pp, pq, ip = np.zeros(m), np.zeros(m, complex), np.ones(m + 1, complex), np.zeros(m, complex), 1 + 0j
    for j in range(m):
        h = rng.standard_normal(j + 1) + 1j * rng.standard_normal(j + 1)
        a = h[0]
        ref = np.zeros(j + 1, complex)
        for i in range(j):
            ref[i] = cs[i] * a + sn[i] * h[i + 1]
            a = -np.conj(sn[i]) * a + cs[i] * h[i + 1]
        hn = abs(a) * fall / np.sqrt(1 - fall * fall)     # |s_j| = fall
        ref[j] = np.sqrt(abs(a) ** 2 + hn * hn) * a / abs(a)
        r, cs[j], sn[j], pp[j + 1], ip = _step(j, h, hn, cs, sn, pp, pq, ip)
        pq[j] = cs[j] * ip
        assert np.abs(r - ref).max() <= 1e-12 * np.abs(h).max()
    assert abs(np.prod(np.abs(sn)) - fall ** m) <= 1e-11 * fall ** m
    assert np.prod(np.abs(sn)) >= 1e-14
