"""The second-order matrix functions of the FP64 observation-space analysis
(numpy restatement) against eigendecompositions: what they neglect is third
order in the off-diagonal part that the eigensolve leaves."""
import numpy as np
import pytest


def _second_order(a, s, O, t):
    """h(S) t and g(S) for S = diag(s) + O: h = (aI + S)^{-1},
    g = ((aI + S)^{-1/2} - a^{-1/2} I) S^{-1}."""
    r = np.sqrt(a)
    u = np.sqrt(a + s)
    h0 = 1.0 / (a + s)
    w = h0 * t
    w1 = h0 * (O @ w)
    h = w - w1 + h0 * (O @ w1)
    den = u[:, None] + u[None, :]
    X1 = O / den
    P = O + r * X1 - r * (X1 @ X1) / den
    al = 1.0 / (u * (u + r))
    APA = al[:, None] * P * al[None, :]
    return h, -(np.diag(al) - APA + APA @ (P * al[None, :])) / r


@pytest.mark.parametrize("n", [2, 7, 28, 64])
@pytest.mark.parametrize("top", [0.01, 1.0, 100.0])
@pytest.mark.parametrize("off", [1e-6, 1e-4, 1e-3])
def test_error_is_third_order(n, top, off):
    rng = np.random.default_rng(n)
    a = 60.0
    s = a * top * rng.random(n)
    O = np.triu(rng.choice([-1.0, 1.0], (n, n)), 1) * off * a
    O = O + O.T
    t = rng.standard_normal(n)
    h, g = _second_order(a, s, O, t)
    lam, V = np.linalg.eigh(np.diag(s) + O)
    h_ref = V @ ((V.T @ t) / (a + lam))
    # g without the cancellation in ((a + x)^{-1/2} - a^{-1/2}) / x.
    ur = np.sqrt(a + lam)
    g_ref = -(V / (ur * (ur + np.sqrt(a)))) @ V.T / np.sqrt(a)
    o = np.linalg.norm(O, 2) / a
    # With |X1| <= o r / 2, |X2| <= o^2 r / 8 and |alpha P| <= 3 o / 4 the first
    # neglected terms are below o^3 of the leading ones; 1e-14 for rounding.
    bound = o ** 3 / (1 - o) + 1e-14
    assert np.linalg.norm(h - h_ref) <= bound * np.linalg.norm(t) / a
    assert np.linalg.norm(g - g_ref, 2) <= bound / (2 * a ** 1.5)
