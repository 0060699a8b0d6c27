"""The polynomial form of the coefficients loses nothing against the Chebyshev expansions.

A plan keeps the first kMono terms of each kCheb-term expansion as a polynomial (plan.cu).
What the dropped terms could add has to stay below what evaluating the kept ones in
64 bits rounds away in the worst case, 2 kMono 2^-53 sum |m_i| for kMono multiply-adds in
Horner's order, both of the largest coefficient (the expansions are no better for the
small ones), for coefficients and derivatives.  J stays at 8: beyond it the sums behind the
tables cancel so far that 80-bit arithmetic does not show the dropped terms.
"""
import os
import re

import numpy as np
import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1710_03197_gb300", "csrc", "plan.cu")
LD = np.longdouble
PI = LD("3.14159265358979323846264338327950288")


def _constant(name):
    return int(re.search(r"constexpr int %s = (\d+);" % name, open(SRC).read()).group(1))


def _tables(N, K, J):
    t = np.arange(N) - N / 2
    q = (2.34 * J) ** 2 - (np.pi * J * t / K) ** 2
    z = np.maximum(np.sqrt(np.abs(q)), 1e-300)
    s = 1 / np.where(q > 0, np.sinh(z) / z, np.sin(z) / z)
    s = s / s.max()
    j = np.arange(1, J + 1)
    G = (np.exp(2j * np.pi / K * (j[:, None] - j)[..., None] * t) * s * s).sum(-1)
    return t, s, np.linalg.inv(G)


def _coefs(delta, N, K, J, deriv):
    t, s, T = _tables(N, K, J)
    theta = 2 * PI / K * ((delta + LD(J) / 2 - 1)[:, None] - np.arange(J).astype(LD))
    ph = theta[..., None] * t.astype(LD)
    w = (s * t if deriv else s).astype(LD)
    c, n = (np.cos(ph) * w).sum(-1), (np.sin(ph) * w).sum(-1)
    re, im = (-n, -c) if deriv else (c, -n)
    Tr, Ti = T.real.astype(LD), T.imag.astype(LD)
    return re @ Tr.T - im @ Ti.T, re @ Ti.T + im @ Tr.T


@pytest.mark.parametrize("deriv", [0, 1])
@pytest.mark.parametrize("J", [1, 2, 4, 6, 7, 8])
@pytest.mark.parametrize("N,K", [(64, 128), (40, 60), (80, 100), (16, 20), (16, 16), (120, 120), (90, 96)])
def test_dropped_terms_are_below_rounding(N, K, J, deriv):
    terms, n = _constant("kCheb"), _constant("kMono")
    m = np.arange(terms).astype(LD)
    x = np.cos(PI * (m + LD(0.5)) / terms)
    cos = np.cos(PI * m[:, None] * (m + LD(0.5)) / terms)
    a = [(np.where(m == 0, LD(1), LD(2)) / terms)[:, None] * (cos @ v) for v in _coefs((x + 1) / 2, N, K, J, deriv)]
    dropped = max(np.abs(part[n:]).sum(0).max() for part in a)
    kept = max(np.abs(np.polynomial.chebyshev.cheb2poly(part[:n, j])).sum() for part in a for j in range(J))
    assert dropped <= 2 * n * LD(2) ** -53 * kept, float(dropped / kept)
