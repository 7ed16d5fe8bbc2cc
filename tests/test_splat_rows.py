"""The splat's moment form at every number of rows a bin (sigma from 0.25 bins
up): the truncation of its Taylor polynomials about a row's centre, six terms
of the forward and eight of the adjoint with their derivative, against the
remainders' bounds; the sizes of the tables; and the rules between moments and
taps."""
import math

import numpy as np
import pytest
from numpy.polynomial.hermite_e import hermeval

from tests import rules_lib

# the ends of each range of rows a bin: 16, 8, 4, 2 and 1
SIGMAS = [0.25, 0.3, 0.390, 0.391, 0.5, 0.781, 0.782, 1.1, 1.562, 1.563, 2.0, 2.499, 2.5, 3.2, 9.8]


@pytest.fixture(scope="module")
def rules():
    return rules_lib.load()


def _derivative(x, sigma, n):
    """phi^(n)(x) in units of phi(0) / sigma^n."""
    he = np.zeros(n + 1)
    he[n] = 1.0
    return (-1) ** n * hermeval(x / sigma, he) * np.exp(-0.5 * (x / sigma) ** 2)


def _errors(sigma, q, terms):
    """Largest error of the polynomial and of its derivative over all rows, relative to
    phi(0) and to phi(0) / sigma."""
    reach = math.ceil(6 * sigma) + 1
    x = 0.5 - (np.arange((2 * reach + 1) * q)[:, None] - reach * q + 0.5) / q  # the rows' centres
    h = np.linspace(-0.5, 0.5, 101)[None, :] / q / sigma  # offsets in units of sigma
    d = [_derivative(x, sigma, n) / math.factorial(n) for n in range(terms)]
    value = sum(d[n] * h ** n for n in range(terms))
    slope = sum(n * d[n] * h ** (n - 1) for n in range(1, terms))
    at = x + h * sigma
    return (np.abs(value - _derivative(at, sigma, 0)).max(), np.abs(slope - _derivative(at, sigma, 1)).max())


@pytest.mark.parametrize("sigma", SIGMAS)
def test_truncation_within_the_remainder(rules, sigma):
    q = rules.rows_per_bin(sigma)
    half = 0.5 / q / sigma
    assert half <= (0.2 if sigma >= 2.5 else 0.16) * (1 + 1e-12)
    # max |He_n(t) exp(-t^2 / 2)| of an even n is (n - 1)!! at t = 0
    six, eight = 15.0, 105.0
    value, _ = _errors(sigma, q, 6)
    assert value <= six / math.factorial(6) * half ** 6 * (1 + 1e-6) + 1e-14
    assert value <= (1.34e-6 if sigma >= 2.5 else 3.5e-7)
    value, slope = _errors(sigma, q, 8)
    assert value <= eight / math.factorial(8) * half ** 8 * (1 + 1e-6) + 1e-14
    assert slope <= eight / math.factorial(7) * half ** 7 * (1 + 1e-6) + 1e-14


def test_tables_hold_every_width(rules):
    for sigma in np.concatenate([np.linspace(0.25, 2.6, 4701), np.linspace(2.6, 9.9, 731)]):
        if not rules.fits(sigma):
            assert sigma > 9.8
            continue
        j = math.ceil(6 * sigma) + 1
        assert j <= rules.max_j() and (2 * j + 1) * rules.rows_per_bin(sigma) <= rules.max_taps()


def test_forms_by_width_points_and_bins(rules):
    big = 1 << 31
    for sigma, q in [(0.25, 16), (0.39, 16), (0.4, 8), (0.78, 8), (0.79, 4), (1.56, 4), (1.57, 2), (2.5, 1)]:
        assert rules.rows_per_bin(sigma) == q
        # the forward takes no more than four rows a bin, however many points
        assert rules.forward_mom(sigma, big, 1) == (q <= 4)
        assert rules.forward_mom(sigma, 1, 65536) == (q <= 2)
        assert rules.adjoint_mom(sigma, big, 1) == 1
        assert rules.adjoint_mom(sigma, 1, 65536) == (q <= 2)
    assert not rules.forward_mom(9.9, big, 1) and not rules.adjoint_mom(9.9, big, 1)
    # widths near 1.6 and 3.2 bins (30 and 60 ps jitter at 8 ps bins) at any size
    for sigma in (1.6, 3.2):
        for P, B in ((1000, 1024), (16384, 512), (65536, 512)):
            assert rules.forward_mom(sigma, P, B) and rules.adjoint_mom(sigma, P, B)
