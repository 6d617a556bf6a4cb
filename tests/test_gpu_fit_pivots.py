"""The fit's pivots and quotients, which are formed from reciprocals and corrected by
remainders, against square roots and divisions of 60 digits over a wide range."""
from decimal import Decimal, getcontext

import numpy as np
import pytest

import scenarios as S

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -52
FAR = 1.0e3          # points this many lengthscales apart: their kernel value is zero


def _linv(lib, X, sf2, sn2, ell=1.0):
    h = S.Hyper((ell,) * 4, sf2, sn2)
    g = lib.gp_fit(X, np.zeros((len(X), 2)), (h, S.Hyper((ell,) * 4, sf2, sn2)))
    return np.asarray(lib.gp_factors(g, 0)[0]).reshape(len(X), len(X))


def test_single_pivots(lib):
    """L^-1 = 1 / sqrt(d): the root and the reciprocal each within a unit in the last place."""
    getcontext().prec = 60
    rng = np.random.default_rng(1)
    X = np.zeros((1, 4))
    for e in np.concatenate([rng.uniform(-30.0, 30.0, 200), np.arange(-30.0, 31.0, 10.0)]):
        sf2 = float(10.0 ** e)
        got = _linv(lib, X, sf2, 0.25 * sf2)[0, 0]
        ref = 1 / Decimal(sf2 + 0.25 * sf2).sqrt()
        assert abs(Decimal(float(got)) / ref - 1) <= Decimal(2 * EPS), (sf2, got)


def test_two_points(lib):
    """One quotient by the pivot's root, one difference, one more pivot: twelve roundings
    (the kernel value's exponent has four), magnified by the difference."""
    getcontext().prec = 60
    rng = np.random.default_rng(2)
    for e in rng.uniform(-30.0, 30.0, 100):
        sf2, r = float(10.0 ** e), float(rng.uniform(0.05, 2.0))
        X = np.zeros((2, 4))
        X[1, 0] = r
        got = _linv(lib, X, sf2, 1e-3 * sf2)
        d, k = Decimal(sf2 + 1e-3 * sf2), Decimal(sf2) * (Decimal(r) * Decimal(r) / -2).exp()
        l11 = d.sqrt()
        l21 = k / l11
        l22 = (d - l21 * l21).sqrt()
        for a, b in ((got[0, 0], 1 / l11), (got[1, 1], 1 / l22), (got[1, 0], -l21 / (l11 * l22))):
            assert abs(Decimal(float(a)) / b - 1) <= Decimal(12 * EPS) * d / (l22 * l22), (sf2, r)


@pytest.mark.parametrize("N", [31, 32, 33, 100])
def test_powers_of_four_scale_exactly(lib, N):
    """Every operation commutes with a power of two: 4^k K gives 2^-k L^-1, bit for bit."""
    X = np.random.default_rng(N).random((N, 4))
    ref = _linv(lib, X, 0.1, 1e-3)
    for k in (-40, -7, 1, 12, 40):
        assert np.array_equal(_linv(lib, X, 0.1 * 4.0 ** k, 1e-3 * 4.0 ** k) * 2.0 ** k, ref)


def test_uncorrelated_points(lib):
    """Pivots side by side in a block and past it: a diagonal factor."""
    X = np.zeros((70, 4))
    X[:, 0] = FAR * np.arange(70)
    L = _linv(lib, X, 0.3, 0.02)
    assert np.array_equal(L, np.diag(np.diag(L)))
    assert np.all(np.abs(np.diag(L) * np.sqrt(0.32) - 1.0) <= 4 * EPS)
