"""Accuracy of the FP64 path's products of probabilities on the device: independent
variables, whose joint CDF is a product of Phi, at thresholds where the first
probabilities are small."""
import math

import numpy as np
import pytest

from paper_2007_15195_gb300 import binding as B

pytestmark = pytest.mark.gpu

COV = (0, 1.0, 1e-3, 0.5, 0.0)  # sites a unit apart: exp(-1000) is 0, every L is the identity


@pytest.fixture(scope="module")
def ctx():
    import torch  # noqa: F401
    c = B.Context(0)
    yield c
    c.close()


def _line(D):
    return np.stack([np.arange(float(D)), np.zeros(D)], 1)


def _phi(z):
    return 0.5 * math.erfc(-z * math.sqrt(0.5))


def test_pairs(ctx):
    """Phi(u_0) Phi(u_1).  The reference's argument z sqrt(1/2) has two roundings
    (2^-53 each), which Phi(z) takes up to z^2 + 1 < 13 times, and erfc's own ulp: below
    4e-15 a factor; the step's Phi is within 2^-51.5 (5e-16 in all)."""
    v = [-3.45, -3.4, -3.29, -3.25, -3.2, -3.0, -2.5, -1.5, -0.5, 0.4, 2.0]
    u = np.array([x for a in v for b in v for x in (a, b)])
    nbr = np.maximum(np.arange(len(u)) - 1, 0).astype(np.int32)[:, None]
    nbr[0] = -1
    _, _, _, num, den = B.vecchia_log_cdf_terms(ctx, _line(len(u)), nbr, 1, COV, u, 64, 2, 1, B.FP64)
    for i in range(1, len(u)):
        ref = _phi(u[i - 1]) * _phi(u[i])
        assert np.all(np.abs(num[i] / ref - 1) < 1e-14), (u[i - 1], u[i])
        assert np.all(np.abs(den[i] / _phi(u[i - 1]) - 1) < 1e-14)


@pytest.mark.parametrize("D", [2, 40, 70])
@pytest.mark.parametrize("z", [-3.29, -3.0, -1.0])
def test_full(ctx, D, z):
    """Both forms of the full recursion: two deep thresholds, the others at 3, whose
    factors are within 2^-53 or so of their values (70 of them: 1e-14)."""
    u = np.full(D, 3.0)
    u[:2] = z
    lp, _ = B.vecchia_full_genz(ctx, _line(D), COV, u, 64, 2, 1, B.FP64)
    ref = 2 * math.log(_phi(z)) + (D - 2) * math.log1p(-_phi(-3.0))
    assert abs(lp - ref) < 5e-14
