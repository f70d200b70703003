"""The FP64 path's 64-bit fixed-point step against the oracle: every bucket's
edge sizes, thresholds in each range of the step (beyond z = 9.25, far beyond,
below z = -7 and below the quantile's table) and nearly singular blocks."""
import numpy as np
import pytest

import oracle as O
from paper_2007_15195_gb300 import binding as B
from paper_2007_15195_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch  # noqa: F401
    c = B.Context(0)
    yield c
    c.close()


def _check(ctx, s, u, m, cov, N, S, seed, rel=1e-10):
    nbr = O.neighbors(s, m)
    lp, se, terms, num, den = B.vecchia_log_cdf_terms(ctx, s, nbr, m, cov, u, N, S, seed, B.FP64)
    onum, oden = O.vecchia_partials(s, nbr, m, cov, u, N, S, seed)
    # products rather than quotients: partials far below the double range are 0 on both sides
    assert np.all(np.abs(num - onum) <= rel * onum)
    assert np.all(np.abs(den - oden) <= rel * oden)


@pytest.mark.parametrize("m", [1, 2, 8, 9, 12, 13, 16, 17, 20, 21, 24, 28, 31, 32, 47, 48, 63])
def test_bucket_edges(ctx, m):
    s = inputs.uniform_sites(m + 5, 100 + m)
    u = inputs.rng(m, 1).normal(0.3, 0.5, size=m + 5)
    _check(ctx, s, u, m, (0, 1.3, 0.3, 0.5, 0.0), 97, 3 + m % 9, m)


@pytest.mark.parametrize("u0", [-12.0, -7.0, -4.0, 6.9, 9.0, 9.3, 30.0, 1e300])
def test_threshold_ranges(ctx, u0):
    """Every third threshold at u0 (standard deviations), the rest ordinary."""
    D, m = 40, 10
    s = inputs.uniform_sites(D, 7)
    u = inputs.rng(8, 1).normal(0.3, 0.5, size=D)
    u[::3] = u0
    _check(ctx, s, u, m, (1, 1.0, 0.2, 1.5, 0.0), 256, 4, 5)


@pytest.mark.parametrize("gap,rel", [(1e-3, 1e-10), (1e-6, 1e-8)])
def test_nearly_duplicate_sites(ctx, gap, rel):
    """Pairs of sites a tiny distance apart: 1/L_vv up to ~1/sqrt(2 gap / range),
    so rounding of the conditional mean grows by that factor on both sides."""
    D, m = 40, 12
    s = inputs.uniform_sites(D, 9)
    s[1::2] = s[::2] + gap
    u = np.repeat(inputs.rng(9, 1).normal(0.5, 0.4, size=D // 2), 2)
    _check(ctx, s, u, m, (0, 1.0, 0.5, 0.5, 0.0), 128, 4, 6, rel)


def test_singular_block_is_reported(ctx):
    s = inputs.uniform_sites(12, 10)
    s[7] = s[3]
    with pytest.raises(B.VecchiaError) as e:
        B.vecchia_log_cdf(ctx, s, O.neighbors(s, 5), 5, (0, 1.0, 0.3, 0.5, 0.0), np.zeros(12), 64, 2, 1, B.FP64)
    assert e.value.status == B.ERR_NOT_PD
