"""The FP64 path's partials against the oracle as closely as the oracle's own FP64
rounding allows, on blocks that do not amplify it: 64-bit fixed point on the device loses
nothing that FP64 keeps."""
import numpy as np
import pytest

import oracle as O
from paper_2007_15195_gb300 import binding as B
from paper_2007_15195_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 5, 12, 20, 31])
@pytest.mark.parametrize("N,S", [(97, 3), (256, 4)])
def test_partials(m, N, S):
    """A mean of m + 1 products and a division, each rounded at 2^-53 of at most 5 (|y| and
    |z| below 5, |L| <= 1), moves Phi(z) by at most |z| + 1 < 6 times that, and the
    quantile passes it on to the later variables at a weight below 1/2 (weakly
    correlated sites): below 60 (m + 2) 2^-53 a factor, m + 1 factors."""
    D = m + 25
    s = inputs.uniform_sites(D, 700 + m)
    u = inputs.rng(m, 3).normal(0.3, 0.7, size=D)
    nbr = O.neighbors(s, m)
    cov = (0, 1.0, 0.05, 0.5, 0.0)
    with B.Context(0) as ctx:
        _, _, _, num, den = B.vecchia_log_cdf_terms(ctx, s, nbr, m, cov, u, N, S, 11, B.FP64)
    onum, oden = O.vecchia_partials(s, nbr, m, cov, u, N, S, 11)
    tol = 60 * (m + 2) * (m + 1) * 2.0 ** -53
    assert np.all(np.abs(num / onum - 1) < tol) and np.all(np.abs(den / oden - 1) < tol)
