"""vecchia_log_cdf_unordered in XY order at the sizes of its one-launch form (up to 512
sites: box, order, gather and quantised coordinates in one CTA) and just beyond,
against the four calls and the host's order: partial warps, one site, ties,
duplicates, all sites equal, conditioning sets above 32."""
import numpy as np
import pytest

from paper_2007_15195_gb300 import binding as B
from paper_2007_15195_gb300 import inputs

pytestmark = pytest.mark.gpu

COV = (0, 1.0, 0.3, 0.5, 0.05)  # a nugget: equal sites are not singular


@pytest.fixture(scope="module")
def ctx():
    import torch  # noqa: F401
    c = B.Context(0)
    yield c
    c.close()


def _sites(D, what):
    s = inputs.uniform_sites(D, 600 + D)
    if what == "ties":
        s = np.round(s, 1)  # equal x, and duplicates
    elif what == "equal":
        s[:] = s[0]
    elif what == "signs":
        s = np.where(s < 0.3, -0.0, s - 0.5)
    return s


@pytest.mark.parametrize("D", [1, 2, 31, 32, 33, 100, 511, 512, 513])
@pytest.mark.parametrize("what", ["uniform", "ties", "equal", "signs"])
def test_equals_the_four_calls(ctx, D, what):
    import torch
    s = _sites(D, what)
    u = inputs.rng(D, 2).normal(0.4, 0.3, size=D)
    order = B.vecchia_order(None, s, "xy")
    so, uo = np.ascontiguousarray(s[order]), np.ascontiguousarray(u[order])
    for m, prec in ((0, B.MIXED), (10, B.MIXED), (40, B.MIXED), (7, B.FP64)):
        nbr = B.vecchia_neighbors(ctx, so, m) if m else None
        ref = B.vecchia_log_cdf(ctx, so, nbr, m, COV, uo, 128, 3, 9, prec)
        for dev in (False, True):
            a, b = (torch.from_numpy(s).cuda(), torch.from_numpy(u).cuda()) if dev else (s, u)
            perm = np.full(D, -1, np.int32)
            got = B.vecchia_log_cdf_unordered(ctx, a, b, m, COV, 128, 3, 9, prec, order="xy", perm_out=perm)
            assert np.array_equal(perm, order)
            assert got == ref
