"""Device orderings, neighbour rows and calls on coordinates that the bounding box does
not bound (NaN beside a wide axis, infinities, extents whose scale overflows): cell
indices stay in the grid, the covariance reports such a site, the context goes on."""
import numpy as np
import pytest

from paper_2007_15195_gb300 import binding as B
from paper_2007_15195_gb300 import inputs

pytestmark = pytest.mark.gpu

COV = (0, 1.0, 0.3, 0.5, 0.0)


@pytest.fixture(scope="module")
def ctx():
    import torch  # noqa: F401
    c = B.Context(0)
    yield c
    c.close()


def _sites(D, what):
    s = inputs.uniform_sites(D, D)
    if what == "nan":
        s[:, 0] *= 100.0
        s[::7, 0] = np.nan
        s[3, 1] = -np.nan
    elif what == "inf":
        s[5, 0], s[9, 1] = np.inf, -np.inf
    else:
        s *= 1e-305
    return s


@pytest.mark.parametrize("what", ["nan", "inf", "tiny"])
@pytest.mark.parametrize("D", [20, 512, 600, 7000, 9000])
def test_orders_rows_and_calls(ctx, D, what):
    import torch
    s = _sites(D, what)
    sd = torch.from_numpy(s).cuda()
    for kind in ("xy", "maxmin"):
        p = B.vecchia_order(ctx, sd, kind).cpu().numpy()
        assert np.array_equal(np.sort(p), np.arange(D))
        if what == "tiny":
            assert np.array_equal(p, B.vecchia_order(None, s, kind))
    for m in (4, 40):
        nbr = B.vecchia_neighbors(ctx, sd, m).cpu().numpy()
        for i in (0, 1, 5, 19, D // 2, D - 1):
            q = min(m, i)
            assert np.all(np.diff(nbr[i, :q]) > 0) and np.all((nbr[i, :q] >= 0) & (nbr[i, :q] < i))
            assert np.all(nbr[i, q:] == -1)
    if what != "tiny":
        u = torch.zeros(D, dtype=torch.float64, device="cuda")
        for kind in ("xy", "maxmin", "identity"):
            with pytest.raises(B.VecchiaError) as e:
                B.vecchia_log_cdf_unordered(ctx, sd, u, 4, COV, 64, 2, order=kind)
            assert e.value.status in (B.ERR_NOT_PD, B.ERR_NONFINITE)
    ok = inputs.uniform_sites(50, 1)
    assert np.isfinite(B.vecchia_log_cdf_unordered(ctx, ok, np.zeros(50), 4, COV, 64, 2)[0])
