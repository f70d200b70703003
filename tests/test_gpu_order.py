"""Device orderings against the host's (bit-exact): the maxmin rounds at the
sizes where their launch changes (serial picks only, one CTA, clusters,
grid-wide rounds; sort tiles and merges), on spreads that make long chains of
dependent picks, ties, duplicates and crowded cells; the XY sort beyond the
counting kernel's range."""
import numpy as np
import pytest

from paper_2007_15195_gb300 import binding as B
from paper_2007_15195_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch  # noqa: F401
    c = B.Context(0)
    yield c
    c.close()


def _equal(ctx, s, kind):
    import torch
    s = np.ascontiguousarray(s)
    got = B.vecchia_order(ctx, torch.from_numpy(s).cuda(), kind).cpu().numpy()
    assert np.array_equal(got, B.vecchia_order(None, s, kind))


@pytest.mark.parametrize("D", [1, 2, 31, 32, 33, 1023, 2048, 2049, 4096, 4097, 5999, 6000, 8193, 12289])
def test_maxmin_sizes(ctx, D):
    _equal(ctx, inputs.uniform_sites(D, D), "maxmin")


def _spreads():
    r = np.random.default_rng(0)
    line = np.stack([np.arange(1500.0), np.zeros(1500)], 1)
    grow = np.stack([np.cumsum(1.002 ** np.arange(1500)), np.zeros(1500)], 1)
    crowd = np.concatenate([inputs.uniform_sites(7000, 5) * 1e-3, [[1e3, 1e3], [-5e2, 3.0]]])
    return {"grid": inputs.grid_sites(79), "line": line, "growing gaps": grow, "crowded": crowd,
            "duplicates": np.repeat(inputs.uniform_sites(1300, 3), 5, axis=0), "one point": np.zeros((2500, 2)),
            "heavy tails": r.normal(size=(3000, 2)) ** 3}


@pytest.mark.parametrize("name", sorted(_spreads()))
def test_maxmin_spreads(ctx, name):
    _equal(ctx, _spreads()[name], "maxmin")


@pytest.mark.parametrize("D", [8192, 8193, 20000])
def test_xy_sizes(ctx, D):
    s = inputs.uniform_sites(D, D)
    s[::3, 0] = np.round(s[::3, 0], 2)  # equal x: ordered by y, then index
    s[::9] = s[0]
    _equal(ctx, s, "xy")
    _equal(ctx, -s, "xy")
