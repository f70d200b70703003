"""Neighbour rows against the oracle where cells are crowded or empty: the rule that
searches a crowded cell by itself, both list lengths (m <= 32, above), sites about
one another and duplicates; groups too."""
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


def _spread(name, D):
    r = np.random.default_rng(3)
    if name == "line":
        return np.stack([r.permutation(D) * 1.0, np.zeros(D)], 1)
    if name == "clusters":
        return r.random((9, 2))[r.integers(0, 9, D)] + r.normal(size=(D, 2)) * 0.004
    if name == "crowd":
        s = inputs.uniform_sites(D, 5) * 1e-3
        s[::500] = r.random((len(s[::500]), 2)) * 100
        return s
    if name == "duplicates":
        return np.repeat(inputs.uniform_sites(D // 30, 3), 30, axis=0)[r.permutation(D // 30 * 30)]
    return r.normal(size=(D, 2)) ** 3


@pytest.mark.parametrize("name", ["line", "clusters", "crowd", "duplicates", "heavy tails"])
@pytest.mark.parametrize("m", [1, 20, 32, 33, 63])
def test_rows(ctx, name, m):
    s = np.ascontiguousarray(_spread(name, 2400))
    assert np.array_equal(B.vecchia_neighbors(ctx, s, m), O.neighbors(s, m))


@pytest.mark.parametrize("name", ["line", "crowd"])
def test_groups(ctx, name):
    s = np.ascontiguousarray(_spread(name, 1500))
    cond, count = B.vecchia_group_conditioning(ctx, s, 4, 6)
    ocond, ocount = O.group_cond_nearest(s, 4, 6, 24)
    assert np.array_equal(cond, ocond) and np.array_equal(count, ocount)
