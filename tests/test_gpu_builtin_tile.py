"""The built-in rule's tile as a tile: its launches give the rule's results bit for bit,
and the tuner's default candidates hold it, so that a tuned tile is no slower than none."""
import numpy as np
import pytest

from paper_2007_15195_gb300 import autotune
from paper_2007_15195_gb300 import binding as B
from paper_2007_15195_gb300 import inputs

pytestmark = pytest.mark.gpu

COV = (0, 1.0, 0.2, 0.5, 0.0)


@pytest.fixture(scope="module")
def ctx():
    import torch  # noqa: F401
    c = B.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("prec", [B.FP64, B.MIXED])
@pytest.mark.parametrize("D,m,N,S", [(60, 8, 512, 5), (400, 20, 300, 6), (3000, 10, 256, 9), (300, 40, 256, 7)])
def test_builtin_tile(ctx, prec, D, m, N, S, tmp_path):
    s = inputs.uniform_sites(D, D)
    s = np.ascontiguousarray(s[B.vecchia_order(None, s, "xy")])
    u = inputs.rng(D, 1).normal(0.5, 0.3, size=D)
    nbr = B.vecchia_neighbors(ctx, s, m)
    ref = B.vecchia_log_cdf(ctx, s, nbr, m, COV, u, N, S, 3, prec)
    tile = B.vecchia_builtin_tile(ctx, prec, autotune.bucket_of(m), D, S, N)
    try:
        B.vecchia_set_tile(ctx, prec, -1, *tile)
        assert B.vecchia_log_cdf(ctx, s, nbr, m, COV, u, N, S, 3, prec) == ref
        item = dict(sites=s, nbr=nbr, m=m, cov=COV, u=u, N=N, S=S, seed=3)
        r = autotune.tune(ctx, [item], prec, reps=1, cache_path=str(tmp_path / "t.json"))
        assert tile in [tuple(t) for _, t in r["timings"]] and r["ms"] <= min(ms for ms, t in r["timings"])
    finally:
        B.vecchia_reset_tiles(ctx)
