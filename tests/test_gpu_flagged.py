"""Terms of the log-space form in the shapes that their number and N pick (16 or 8 warps a
term, 4 from 609 terms on): against FP64 where few and many terms are flagged, and bit for
bit alone and in a batch, where the other problem's flagged terms change the shape."""
import numpy as np
import pytest

from paper_2007_15195_gb300 import binding as B
from paper_2007_15195_gb300 import inputs

from _prep import mixed_tol

pytestmark = pytest.mark.gpu

COV = (0, 1.0, 0.2, 0.5, 0.0)


@pytest.fixture(scope="module")
def ctx():
    import torch  # noqa: F401
    c = B.Context(0)
    yield c
    c.close()


def _problem(ctx, D, m, N, S, deep, seed):
    import torch
    s = torch.from_numpy(inputs.uniform_sites(D, seed)).cuda()
    u = inputs.rng(seed, 1).normal(0.5, 0.3, size=D)
    so, uo = B.vecchia_apply_order(ctx, B.vecchia_order(ctx, s, "xy"), s, torch.from_numpy(u).cuda())
    uo[:deep] -= 11.0
    return dict(sites=so, nbr=B.vecchia_neighbors(ctx, so, m), m=m, cov=COV, u=uo, N=N, S=S, seed=seed)


def _alone(ctx, p, prec=B.MIXED):
    return B.vecchia_log_cdf(ctx, p["sites"], p["nbr"], p["m"], p["cov"], p["u"], p["N"], p["S"], p["seed"], prec)


@pytest.mark.parametrize("m,N,S", [(8, 100, 3), (20, 512, 5), (31, 600, 4), (12, 4096, 2), (40, 300, 3)])
@pytest.mark.parametrize("deep", [5, 700, 900])
def test_against_fp64(ctx, m, N, S, deep):
    p = _problem(ctx, 900, m, N, S, deep, 31 + m)
    ref, got = _alone(ctx, p, B.FP64), _alone(ctx, p)
    assert abs(got[0] - ref[0]) <= mixed_tol(ref[0])


@pytest.mark.parametrize("N", [100, 1024])
def test_alone_and_in_a_batch(ctx, N):
    few, many = _problem(ctx, 200, 10, N, 4, 20, 41), _problem(ctx, 900, 10, N, 4, 900, 42)
    lp, se, st = B.vecchia_log_cdf_batch(ctx, [few, many], B.MIXED)
    assert (lp[0], se[0]) == _alone(ctx, few) and (lp[1], se[1]) == _alone(ctx, many)
