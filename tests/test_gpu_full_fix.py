"""The FP64 full D-dimensional estimate in 64-bit fixed point against the oracle:
sizes about the panel (32), the tensor-core path's first size and its groups of
128 history variables, ragged point tiles, thresholds beyond the step's tables."""
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


def _check(ctx, s, cov, u, N, S, seed):
    olp, ose = O.full_genz(s, cov, u, N, S, seed)
    if not np.isfinite(olp):  # every product below the double range: reported as such
        with pytest.raises(B.VecchiaError) as e:
            B.vecchia_full_genz(ctx, s, cov, u, N, S, seed, B.FP64)
        assert e.value.status == B.ERR_NONFINITE
        return
    lp, se = B.vecchia_full_genz(ctx, s, cov, u, N, S, seed, B.FP64)
    # the log of a mean whose relative error is 1e-10, and a spread that cancels to ~se
    assert abs(lp - olp) <= 1e-10 * max(1.0, abs(olp))
    assert abs(se - ose) <= 1e-8 * ose


@pytest.mark.parametrize("D,N", [(1, 64), (31, 63), (32, 64), (33, 65), (97, 130), (127, 128), (128, 127), (129, 129),
                                 (160, 200), (161, 40), (257, 300), (289, 129), (420, 257)])
def test_sizes(ctx, D, N):
    s = inputs.uniform_sites(D, 200 + D)
    u = inputs.rng(D, 1).normal(0.6, 0.4, size=D)
    _check(ctx, s, (0, 1.2, 0.2, 0.5, 0.0), u, N, 3, D)


@pytest.mark.parametrize("D,deep", [(60, 31), (200, 31), (200, 101)])
def test_threshold_ranges(ctx, D, deep):
    s = inputs.uniform_sites(D, 300 + D)
    u = inputs.rng(D, 1).normal(0.8, 0.4, size=D)
    u[::7] = 12.0
    u[3::deep] = -7.5
    u[5::41] = 1e300
    _check(ctx, s, (1, 1.0, 0.15, 1.5, 0.0), u, 140, 4, 9)


@pytest.mark.parametrize("D,N", [(64, 257), (97, 385), (129, 300), (289, 257)])
def test_two_tiles_a_cta(ctx, D, N):
    """64 shifts of a few tiles: more tiles than SMs, so a CTA takes two, the second
    of a shift partly or wholly beyond its points."""
    s = inputs.uniform_sites(D, 400 + D)
    u = inputs.rng(D, 1).normal(0.7, 0.4, size=D)
    _check(ctx, s, (0, 1.1, 0.2, 0.5, 0.0), u, N, 64, D + 1)


def test_scratch_limit(ctx):
    """With room for the integer form's history (2.1 GB) but not for the tensor-core
    form's (4.3 GB), the call takes the integer form."""
    import torch
    D, N, S = 1024, 4096, 64
    s = inputs.uniform_sites(D, 77)
    u = inputs.rng(D, 1).normal(0.6, 0.4, size=D)
    cov = (0, 1.0, 0.2, 0.5, 0.0)
    c = B.Context(0)
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (13 << 28), dtype=torch.uint8, device="cuda")
    try:
        few = B.vecchia_full_genz(c, s, cov, u, N, S, 5, B.FP64)
    finally:
        c.close()
        del hold
        torch.cuda.empty_cache()
    full = B.vecchia_full_genz(ctx, s, cov, u, N, S, 5, B.FP64)
    assert abs(few[0] - full[0]) <= 1e-10 * max(1.0, abs(full[0]))
    assert abs(few[1] - full[1]) <= 1e-8 * full[1]
