"""The bounded device waits of the FP64 recursion on the tensor cores: a wait made to run
out without any fault (a short limit and a copy lane that issues nothing, so that the
accumulators' barrier is one that nothing completes, with nothing in flight) is reported
as VECCHIA_ERR_TIMEOUT with one and with two tiles a CTA, and the next call on the
context equals the oracle.  The mixed precision's limit does not reach it."""
import numpy as np
import pytest

import oracle as O
from paper_2007_15195_gb300 import binding as B
from paper_2007_15195_gb300 import inputs

pytestmark = pytest.mark.gpu

COV = (0, 1.1, 0.2, 0.5, 0.0)


def _inputs(D):
    return inputs.uniform_sites(D, 500 + D), inputs.rng(D, 1).normal(0.7, 0.4, size=D)


@pytest.mark.parametrize("D,N,S", [(64, 200, 4), (200, 512, 4), (97, 257, 64)])
def test_wait_runs_out_and_context_recovers(D, N, S):
    s, u = _inputs(D)
    olp, ose = O.full_genz(s, COV, u, N, S, 5)
    with B.Context(0) as ctx:
        for _ in range(2):
            B.vecchia_set_full_genz_wait(ctx, limit_ns=1_000_000, withhold=2)
            with pytest.raises(B.VecchiaError) as e:
                B.vecchia_full_genz(ctx, s, COV, u, N, S, 5, B.FP64)
            assert e.value.status == B.ERR_TIMEOUT
            B.vecchia_set_full_genz_wait(ctx, 0, False)
            lp, se = B.vecchia_full_genz(ctx, s, COV, u, N, S, 5, B.FP64)
            assert abs(lp - olp) <= 1e-10 * abs(olp) and abs(se - ose) <= 1e-8 * ose


def test_mixed_limit_does_not_reach_it():
    """A limit that no wait of a kernel that does work can keep to."""
    D, N, S = 300, 1000, 4
    s, u = _inputs(D)
    with B.Context(0) as ctx:
        ref = B.vecchia_full_genz(ctx, s, COV, u, N, S, 5, B.FP64)
        for withhold in (False, True):
            B.vecchia_set_full_genz_wait(ctx, limit_ns=1, withhold=withhold)
            assert B.vecchia_full_genz(ctx, s, COV, u, N, S, 5, B.FP64) == ref
