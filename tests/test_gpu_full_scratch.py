"""Device memory that the FP64 full estimate holds: its history within what the integer
form's takes (8 bytes a value), by launches that share it, and results that the launches
do not change."""
import numpy as np
import pytest

import oracle as O
from paper_2007_15195_gb300 import binding as B
from paper_2007_15195_gb300 import inputs

pytestmark = pytest.mark.gpu

COV = (0, 1.0, 0.2, 0.5, 0.0)


def test_history_of_many_tiles():
    import torch
    D, N, S = 512, 4096, 64
    s, u = inputs.uniform_sites(D, 1), inputs.rng(D, 1).normal(0.7, 0.4, size=D)
    sd, ud = torch.from_numpy(s).cuda(), torch.from_numpy(u).cuda()
    with B.Context(0) as ctx:
        B.vecchia_full_genz(ctx, sd[:64], COV, ud[:64], 64, 2, 1, B.FP64)  # modules loaded
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        lp, se = B.vecchia_full_genz(ctx, sd, COV, ud, N, S, 5, B.FP64)
        held = free - torch.cuda.mem_get_info()[0]
        again = B.vecchia_full_genz(ctx, sd, COV, ud, N, S, 5, B.FP64)
    # factor and rows 16 D^2, shifts and sums 12 D S + 8 S N / 64, history 8 D N S
    assert held <= 16 * D * D + 12 * D * S + S * N // 8 + 8 * D * N * S + (8 << 20)
    assert again == (lp, se)


@pytest.mark.parametrize("D,N,S", [(64, 2500, 64), (97, 2048, 33)])
def test_several_launches(D, N, S):
    """More CTAs than four rounds: against the oracle."""
    s, u = inputs.uniform_sites(D, 500 + D), inputs.rng(D, 1).normal(0.7, 0.4, size=D)
    olp, ose = O.full_genz(s, COV, u, N, S, 5)
    with B.Context(0) as ctx:
        lp, se = B.vecchia_full_genz(ctx, s, COV, u, N, S, 5, B.FP64)
    assert abs(lp - olp) <= 1e-10 * abs(olp) and abs(se - ose) <= 1e-8 * ose
