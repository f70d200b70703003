"""Device memory that the orderings hold, in bytes a site: the maxmin rounds' sort runs in
the rounds' own arrays, the XY sort of an unordered call in the room of what the call
writes later.  (Neighbour search: 24 bytes a site and up to 13 MB of cells.)"""
import numpy as np
import pytest

from paper_2007_15195_gb300 import binding as B
from paper_2007_15195_gb300 import inputs

pytestmark = pytest.mark.gpu

D = 3_000_000
SLACK = 20 << 20  # cells, alignment, the allocator's granularity
COV = (0, 1.0, 0.01, 0.5, 0.1)


def _held(call):
    """Device memory that a fresh context keeps after the call."""
    import torch
    torch.cuda.synchronize()
    with B.Context(0) as ctx:
        B.vecchia_order(ctx, torch.zeros(600, 2, dtype=torch.float64, device="cuda"), "maxmin")  # modules loaded
        free = torch.cuda.mem_get_info()[0]
        out = call(ctx)
        torch.cuda.synchronize()
        return free - torch.cuda.mem_get_info()[0], out


def test_maxmin():
    import torch
    s = torch.from_numpy(inputs.uniform_sites(D, 1)).cuda()
    torch.empty(D, dtype=torch.int32, device="cuda")  # the allocator's block for the result
    held, perm = _held(lambda ctx: B.vecchia_order(ctx, s, "maxmin"))
    assert held <= 49 * D + SLACK
    assert torch.equal(torch.sort(perm)[0], torch.arange(D, dtype=torch.int32, device="cuda"))


def test_unordered_xy():
    import torch
    m = 1
    s = torch.from_numpy(inputs.uniform_sites(D, 2)).cuda()
    u = torch.zeros(D, dtype=torch.float64, device="cuda")
    with B.Context(0) as ctx:
        so, uo = B.vecchia_apply_order(ctx, B.vecchia_order(ctx, s, "xy"), s, u)
        nbr = B.vecchia_neighbors(ctx, so, m)
    base, ref = _held(lambda ctx: B.vecchia_log_cdf(ctx, so, nbr, m, COV, uo, 32, 2, 1))
    held, got = _held(lambda ctx: B.vecchia_log_cdf_unordered(ctx, s, u, m, COV, 32, 2, 1, order="xy"))
    assert got == ref
    # beside the log-CDF's own: ordering 4, ordered copies 24, rows 4 m, neighbour search 24
    assert held - base <= (4 + 24 + 4 * m + 24) * D + SLACK
