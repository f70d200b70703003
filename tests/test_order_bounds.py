"""Host orderings of coordinates that the bounding box does not bound: NaN beside a
wide axis, extents whose scale overflows.  Every result is a permutation, and
non-finite values do not reach the heap (each case in a process of its own)."""
import subprocess
import sys

import pytest

CODE = r"""
import sys
import numpy as np
sys.path.insert(0, %r)
from paper_2007_15195_gb300 import binding as B
D, kind, what = int(sys.argv[1]), sys.argv[2], sys.argv[3]
s = np.random.default_rng(D).random((D, 2))
if what == "nan":
    s[:, 0] *= 100.0
    s[::7, 0] = np.nan
    s[3, 1] = -np.nan
elif what == "inf":
    s[5, 0], s[9, 1] = np.inf, -np.inf
else:
    s *= 1e-305
p = B.vecchia_order(None, s, kind)
assert np.array_equal(np.sort(p), np.arange(D)), what
if what == "tiny" and kind == "xy":
    assert np.array_equal(p, np.lexsort((s[:, 1], s[:, 0])))
"""


@pytest.mark.parametrize("what", ["nan", "inf", "tiny"])
@pytest.mark.parametrize("kind", ["xy", "maxmin"])
@pytest.mark.parametrize("D", [20, 600])
def test_host_orders(D, kind, what):
    import os
    from paper_2007_15195_gb300 import build
    build.build()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CODE % root, str(D), kind, what], capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr[-500:]
