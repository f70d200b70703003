"""Phi as the fixed-point step takes it (csrc/special_fix.h, phi_of), compiled for the
host: both signs over the whole range, above all where the tail lies below 2^-64, so
that its shift reaches the width of a word."""
import ctypes as C
import os
import random
import subprocess

import pytest

mp = pytest.importorskip("mpmath")

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2007_15195_gb300", "csrc")

SHIM = r"""
#include "special_fix.h"
using namespace vk::fix;
extern "C" int phi(long long hi, long long lim, int shift, unsigned long long* E, unsigned long long* mt, int* et) {
    FixProb e;
    const bool deep = phi_of(kTailRow, kTailMeta, hi, lim, shift, e, kMid);
    *E = e.E;
    *mt = e.mt;
    *et = e.et;
    return deep;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("phi")
    src, so = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)], check=True)
    return C.CDLL(str(so))


@pytest.mark.parametrize("shift", [4, 10])
def test_phi(lib, shift):
    """E within 2 units of 2^-64 and the tail's error (2^-55 relative below 4, 2^-51.5
    below 7, 2^-49 above; nothing of it is left beyond 9.25); the tail itself beside it."""
    mp.mp.dps = 40
    rng = random.Random(7)
    lim = 37 << (56 - shift)
    zs = [0.0, 6.999, 7.0, 8.99, 9.05, 9.08, 9.09, 9.1, 9.2, 9.249, 9.26, 30.0]
    zs += [rng.uniform(0, 9.3) for _ in range(300)] + [rng.uniform(9.05, 9.25) for _ in range(100)]
    for z in zs:
        for sign in (1, -1):
            hi = sign * int(z * 2.0 ** (58 - shift))
            E, mt, et = C.c_ulonglong(), C.c_ulonglong(), C.c_int()
            deep = lib.phi(C.c_longlong(hi), C.c_longlong(lim), shift, C.byref(E), C.byref(mt), C.byref(et))
            a = mp.mpf(abs(hi)) * mp.mpf(2) ** (shift - 58)
            assert deep == (hi < 0 and a >= 7)
            if deep:
                continue
            t = mp.erfc(a / mp.sqrt(2)) / 2
            rel = mp.mpf(2) ** (-55 if a < 4 else -51.5 if a < 7 else -49)
            ref = t if hi < 0 else 1 - t
            assert abs(mp.mpf(E.value) - ref * 2 ** 64) <= 2 + t * rel * 2 ** 64, (z, sign)
            if a < 9.25:
                assert abs(mp.mpf(mt.value) * mp.mpf(2) ** (-64 - et.value) / t - 1) < rel
            else:
                assert mt.value == 0
