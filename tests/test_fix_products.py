"""The running product of the fixed-point step (csrc/special_fix.h), compiled for
the host, against exact values: no bits lost whatever the size of the first
probabilities."""
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
extern "C" void product(const unsigned long long* mt, const int* et, const int* neg, unsigned long long* m, int* ex) {
    FixProb p[2];
    for (int i = 0; i < 2; ++i) {
        const uint64_t T = shr64(mt[i], et[i]);
        p[i].mt = mt[i];
        p[i].et = et[i];
        p[i].E = neg[i] ? T : ~T;
    }
    const FixFloat f = times(prob(p[0]), p[1]);
    *m = f.m;
    *ex = f.ex;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("prod")
    src, so = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)], check=True)
    return C.CDLL(str(so))


def test_products_of_probabilities(lib):
    """e_0 e_1 of tails from 2^-1 to 2^-70 and of their complements: both
    mantissas are at least 2^62, so the product's high half is at least 2^60 and
    within 2 of it (2^-59); E = 1 - t is cut at 2^-64 of at least 1/2 on either
    side (2^-62 together).  Every result is normalised."""
    mp.mp.dps = 40
    rng = random.Random(5)
    for k in range(5000):
        et = [1 + k % 70, rng.randint(1, 70)] if k % 3 else [1 + k % 70] * 2
        mt = [rng.getrandbits(63) | 1 << 63, rng.getrandbits(63) | 1 << 63]
        neg = [rng.randint(0, 1), rng.randint(0, 1)]
        m, ex = C.c_ulonglong(), C.c_int()
        lib.product((C.c_ulonglong * 2)(*mt), (C.c_int * 2)(*et), (C.c_int * 2)(*neg), C.byref(m), C.byref(ex))
        ref = mp.mpf(1)
        for i in range(2):
            t = mp.mpf(mt[i]) * mp.mpf(2) ** (-64 - et[i])
            ref *= t if neg[i] else 1 - t
        got = mp.mpf(m.value) * mp.mpf(2) ** (-64 - ex.value)
        assert m.value >> 62 and abs(got / ref - 1) < mp.mpf(2) ** -58
