"""The 64-bit fixed-point normal tail and quantile of the FP64 path
(csrc/special_fix.h): its integer code compiled for the host, against mpmath
at interval edges, binade edges and random points, and the products' rounding
against exact integers."""
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
extern "C" {
long long q_fix(unsigned long long m, int lz) { Digits X; const int r = quant_row(m, lz, X); return poly(kQuantRow[r], X, kQShift3, kMid); }
void t_fix(unsigned long long A, unsigned long long* mt, int* et) { uint64_t m; tail_poly(kTailRow, kTailMeta, A, m, *et, kMid); *mt = m; }
long long muladd(long long a, long long b, long long c) { return mul_add(digits(a), digits(b), c - kMulBias, kMid); }
void smalls(unsigned long long W, unsigned long long mt, int et, int neg, int lower, unsigned long long* m, int* lz) {
    FixProb p; p.mt = mt; p.et = et; p.E = neg ? shr64(mt, et) : ~shr64(mt, et); small_s(W, p, lower != 0, *(uint64_t*)m, *lz); }
unsigned long long bits_of(unsigned long long m, int ex) { return to_bits(FixFloat{m, ex}); }
void of_bits(unsigned long long b, unsigned long long* m, int* ex) { const FixFloat f = from_bits(b); *m = f.m; *ex = f.ex; }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fix")
    src, so = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)], check=True)
    L = C.CDLL(str(so))
    L.q_fix.restype = L.muladd.restype = C.c_longlong
    L.bits_of.restype = C.c_ulonglong
    L.q_fix.argtypes = [C.c_ulonglong, C.c_int]
    L.muladd.argtypes = [C.c_longlong] * 3
    L.bits_of.argtypes = [C.c_ulonglong, C.c_int]
    return L


def _pair(fn, *args):
    m, e = C.c_ulonglong(), C.c_int()
    fn(*args, C.byref(m), C.byref(e))
    return m.value, e.value


def test_quantile(lib):
    mp.mp.dps = 40
    rng = random.Random(1)
    pts = [(m, lz) for lz in (1, 2, 5, 10, 11, 20, 31)
           for m in (1 << 63, (1 << 63) + 1, (1 << 64) - 1, (1 << 63) + (7 << 58), (1 << 63) + (7 << 58) - 1)]
    pts += [(rng.getrandbits(63) | 1 << 63, rng.randint(1, 31)) for _ in range(150)]
    worst = 0
    for m, lz in pts:
        s = mp.mpf(m) * mp.mpf(2) ** (-64 - lz)
        y = mp.sqrt(2) * mp.erfinv(1 - 2 * s)
        worst = max(worst, abs(mp.mpf(lib.q_fix(C.c_ulonglong(m), lz)) * mp.mpf(2) ** -57 - y))
    # the table's own bound (integer evaluation against 40 digits at nine points
    # an interval) is 2^-56.3; rounding of other offsets adds below 2^-57
    assert worst < mp.mpf(2) ** -55.5


def test_tail(lib):
    # the 32-bit coefficients' unit grows with the fourth derivative (a^4 / 24):
    # 2^-52.5 at a = 4, 2^-46 at a = 7, times x^4 <= 2^-8 and the polynomial's three roundings
    mp.mp.dps = 40
    rng = random.Random(2)
    As = [0, 1, (1 << 52) - 1, 1 << 52, (7 << 58) - 1, (37 << 56) - 1] + [rng.randrange(37 << 56) for _ in range(200)]
    for A in As:
        mt, et = C.c_ulonglong(), C.c_int()
        lib.t_fix(C.c_ulonglong(A), C.byref(mt), C.byref(et))
        a = mp.mpf(A) * mp.mpf(2) ** -58
        ref = mp.erfc(a / mp.sqrt(2)) / 2
        rel = abs(mp.mpf(mt.value) * mp.mpf(2) ** (-64 - et.value) / ref - 1)
        assert mt.value >> 62 and rel < mp.mpf(2) ** (-55 if a < 4 else -51.5 if a < 7 else -49)


def test_products(lib):
    rng = random.Random(3)
    edge = [0, 1, -1, (1 << 31) - 1, 1 << 31, -(1 << 31), (1 << 32) - 1, (1 << 62) - 1, -(1 << 62)]
    for k in range(2000):
        a = rng.choice(edge) if k % 4 == 0 else rng.randrange(-(1 << 62), 1 << 62)
        b = rng.choice(edge) if k % 5 == 0 else rng.randrange(-(1 << 62), 1 << 62)
        got = lib.muladd(a, b, 17)
        # |exact / 2^64 - got| <= 1/2 (rounding) + 1/4 (the dropped low product)
        assert abs((got - 17) * (1 << 64) - a * b) <= 3 << 62


def test_small_arguments_keep_their_relative_accuracy(lib):
    mp.mp.dps = 40
    rng = random.Random(4)
    for k in range(600):
        et = rng.randint(2, 60)
        mt = rng.getrandbits(62) | 3 << 62
        t = mp.mpf(mt) * mp.mpf(2) ** (-64 - et)
        if k % 2:  # (1 - w) + w t with w near 1
            W = (1 << 64) - rng.randrange(1, 1 << rng.randint(1, 52))
            if et < 12:
                continue
            w = mp.mpf(W) * mp.mpf(2) ** -64
            m, lz = C.c_ulonglong(), C.c_int()
            lib.smalls(C.c_ulonglong(W), C.c_ulonglong(mt), et, 0, 0, C.byref(m), C.byref(lz))
            ref = (1 - w) + w * t
        else:  # w t
            W = rng.randrange(1, 1 << rng.randint(1, 64))
            w = mp.mpf(W) * mp.mpf(2) ** -64
            m, lz = C.c_ulonglong(), C.c_int()
            lib.smalls(C.c_ulonglong(W), C.c_ulonglong(mt), et, 1, 1, C.byref(m), C.byref(lz))
            ref = w * t
        got = mp.mpf(m.value) * mp.mpf(2) ** (-64 - lz.value)
        assert m.value >> 63 and abs(got / ref - 1) < mp.mpf(2) ** -59


def test_doubles_round_trip(lib):
    import struct
    for v in (0.0, 0.5, 0.1, 1.0 - 2.0 ** -53, 2.0 ** -1022, 5e-324, 3e-310, 1e-300):
        b = struct.unpack("<Q", struct.pack("<d", v))[0]
        m, ex = C.c_ulonglong(), C.c_int()
        lib.of_bits(C.c_ulonglong(b), C.byref(m), C.byref(ex))
        assert lib.bits_of(m.value, ex.value) == b
