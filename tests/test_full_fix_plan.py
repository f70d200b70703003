"""How the FP64 full estimate's tensor-core recursion is cut into CTAs and launches
(csrc/full_fix_plan.h), compiled for the host: every tile once, rounds counted with the
device's own number of SMs, sums within the room a shift has, scratch within the integer
form's or one round's."""
import ctypes as C
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2007_15195_gb300", "csrc")

SHIM = r"""
#include "full_fix_plan.h"
extern "C" void plan(long long D, long long N, int S, int sms, long long* out) {
    const vk::FullFixPlan p = vk::full_fix_plan(D, N, S, sms);
    out[0] = p.halves; out[1] = p.per_shift; out[2] = p.ctas; out[3] = p.launch;
    out[4] = (long long)p.tables; out[5] = (long long)p.history; out[6] = (long long)vk::full_integer_bytes(D, N, S);
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, so = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)], check=True)
    L = C.CDLL(str(so))

    def f(D, N, S, sms):
        out = (C.c_longlong * 7)()
        L.plan(C.c_longlong(D), C.c_longlong(N), S, sms, out)
        return list(out)
    return f


def _ceil(a, b):
    return -(-a // b)


@pytest.mark.parametrize("sms", [1, 96, 132, 148, 152, 160])
@pytest.mark.parametrize("D", [64, 97, 1021, 2500, 10000, 32768])
def test_plan(plan, D, sms):
    for N in (1, 63, 128, 129, 257, 1000, 2000, 4096, 65536, 2 ** 31 - 1):
        for S in (2, 5, 12, 16, 64):
            halves, per_shift, ctas, launch, tables, history, integer = plan(D, N, S, sms)
            assert per_shift == _ceil(N, 128 * halves) and ctas == S * per_shift
            assert per_shift * halves <= max(1, _ceil(N, 64))  # sums a shift
            r1, r2 = _ceil(S * _ceil(N, 128), sms), _ceil(S * _ceil(N, 256), sms)
            assert halves == (2 if N > 128 and 10 * r1 >= 19 * r2 else 1)
            cta = halves * _ceil(D, 32) * 65536
            assert launch == ctas or (launch % sms == 0 and launch <= 4 * sms)
            assert history == launch * cta
            assert tables + history <= max(integer, tables + sms * cta)


def test_sm_count_decides_the_rounds(plan):
    """150 tiles: two rounds of 148 SMs, one of 152."""
    assert plan(500, 128 * 75, 2, 148)[0] == 2
    assert plan(500, 128 * 75, 2, 152)[0] == 1
