"""Tables of the 64-bit fixed-point normal tail and quantile (special_fix.h).

Writes special_fix.cuh next to this script.  Both functions are piecewise
degree-7 polynomials in x, the offset from an interval's centre in units of
twice its width (|x| <= 1/4), coefficients as integers:

  * quantile |Phi^{-1}(s)|, s in [2^-32, 1/2): the binade lz = 1..31 of s
    (s = m 2^-(lz+1), m in [1, 2)), 32 intervals of m a binade, unit 2^-57;
  * tail Phi(-a) 2^e, a in [0, 9.25): 592 intervals of width 1/64, unit 2^-62,
    e the interval's exponent (the largest value in [1/2, 1)).

c0 .. c3 are 64-bit integers of the table's unit; c4 .. c7 are 32-bit integers
of unit 2^-hs (what they add is below 2^-19 of the value, so 32 bits reach
2^-58; c0 .. c2 are written minus 2^31, which the evaluation's products add), hs the same for every quantile row and per row of the tail (its
fourth derivative grows like a^4): shift3 = hs + 32 - unit takes their
partial result, times x, to the 64-bit unit.  Polynomials are Chebyshev fits
(mpmath, 40 digits).  Run:  python fit_fixed.py  (prints the worst errors of
the integer evaluation against 40 digits).
"""
import os

import mpmath as mp

HERE = os.path.dirname(os.path.abspath(__file__))
OUT = os.path.join(HERE, "special_fix.cuh")
mp.mp.dps = 40

DEG = 7
Q_UNIT, T_UNIT = 57, 62
Q_BINADES, Q_SUB = 31, 32
T_SUB, T_ROWS = 64, 592


def tail(a):
    return mp.erfc(a / mp.sqrt(2)) / 2


def quantile(s, guess):
    """a > 0 with Phi(-a) = s, by Newton's method on log Phi."""
    a = guess
    for _ in range(50):
        t = tail(a)
        step = (t / s - 1) * s / (mp.exp(-a * a / 2) / mp.sqrt(2 * mp.pi))
        # a third-order correction keeps the number of iterations small
        a2 = a + step * (1 + a * step / 2)
        if abs(a2 - a) < mp.mpf(10) ** -36:
            return a2
        a = a2
    raise RuntimeError("no convergence at %s" % s)


def quantile_on(centre, scale):
    """x -> |Phi^{-1}| on the interval of the mantissa's centre, each call started from the centre's value."""
    s0 = centre * scale
    if s0 > mp.mpf("0.2"):
        start = (mp.mpf(1) / 2 - s0) * mp.sqrt(2 * mp.pi)
    else:
        t = mp.sqrt(-2 * mp.log(s0))
        start = t - mp.log(t * mp.sqrt(2 * mp.pi)) / t
    y0 = quantile(s0, start)
    return lambda x: quantile((centre + x * 2 / Q_SUB) * scale, y0)


def chebyshev(f, deg):
    """Coefficients in x (ascending) of the Chebyshev interpolant of f on [-1/4, 1/4]."""
    n = deg + 1
    nodes = [mp.cos(mp.pi * (2 * k + 1) / (2 * n)) for k in range(n)]
    vals = [f(z / 4) for z in nodes]
    c = [2 * sum(vals[k] * mp.cos(j * mp.pi * (2 * k + 1) / (2 * n)) for k in range(n)) / n for j in range(n)]
    c[0] /= 2
    # sum_j c_j T_j(z), z = 4 x, into monomials
    T = [[mp.mpf(1)], [mp.mpf(0), mp.mpf(1)]]
    for j in range(2, n):
        p = [mp.mpf(0)] + [2 * v for v in T[-1]]
        for i, v in enumerate(T[-2]):
            p[i] -= v
        T.append(p)
    out = [mp.mpf(0)] * n
    for j in range(n):
        for i, v in enumerate(T[j]):
            out[i] += c[j] * v
    return [out[i] * mp.mpf(4) ** i for i in range(n)]


def rounded(coef, unit, hs):
    c = [int(mp.nint(v * mp.mpf(2) ** (unit if k < 4 else hs))) for k, v in enumerate(coef)]
    assert all(abs(v) < 2 ** 62 for v in c[:4]) and sum(abs(v) >> 2 * k for k, v in enumerate(c[4:])) < 2 ** 31 - 8, c
    return c


def largest_hs(coefs):
    """hs for which c4 + c5 x + c6 x^2 + c7 x^3 stays below 2^31 for every |x| <= 1/4."""
    top = max(sum(abs(v) / 4 ** k for k, v in enumerate(c[4:])) for c in coefs)
    return int(mp.floor(mp.mpf("30.9999") - mp.log(top, 2)))


def wrap32(v):
    return ((v + 2 ** 31) % 2 ** 32) - 2 ** 31


def evaluate(c, X, sh3):
    """The integer evaluation of special_fix.h for X = x 2^64."""
    Xl = wrap32(X)
    Xh = (X - Xl) >> 32
    H = c[7]
    for k in (6, 5, 4):
        H = c[k] + ((H * Xh) >> 32)
    P = c[3] + ((H * Xh) >> sh3)
    for k in (2, 1, 0):
        Pl = wrap32(P)
        Ph = (P - Pl) >> 32
        P = c[k] + Ph * Xh + ((Ph * Xl + Pl * Xh + 2 ** 31) >> 32)
    return P


def check(c, f, unit, sh3, n=9):
    worst = mp.mpf(0)
    for k in range(n):
        X = int(-(2 ** 62) + (2 ** 63 - 1) * k // (n - 1)) + (k % 2) * 12345
        X = max(-(2 ** 62), min(2 ** 62 - 1, X))
        v = mp.mpf(evaluate(c, X, sh3)) / mp.mpf(2) ** unit
        worst = max(worst, abs(v - f(mp.mpf(X) / mp.mpf(2) ** 64)))
    return worst


def main():
    # quantile rows
    qf = []
    for lz in range(1, Q_BINADES + 1):
        for j in range(Q_SUB):
            centre = 1 + (mp.mpf(j) + mp.mpf(1) / 2) / Q_SUB
            f = quantile_on(centre, mp.mpf(2) ** -(lz + 1))
            qf.append((f, chebyshev(f, DEG)))
    qhs = largest_hs([c for _, c in qf])
    qsh = qhs + 32 - Q_UNIT
    qrows = [rounded(c, Q_UNIT, qhs) for _, c in qf]
    qerr = max(check(r, f, Q_UNIT, qsh) for r, (f, _) in zip(qrows, qf))
    print("quantile: hs %d, shift %d, worst absolute error %s (2^%.2f)" % (qhs, qsh, mp.nstr(qerr, 3), mp.log(qerr, 2)))
    # tail rows
    trows, tmeta, terr = [], [], mp.mpf(0)
    for i in range(T_ROWS):
        lo = mp.mpf(i) / T_SUB
        e = int(mp.floor(-mp.log(tail(lo), 2)))
        if tail(lo) * mp.mpf(2) ** e >= 1:
            e -= 1
        centre = (mp.mpf(i) + mp.mpf(1) / 2) / T_SUB

        def g(x, centre=centre, e=e):
            return tail(centre + x * 2 / T_SUB) * mp.mpf(2) ** e
        c = chebyshev(g, DEG)
        hs = min(largest_hs([c]), 60)
        sh = hs + 32 - T_UNIT
        r = rounded(c, T_UNIT, hs)
        err = check(r, g, T_UNIT, sh) / g(mp.mpf(1) / 4)
        terr = max(terr, err)
        if i % 64 == 0:
            print("tail: a = %s hs %d e %d relative error 2^%.2f" % (mp.nstr(lo, 4), hs, e, mp.log(err, 2)))
        trows.append(r)
        tmeta.append(sh | e << 8)
    print("tail: worst relative error %s (2^%.2f)" % (mp.nstr(terr, 3), mp.log(terr, 2)))

    def emit(rows):
        return ["    {%s}," % ", ".join("%dll" % (v - 2 ** 31 if k < 3 else v) if k < 4 else "%d" % v
                                        for k, v in enumerate(r)) for r in rows]

    L = [
        "// special_fix.cuh -- generated by fit_fixed.py; do not edit by hand.",
        "// Integer polynomial tables of the normal tail and quantile (form, units and",
        "// fitting method described in fit_fixed.py).",
        "#pragma once",
        "",
        "constexpr int kQRows = %d, kQSub = %d, kQUnit = %d, kQShift3 = %d;  // worst absolute error %s"
        % (len(qrows), Q_SUB, Q_UNIT, qsh, mp.nstr(qerr, 3)),
        "constexpr int kTRows = %d, kTSub = %d, kTUnit = %d;  // worst relative error %s"
        % (len(trows), T_SUB, T_UNIT, mp.nstr(terr, 3)),
        "VK_FIX_TABLE FixRow kQuantRow[kQRows] = {", *emit(qrows), "};",
        "VK_FIX_TABLE FixRow kTailRow[kTRows] = {", *emit(trows), "};",
        "// shift3 | e << 8 of each tail row",
        "VK_FIX_TABLE uint16_t kTailMeta[kTRows] = {",
        *["    " + ", ".join("%d" % v for v in tmeta[k:k + 16]) + "," for k in range(0, len(tmeta), 16)],
        "};",
        "",
    ]
    with open(OUT, "w") as f:
        f.write("\n".join(L))
    print("wrote", OUT)


if __name__ == "__main__":
    main()
