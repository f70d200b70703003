// exact_math.h -- correctly rounded square root and quotients of doubles by
// integer arithmetic, for the pivot chain of a Cholesky factor.
//
// A column of the factor waits for piv = sqrt(s) and then x / piv.  On GB300
// each is a chain of dependent FP64 instructions at about 80 cycles apiece
// (1.7 us the two together); the same values come from a 64-bit reciprocal square
// root (one Newton-Raphson step of third order from the FP32 approximation,
// on integers), a candidate rounded to 53 bits and the exact remainder that
// tells whether it is the nearest double: about 100 integer instructions.  The
// results equal IEEE's bit for bit (round to nearest, even ties cannot occur for
// either operation at normal results); operands outside 2^-500 .. 2^500, zeros
// and specials go to the FP64 operations.  Compiles for the host too (tests).
#pragma once

#include <math.h>
#include <stdint.h>

#include "special_fix.h"

namespace vk {
namespace exact {

VK_FIX_FN uint64_t to_u64(double x) {
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    union { double d; uint64_t u; } v;
    v.d = x;
    return v.u;
#endif
}
VK_FIX_FN double to_f64(uint64_t u) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    union { double d; uint64_t u; } v;
    v.u = u;
    return v.d;
#endif
}
#ifndef VK_APPROX_TEST
#define VK_APPROX_TEST(y) (y)  // (tests scale the host's approximations by their largest error)
#endif
VK_FIX_FN float rcp_f32(float x) {  // within 2^-21 relative
#ifdef __CUDA_ARCH__
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
#else
    return VK_APPROX_TEST(1.0f / x);
#endif
}
VK_FIX_FN float rsqrt_f32(float x) {  // within 2^-21 relative
#ifdef __CUDA_ARCH__
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
#else
    return VK_APPROX_TEST(1.0f / sqrtf(x));
#endif
}

constexpr uint64_t kMant = (1ull << 52) - 1;

VK_FIX_FN bool mid_range(int biased) { return biased >= 523 && biased <= 1523; }

// A pivot and what its quotients need: piv = P 2^(e - 1075), V = 2^62 / (P 2^-53).
struct Pivot {
    double piv;
    uint64_t P, V;
    int e;  // biased exponent; 0: quotients by the FP64 division
};

// piv = sqrt(s), s > 0.
VK_FIX_FN Pivot pivot(double s) {
    Pivot r;
    const uint64_t b = to_u64(s);
    const int eb = (int)(b >> 52);
    if (!mid_range(eb)) {
        r.piv = sqrt(s);
        r.P = r.V = 0;
        r.e = 0;
        return r;
    }
    // s = M 2^(E - 52), E even, M in [2^52, 2^54): sqrt(s) = sqrt(M 2^52) 2^(E/2 - 52)
    const int odd = (eb + 1) & 1;  // E = eb - 1023 odd
    const uint64_t M = ((b & kMant) | (1ull << 52)) << odd;
    const int half = (eb - 1023 - odd) / 2;
    // x = M 2^-54 in [1/4, 1); y ~ 1 / sqrt(x), Q2.30
    const uint64_t X = M << 10;
    const float yf = rsqrt_f32((float)(uint32_t)(X >> 40) * 0x1p-24f);
    const uint32_t Y0 = (uint32_t)(yf * 0x1p30f);
    // t = 1 - x y^2 (Q60, |t| < 2^-19), y (1 + t/2 + 3 t^2/8)
    const int64_t T = (int64_t)((1ull << 60) - fix::umul_hi(X, (uint64_t)Y0 * Y0));
    const int64_t U = (T >> 1) + (int64_t)((uint64_t)(3 * (T >> 12) * (T >> 12)) >> 39);
    const int64_t Y1s = (int64_t)((uint64_t)Y0 << 32) + (((int64_t)Y0 * (U >> 16)) >> 12) +
                        (int64_t)(((uint64_t)Y0 * (uint64_t)(U & 0xffff)) >> 28);
    const uint64_t Y1 = (uint64_t)Y1s;  // Q62
    // sqrt(x) = x y, Q62; R = sqrt(x) 2^53, rounded to nearest by its remainder
    const uint64_t S = fix::umul_hi(X, Y1);
    uint64_t R = (S + 256) >> 9;
    const int64_t rem = (int64_t)((M << 52) - R * R);
    if (rem > (int64_t)R)
        ++R;
    else if (rem <= -(int64_t)R)
        --R;
    r.piv = to_f64(((uint64_t)(half + 1023) << 52) + (R - (1ull << 52)));
    r.e = half + 1023;
    if (R >> 53) {  // rounded up to 2^53
        r.P = 1ull << 52;
        r.V = 1ull << 63;
        ++r.e;
    } else {
        r.P = R;
        // 1 / (R 2^-53) = y (1 + t), t = 1 - R 2^-53 y (below 2^-52)
        const int64_t t = (int64_t)((1ull << 62) - fix::umul_hi(R << 11, Y1));
        r.V = Y1 + (uint64_t)(((int64_t)(Y1 >> 32) * t) >> 30);
    }
    return r;
}

// The pivot given itself (piv > 0).
VK_FIX_FN Pivot pivot_of(double piv) {
    Pivot r;
    const uint64_t b = to_u64(piv);
    r.piv = piv;
    r.e = (int)(b >> 52);
    r.P = (b & kMant) | (1ull << 52);
    if (!mid_range(r.e)) r.e = 0;
    // d = P 2^-53 in [1/2, 1); v ~ 1/d, Q2.30; t = 1 - d v (|t| < 2^-19), v (1 + t + t^2)
    const float vf = rcp_f32((float)(uint32_t)(r.P >> 29) * 0x1p-24f);
    const uint32_t v0 = (uint32_t)(vf * 0x1p30f);
    const int64_t t = (int64_t)((1ull << 62) - fix::umul_hi(r.P << 11, (uint64_t)v0 << 32));  // Q62
    const int64_t u = t + (((t >> 14) * (t >> 14)) >> 34);
    r.V = ((uint64_t)v0 << 32) + (uint64_t)((((int64_t)v0 * (u >> 16)) >> 14) +
                                            (int64_t)(((uint64_t)v0 * (uint64_t)(u & 0xffff)) >> 30));
    return r;
}

// x / piv.
VK_FIX_FN double quotient(double x, const Pivot& p) {
    const uint64_t b = to_u64(x);
    const int eb = (int)((b >> 52) & 0x7ff);
    if (p.e == 0 || !mid_range(eb)) return x / p.piv;
    uint64_t A = (b & kMant) | (1ull << 52);
    const int less = A < p.P ? 1 : 0;
    A <<= less;  // A / P in [1, 2)
    const uint64_t W = fix::umul_hi(A << 10, p.V);  // Q62 of half of it
    uint64_t q = (W + 256) >> 9;
    const int64_t rem = (int64_t)((A << 52) - q * p.P);
    if (2 * rem > (int64_t)p.P)
        ++q;
    else if (2 * rem < -(int64_t)p.P)
        --q;
    return to_f64((b & (1ull << 63)) | (((uint64_t)(eb - p.e - less + 1023) << 52) + (q - (1ull << 52))));
}

}  // namespace exact
}  // namespace vk
