// fix_step.cuh -- the pieces of the 64-bit fixed-point step (special_fix.h)
// that the FP64 kernels share: a row's scale, the quantile of a lattice
// coordinate and Phi of a conditional mean.
#pragma once

#include "special_f64.h"
#include "special_fix.h"

namespace vk {

// What a variable's conditional mean needs to become z: with 1/L_vv =
// rdiag 2^(shift - e - 62) (see fix_scale), z 2^58 = hi(rdiag acc) << shift;
// lim is that product's value at |z| = 9.25.
struct FixVar {
    fix::Digits rdiag;
    int64_t lim;
    int shift;
    int kL;      // scale of the row's coefficients: integers of 2^-kL
    int64_t up;  // u_v as an integer of 2^(7 - kL), less the products' biases
};

// The scale of row v.  With B above |u_v| + 38.6 sum_t |L_vt| (|y| < 38.6: the
// quantile is clamped at 2^-1000) and 2^e <= B < 2^(e + 1), L_vt is kept as an
// integer of 2^-kL, kL = 67 - e (|L_vt| < B / 38.6: below 2^63), and sums as
// integers of 2^(7 - kL) (below 2^61).  u_v is clamped where Phi is 0 or 1
// whatever the y_t (NaN as +inf, as the FP64 functions took it).
__device__ __forceinline__ FixVar fix_scale(double lvv, double sum, double uv, int products) {
    const double rd = 1.0 / lvv;
    const double reach = 38.6 * sum, umax = reach + 39.0 * lvv;
    const double u = fmax(-umax, fmin(umax, uv));
    const double B = fmax(fabs(u) + reach, 32.0 * lvv);
    const int e = ilogb(B);
    const long long rb = __double_as_longlong(rd);
    const int S = (int)((rb >> 52) & 0x7ff) - 1023 + e;
    FixVar r;
    r.kL = 67 - e;
    r.up = __double2ll_rn(ldexp(u, r.kL - 7)) - products * fix::kMulBias;
    r.rdiag = fix::digits(((rb & 0xfffffffffffffll) | (1ll << 52)) << 10);
    r.lim = S <= 56 ? 37ll << (56 - S) : S < 62 ? (37 + (1 << (S - 56)) - 1) >> (S - 56) : 1;
    r.shift = S;
    return r;
}

// -L as digits of the row's scale.
__device__ __forceinline__ fix::Digits fix_coef(double l, int kL) {
    return fix::digits(__double2ll_rn(ldexp(-l, kL)));
}

// 2^64 g / N rounded to the nearest integer (g < N < 2^32), by two steps of
// long division.
__device__ __forceinline__ uint64_t fix64_ratio(uint32_t g, uint64_t N) {
    const uint64_t a = ((uint64_t)g << 32), q1 = a / N, r1 = a % N;
    const uint64_t b = r1 << 32, q2 = b / N, r2 = b % N;
    return (q1 << 32) + q2 + ((2 * r2 >= N) ? 1u : 0u);
}

// A 53-bit shift Delta = M 2^-53 in 64-bit fixed point (exact).
__device__ __forceinline__ uint64_t fix_shift(double delta) {
    return (uint64_t)__double2ull_rn(delta * 9007199254740992.0) << 11;
}

__device__ __forceinline__ void load_fix_tables(fix::FixTables& tb) {
    for (int i = threadIdx.x; i < fix::kQShared * fix::kQSub; i += blockDim.x) tb.quant[i] = fix::kQuantRow[i];
    for (int i = threadIdx.x; i < fix::kTRows; i += blockDim.x) {
        tb.tail[i] = fix::kTailRow[i];
        tb.meta[i] = fix::kTailMeta[i];
    }
}

// |Phi^{-1}(s)| 2^57 of s = m 2^-64 2^-lz below 2^-32 (one step in 2^31 unless
// the thresholds themselves are that deep): the FP64 quantile.
__device__ __forceinline__ int64_t quantile_tail(uint64_t m, int lz) {
    const double s = __longlong_as_double((long long)fix::to_bits(fix::FixFloat{m, lz}));
    const double y = special64::phiinv_pq(special64::global_tables(), s, 1.0);
    return __double2ll_rn(-y * 0x1p57);
}

// Phi at z = hi 2^(shift - 58) <= -7: the FP64 tail.
__device__ __forceinline__ void deep_prob(int64_t hi, int shift, fix::FixProb& p) {
    double unused;
    const double z = ldexp((double)hi, shift - 58);
    const double t = special64::tail<false>(special64::global_tables(), -z, unused);
    p = fix::prob_of((uint64_t)__double_as_longlong(t), true);
}

// Digits of y 2^57, y = Phi^{-1}(w e) at the lattice coordinate X 2^-64.
__device__ __forceinline__ fix::Digits fix_quantile(const fix::FixTables& tb, uint64_t lattice, const fix::FixProb& e,
                                                    uint64_t K) {
    const uint64_t w = fix::tent(lattice);
    const uint64_t pp = fix::umul_hi(w, e.E);
    const int64_t upper = (int64_t)pp >> 63;  // all ones where 1 - w e is the smaller
    const uint64_t s = pp ^ (uint64_t)upper;
    int lz = fix::clz32((uint32_t)(s >> 32));
    uint64_t m = s << lz;
    fix::Digits X;
    const int row = fix::quant_row(m, min(lz, fix::kQShared), X);
    int64_t y = fix::poly(tb.quant[row], X, fix::kQShift3, K);
    if (lz > fix::kQShared) {
        fix::small_s(w, e, upper == 0, m, lz);
        if (lz <= 31) {
            const int far = fix::quant_row(m, lz, X);
            y = fix::poly(fix::kQuantRow[far], X, fix::kQShift3, K);
        } else
            y = quantile_tail(m, lz);
    }
    return fix::digits((y ^ ~upper) - ~upper);
}

// Phi of the conditional mean whose product with rdiag is hi.
__device__ __forceinline__ void fix_phi(const fix::FixTables& tb, int64_t hi, int64_t lim, int shift, fix::FixProb& e,
                                        uint64_t K) {
    if (fix::phi_of(tb.tail, tb.meta, hi, lim, shift, e, K)) deep_prob(hi, shift, e);
}

}  // namespace vk
