// genz.cu -- the fused per-term kernel of the Vecchia log-CDF and the log-sum.
//
// One CTA takes one Vecchia term at a time (a site i of a problem):
//   prologue (FP64, all warps): the block b = (N_i ascending, i) of
//     Sec. 2.2 / Eq. (vecchia-cdf), its covariance from the covariance
//     function (Sec. 3, Sec. 4.1), the Cholesky factor;
//   body (all warps): Genz's separation-of-variables recursion at the
//     shifted lattice points, one lane per point, the numerator (d-dim) and
//     denominator ((d-1)-dim, the leading block) sharing every sample;
//   epilogue: per-shift lattice means num[i,s], den[i,s] in FP64.
// The log-sum kernel then forms each term on the log scale and sums them in a
// fixed order (Sec. 3.1), with the delta-method standard error over shifts.
//
// Genz's recursion for the d-dim CDF at u with Cholesky factor L (variables
// v = 0..d-1, lattice coordinates t = 0..d-2):
//   e_0 = Phi(u_0 / L_00)
//   y_t = Phi^{-1}(w_t e_t),  w_t = tent(x_t) = 1 - |2 x_t - 1|
//   e_{t+1} = Phi((u_{t+1} - sum_{j<=t} L_{t+1,j} y_j) / L_{t+1,t+1})
//   numerator sample = e_0 ... e_{d-1},  denominator sample = e_0 ... e_{d-2}.
// The partial sums u_v - sum_j L_vj y_j of all later variables are kept in
// registers and updated right after each y_t (right-looking), so the loop over
// t runs at run time with a fixed register array per lane.
//
// A term is a block of d variables whose first c are the conditioning set:
// one site i with c = |N_i| (Eq. vecchia-cdf), or a group of p sites with
// its conditioning set (Sec. 3.2).  Its denominator is the c-dim CDF of the
// leading block, i.e. the product e_0 ... e_{c-1} of the same run (1 when
// c = 0); the numerator is the full product.
#include <cfloat>
#include <climits>
#include <map>
#include <mutex>
#include <tuple>

#include "cov.cuh"
#include "exact_math.h"
#include "fix_step.cuh"
#include "special_f32.h"
#include "vk_internal.h"

namespace vk {
namespace {

constexpr int kMaxWarps = 16;
constexpr int kMaxUnits = 64;  // shifts x slices handled by one CTA item

// Entry e of a packed lower triangle (row-major: e = r (r + 1) / 2 + c, c <= r).
__device__ __forceinline__ void tri_index(int e, int& r, int& c) {
    r = (int)((sqrtf((float)(8 * e + 1)) - 1.0f) * 0.5f);
    while ((r + 1) * (r + 2) / 2 <= e) ++r;
    while (r * (r + 1) / 2 > e) --r;
    c = e - r * (r + 1) / 2;
}

// FP64 path, step t: the lattice coordinate's multiplier round(g_t 2^64 / N),
// the coefficient -L_{t+1,t} and what takes variable t + 1 to z (FixVar).
struct __align__(16) FixStep {
    uint64_t G;
    fix::Digits nlz, rdiag;
    int64_t lim;
    int shift, pad[3];
};

// Shared memory of a CTA: this fixed part, then (mixed path) the dynamic
// tail dfix[S][DMAX] (the shifts in 32-bit fixed point) and
// stepw[warps][DMAX] (per warp, the step constants of its current shift).
// FP64: e0, each step's constants and each row's scale kL.
template <int DMAX>
struct FixSmem {
    fix::FixProb p0;
    __align__(16) FixStep step[DMAX];
    int scale[DMAX];
};
struct NoFixSmem {};

template <int DMAX, bool MIXED>
struct GenzSmem : std::conditional<MIXED, NoFixSmem, FixSmem<DMAX>>::type {
    using T = typename std::conditional<MIXED, float, fix::Digits>::type;
    double A[DMAX][DMAX + 1];  // covariance block, overwritten by its Cholesky factor
    double bx[DMAX], by[DMAX], bu[DMAX];
    double diag[DMAX];
    int bidx[DMAX];            // the block's ordered sites
    // Recursion tables, step t (lattice coordinate t, variable t + 1 next):
    //   Lz[t]      = L_{t+1,t}          coefficient of y_t in variable t+1
    //   Lup[t][r]  = L_{t+2+r,t}        coefficients of y_t in the later variables
    // MIXED multiplies each row v by kZs/L_vv (so the conditional mean arrives
    // standardised and times kZs = sqrt(log2(e)/2), the form its Phi takes);
    // FP64 keeps -L as integers of the row's scale (Lup; Lz in step), exact to
    // 2^-60 of the row's largest possible sum, and multiplies the conditional mean
    // by 1/L_vv, one rounding more than the definition's division.
    static constexpr int LS = (DMAX + 3) & ~3;  // row stride: 16-byte aligned rows
    __align__(16) T Lup[DMAX][LS];
    __align__(16) T Lz[MIXED ? DMAX : 1];
    __align__(16) typename std::conditional<MIXED, float, int64_t>::type up[DMAX];  // MIXED: kZs u_v / L_vv
    uint32_t gl[MIXED ? DMAX : 1];  // round(g_t 2^32 / N)
    // (16-byte aligned, e0 and ec0 included: 0.2 to 0.6 % faster than at an odd multiple of 8)
    __align__(16) double part_num[kMaxUnits], part_den[kMaxUnits];
    double e0, ec0;
    float le2_0;  // log2 e0 when e0 < 2^-64 (mixed path)
    int q, c, bad, flag;
};

__host__ __device__ constexpr size_t align16(size_t b) { return (b + 15) & ~(size_t)15; }

// Bytes of shared memory for a CTA of `warps` warps on problems with <= max_S
// shifts: the fixed part, then (mixed) the shifts in fixed point and the
// per-warp step constants, or (FP64) the function tables and each warp's shift.
template <int DMAX, bool MIXED>
constexpr size_t smem_bytes(int max_S, int warps) {
    return align16(sizeof(GenzSmem<DMAX, MIXED>)) +
           (MIXED ? align16((size_t)max_S * DMAX * 4) + (size_t)warps * DMAX * 16
                  : align16(sizeof(fix::FixTables)) + (size_t)warps * DMAX * sizeof(uint64_t));
}

extern __shared__ __align__(16) unsigned char vk_smem[];

// The dynamic tail: dfix row of shift s, and the step constants of a warp:
// {-L_{t+1,t}/L_{t+1,t+1}, round(g_t 2^32/N), shift_t 2^32, 0}, one 16-byte load per step.
template <int DMAX>
__device__ __forceinline__ uint32_t* dfix_row(int s) {
    return (uint32_t*)(vk_smem + align16(sizeof(GenzSmem<DMAX, true>))) + s * DMAX;
}
template <int DMAX>
__device__ __forceinline__ float4* stepw_of(int max_S, int warp) {
    return (float4*)(vk_smem + align16(sizeof(GenzSmem<DMAX, true>)) + align16((size_t)max_S * DMAX * 4)) +
           warp * DMAX;
}
template <int DMAX>
__device__ __forceinline__ fix::FixTables& fix_tables() {
    return *reinterpret_cast<fix::FixTables*>(vk_smem + align16(sizeof(GenzSmem<DMAX, false>)));
}
template <int DMAX>
__device__ __forceinline__ uint64_t* shift64_of(int warp) {
    return reinterpret_cast<uint64_t*>(vk_smem + align16(sizeof(GenzSmem<DMAX, false>)) +
                                       align16(sizeof(fix::FixTables))) +
           warp * DMAX;
}

// Phi(z) and 1 - Phi(z), the smaller one from the tail to full precision.
__device__ __forceinline__ void phi_pair64(double z, double& e, double& ec) {
    const double t = normcdf(-fabs(z));
    e = (z < 0.0) ? t : 1.0 - t;
    ec = (z < 0.0) ? 1.0 - t : t;
}


// 2^-E as a double (0 once below the normal range).
__device__ __forceinline__ double pow2_neg(int E) {
    return (E < 1022) ? __longlong_as_double((long long)(1023 - E) << 52) : 0.0;
}

// ------------------------ mixed (FP32 integrand) path ------------------------
// Per lane and point: the standardised partial sums R of the later variables,
// the current conditional probability e (and 1 - e, and log2 e once e is below
// 2^-64), and the running product g 2^-E of e_1 .. e_t (e_0 is factored out
// and applied in FP64), its exponent tracked so it never underflows.

template <int DMAX, int P>
struct MixedLanes {
    float R[P][DMAX - 1];
    float e[P], ec[P], le2[P], g[P];
    int E[P];
    bool tiny[P];
    uint32_t kk[P];
};

__device__ __forceinline__ void scale_by(float& g, int& E, float v) {
    g *= v;
    if (g < 0x1p-32f) {
        g *= 0x1p32f;
        E += 32;
    }
}

// g 2^-E times 2^l2 (l2 << 0), kept normal
__device__ __forceinline__ void scale_by_log2(float& g, int& E, float l2) {
    const float k = floorf(l2);
    g *= special::ex2(l2 - k);
    E -= (int)k;
    if (g < 0x1p-32f) {
        g *= 0x1p32f;
        E += 32;
    }
}

// Steps t0 <= t < t1 with update width W: each step needs q - t - 1 <= W.
template <int DMAX, int P, int W>
__device__ __forceinline__ void mixed_steps(const GenzSmem<DMAX, true>& sm, const uint32_t* dfs,
                                            int t0, int t1, MixedLanes<DMAX, P>& L) {
    for (int t = t0; t < t1; ++t) {
        const float* lup = sm.Lup[t];
        const float lz = sm.Lz[t];
        const uint32_t G = sm.gl[t], Dt = dfs[t];
#pragma unroll
        for (int p = 0; p < P; ++p) {
            if (t > 0) {  // g *= e_t
                if (!L.tiny[p])
                    scale_by(L.g[p], L.E[p], L.e[p]);
                else
                    scale_by_log2(L.g[p], L.E[p], L.le2[p]);
            }
            // lattice coordinate in 32-bit fixed point, tent transform w = 1 - |2x - 1|
            // of x = X 2^-32: exactly |int32(X)| 2^-31
            const uint32_t X = L.kk[p] * G + Dt;
            const uint32_t V = ((int32_t)X < 0) ? 0u - X : X;
            const float w = __uint2float_rn(V) * 0x1p-31f;
            float y;
            if (!L.tiny[p]) {
                const float a = __uint2float_rn(0x80000000u - V) * 0x1p-31f;  // |2x - 1|
                y = special::phiinv_pq(w * L.e[p], fmaf(w, L.ec[p], a));
            } else {  // w e_t below 2^-64: from log2(w e_t)
                y = special::phiinv_log2(special::lg2(w) + L.le2[p]);
            }
            const float z = fmaf(-lz, y, L.R[p][0]);  // kZs z (the tables carry kZs)
#pragma unroll
            for (int r = 0; r < W; ++r) L.R[p][r] = fmaf(-lup[r], y, L.R[p][r + 1]);
            special::phi_pair_s(z, L.e[p], L.ec[p], L.tiny[p], L.le2[p]);
        }
    }
}

// Steps t <= t' < t_stop of a term with q steps, in phases of update width
// W, W - 8, ...: a step needs width q - t' - 1.
template <int DMAX, int P, int W>
__device__ __forceinline__ void mixed_phases(const GenzSmem<DMAX, true>& sm, const uint32_t* dfs,
                                             int t, int t_stop, int q, MixedLanes<DMAX, P>& L) {
    constexpr int WN = W - 8;
    const int t_end = (WN > 0) ? max(t, min(t_stop, q - 1 - WN)) : t_stop;
    mixed_steps<DMAX, P, W>(sm, dfs, t, t_end, L);
    if constexpr (WN > 0) mixed_phases<DMAX, P, WN>(sm, dfs, t_end, t_stop, q, L);
}

template <int DMAX, int P>
__device__ __forceinline__ void genz_points_safe(const GenzSmem<DMAX, true>& sm, int q, int c, int s,
                                                  int64_t k_begin, int64_t k_end, double& acc_num,
                                                  double& acc_den) {
    constexpr int W0 = (DMAX - 2 > 0) ? DMAX - 2 : 1;
    const int lane = threadIdx.x & 31;
    const uint32_t* dfs = dfix_row<DMAX>(s);
    const int cut = (c >= 1) ? c : q;  // after steps 0 .. cut-1, g = e_1 ... e_{c-1}
    const float e0f = (float)sm.e0, ec0f = (float)sm.ec0;
    const bool tiny0 = sm.e0 < 0x1p-64;
    for (int64_t kb = k_begin; kb < k_end; kb += 32 * P) {
        MixedLanes<DMAX, P> L;
        bool valid[P];
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const int64_t k = kb + p * 32 + lane;
            valid[p] = k < k_end;
            L.kk[p] = (uint32_t)(valid[p] ? k : k_begin);
#pragma unroll
            for (int r = 0; r < DMAX - 1; ++r) L.R[p][r] = sm.up[1 + r];
            L.e[p] = e0f;
            L.ec[p] = ec0f;
            L.tiny[p] = tiny0;
            L.le2[p] = sm.le2_0;
            L.g[p] = 1.0f;
            L.E[p] = 0;
        }
        mixed_phases<DMAX, P, W0>(sm, dfs, 0, cut, q, L);
        double den_c[P];
#pragma unroll
        for (int p = 0; p < P; ++p) den_c[p] = (double)L.g[p] * pow2_neg(L.E[p]);
        mixed_phases<DMAX, P, W0>(sm, dfs, cut, q, q, L);
#pragma unroll
        for (int p = 0; p < P; ++p) {
            if (valid[p]) {
                const double den = den_c[p];
                float gn = L.g[p];
                int En = L.E[p];
                if (!L.tiny[p])
                    scale_by(gn, En, L.e[p]);
                else
                    scale_by_log2(gn, En, L.le2[p]);
                acc_den += den;
                acc_num += (double)gn * pow2_neg(En);
            }
        }
    }
}

// ------------------- mixed path, fast form (the common case) -----------------
// No log-space bookkeeping: a conditional probability below the FP32 range
// simply zeroes its point's sample.  Such a sample is below 2^-62 in absolute
// terms, so whenever the term's lattice means are at least 2^-40 the loss is
// below 2^-22 relative; terms whose means fall under 2^-40 are flagged and
// re-evaluated by the log-space form above (genz_points_safe).  Sums run in
// FP32 with Kahan compensation per lane and are folded into FP64 per unit.

struct Kahan32 {
    float s = 0.0f, c = 0.0f;
    __device__ __forceinline__ void add(float x) {
        const float y = __fsub_rn(x, c);
        const float t = __fadd_rn(s, y);
        c = __fsub_rn(__fsub_rn(t, s), y);
        s = t;
    }
    __device__ __forceinline__ double value() const { return (double)s - (double)c; }
};

template <int DMAX, int P, int W, bool FIRST>
__device__ __forceinline__ void fast_step(const GenzSmem<DMAX, true>& sm, const float4* sc, int t,
                                          float (&R)[P][DMAX - 1], float (&e)[P], float (&ec)[P],
                                          float (&g)[P], const uint32_t (&kk)[P]) {
    const float* lup = sm.Lup[t];
    const float4 c = sc[t];
    const float nlz = c.x;  // -L_{t+1,t}/L_{t+1,t+1}
    const uint32_t G = __float_as_uint(c.y), Dt = __float_as_uint(c.z);
    if constexpr (P == 1) {  // one point per lane: the per-point form keeps fewer values live
        if (!FIRST) g[0] = __fmul_rn(g[0], e[0]);
        const uint32_t X = kk[0] * G + Dt;
        const float wk = __fmul_rn(fabsf(__int2float_rn((int32_t)X)), 0x1p-27f);  // 16 w
        const float yv = special::phiinv16_pq(__fmul_rn(wk, e[0]), fmaf(wk, ec[0], __fsub_rn(16.0f, wk)));
        const float z = fmaf(nlz, yv, R[0][0]);
#pragma unroll
        for (int r = 0; r < W; ++r) R[0][r] = fmaf(-lup[r], yv, R[0][r + 1]);
        special::phi_pair_fast_s(z, e[0], ec[0]);
        return;
    }
    // Phi^{-1} of every point's w_t e_t first, so one full-warp vote decides
    // the tail pieces for all of them (every lane of the warp runs this step)
    float pp[P], qq[P], y[P];
    bool tail[P];
    bool any_tail = false;
#pragma unroll
    for (int p = 0; p < P; ++p) {
        if (!FIRST) g[p] = __fmul_rn(g[p], e[p]);  // g = e_1 ... e_t
        // lattice coordinate in 32-bit fixed point, tent transform w = 1 - |2x - 1|
        // of x = X 2^-32: exactly |int32(X)| 2^-31 (the sign folds into the
        // product); carried as 16 w, 16 w e and 16 (1 - w e), exact scalings
        // that give the quantile's polynomial its variable directly
        const uint32_t X = kk[p] * G + Dt;
        const float wk = __fmul_rn(fabsf(__int2float_rn((int32_t)X)), 0x1p-27f);
        pp[p] = __fmul_rn(wk, e[p]);
        qq[p] = fmaf(wk, ec[p], __fsub_rn(16.0f, wk));
        y[p] = special::phiinv16_central(pp[p], qq[p], tail[p]);
        any_tail = any_tail || tail[p];
    }
    if (__any_sync(0xffffffffu, any_tail)) {
#pragma unroll
        for (int p = 0; p < P; ++p) y[p] = special::phiinv16_with_tail(pp[p], qq[p], tail[p], y[p]);
    }
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const float yv = special::phiinv_finish(pp[p], qq[p], y[p]);
        const float z = fmaf(nlz, yv, R[p][0]);  // kZs z (the tables carry kZs)
#pragma unroll
        for (int r = 0; r < W; ++r) R[p][r] = fmaf(-lup[r], yv, R[p][r + 1]);
        special::phi_pair_fast_s(z, e[p], ec[p]);
    }
}

// Width step between phases: 4 up to 21 variables; 6 above, where fewer
// copies of the step body (instruction cache) beat the extra padding FMAs
// (measured: m = 30 5.7 % faster, m <= 16 0.7 % slower with 6).
#ifndef VK_PHASE_STEP_SMALL
#define VK_PHASE_STEP_SMALL 4
#endif
__host__ __device__ constexpr int phase_step(int dmax) { return dmax <= 21 ? VK_PHASE_STEP_SMALL : 6; }

// Steps t <= t' < q (t >= 1) of a term with q steps, in phases of update width
// W, W - step, ...: a step needs width q - t' - 1, so the phase of width W ends
// where W - step suffices.  CAPTURE (terms whose conditioning set is shorter
// than q): at the start of step c (warp-uniform), gd = g = e_1 ... e_{c-1},
// the conditioning CDF's sample.  A classic term (c = q) uses g at the end
// and runs the instantiation without the check.
template <int DMAX, int P, int W, bool CAPTURE>
__device__ __forceinline__ void fast_phases(const GenzSmem<DMAX, true>& sm, const float4* sc, int t,
                                            int q, int cut, float (&R)[P][DMAX - 1], float (&e)[P],
                                            float (&ec)[P], float (&g)[P], float (&gd)[P],
                                            const uint32_t (&kk)[P]) {
    constexpr int WN = W - phase_step(DMAX);
    const int t_end = (WN > 0) ? max(t, min(q, q - 1 - WN)) : q;
    for (int tt = t; tt < t_end; ++tt) {
        if (CAPTURE && tt == cut) {
#pragma unroll
            for (int p = 0; p < P; ++p) gd[p] = g[p];
        }
        fast_step<DMAX, P, W, false>(sm, sc, tt, R, e, ec, g, kk);
    }
    if constexpr (WN > 0) fast_phases<DMAX, P, WN, CAPTURE>(sm, sc, t_end, q, cut, R, e, ec, g, gd, kk);
}

template <int DMAX, int P, bool CAPTURE>
__device__ __forceinline__ void genz_points_fast(const GenzSmem<DMAX, true>& sm, int q, int c, int s,
                                                 int max_S, int64_t k_begin, int64_t k_end,
                                                 double& acc_num, double& acc_den) {
    constexpr int W0 = (DMAX - 2 > 0) ? DMAX - 2 : 1;
    const int lane = threadIdx.x & 31;
    float4* sc = stepw_of<DMAX>(max_S, threadIdx.x >> 5);
    const uint32_t* dfs = dfix_row<DMAX>(s);
    __syncwarp();
    for (int t = lane; t < q; t += 32)
        sc[t] = make_float4(-sm.Lz[t], __uint_as_float(sm.gl[t]), __uint_as_float(dfs[t]), 0.0f);
    __syncwarp();
    const float e0f = (float)sm.e0, ec0f = (float)sm.ec0;
    // point indices in 32 bits: N <= 2^31 - 1, so kb + 32 P stays below 2^32
    const uint32_t k_lo = (uint32_t)k_begin, k_hi = (uint32_t)k_end;
    Kahan32 kn, kd;
    for (uint32_t kb = k_lo; kb < k_hi; kb += 32 * P) {
        float R[P][DMAX - 1], e[P], ec[P], g[P], gd[P];
        uint32_t kk[P];
        bool valid[P];
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const uint32_t k = kb + p * 32 + lane;
            valid[p] = k < k_hi;
            kk[p] = valid[p] ? k : k_lo;
#pragma unroll
            for (int r = 0; r < DMAX - 1; ++r) R[p][r] = sm.up[1 + r];
            e[p] = e0f;
            ec[p] = ec0f;
            g[p] = 1.0f;
            gd[p] = 1.0f;  // c = 1: e_0 alone (factored out)
        }
        fast_step<DMAX, P, W0, true>(sm, sc, 0, R, e, ec, g, kk);  // q >= 1: step 0 at full width
        fast_phases<DMAX, P, W0, CAPTURE>(sm, sc, 1, q, c, R, e, ec, g, gd, kk);
#pragma unroll
        for (int p = 0; p < P; ++p) {
            if (valid[p]) {
                kd.add(CAPTURE ? gd[p] : g[p]);
                kn.add(__fmul_rn(g[p], e[p]));
            }
        }
    }
    acc_num += kn.value();
    acc_den += kd.value();
}

// ------------------------------- FP64 path ---------------------------------
// The step in 64-bit fixed point (special_fix.h); FP64 only in the tails that
// its tables leave out and in the two sums over points.

// One step t (lattice coordinate t, variable t + 1 next) of a point whose
// later variables are `later` = q - 1 - t (warp-uniform).  x = frac(k g_t / N +
// Delta_t) in 64-bit fixed point X = k G_t + D_t.
//
// Bound by instruction issue: 385 instructions a step at m = 20 (60 IMAD.WIDE
// at 4 cycles each, two or three additions a product), against 77 FP64 ones at
// 76 cycles in the FP64 form.  50 x 50 grid, m = 20, N S = 65,536: 453 ms in
// FP64, 55.5 ms so; m = 30 (N S = 16,384) 182 -> 24.9 ms; m = 50 (8,192)
// 169 -> 37.6 ms.  One copy of the body serves every step and the updates run
// in groups of four variables behind uniform branches: phases with a copy
// each, as the mixed path has them, overran the instruction cache (94.6 ms
// against 73 ms at that point), two or three phases padded more than they saved.
template <int DMAX>
__device__ __forceinline__ void fix_step(const GenzSmem<DMAX, false>& sm, const fix::FixTables& tb, uint64_t Dt,
                                         int t, int later, uint32_t k, uint64_t K, int64_t (&R)[DMAX - 1],
                                         fix::FixProb& e) {
    const FixStep& st = sm.step[t];
    const fix::Digits Y = fix_quantile(tb, (uint64_t)k * st.G + Dt, e, K);
    const int64_t acc = fix::mul_add(st.nlz, Y, R[0], K);
    const fix::Digits* lup = sm.Lup[t];
#pragma unroll
    for (int r0 = 0; r0 < DMAX - 2; r0 += 4) {
        if (later <= r0) break;
#pragma unroll
        for (int r = r0; r < r0 + 4 && r < DMAX - 2; ++r) R[r] = fix::mul_add(lup[r], Y, R[r + 1], K);
    }
    const int64_t hi = fix::mul_add(st.rdiag, fix::digits(acc), -fix::kMulBias, K);
    fix_phi(tb, hi, st.lim, st.shift, e, K);
}

// The scale of row v (v >= 1) and its step constants, one thread a row.
template <int DMAX>
__device__ __forceinline__ void fix_row(GenzSmem<DMAX, false>& sm, int v, uint32_t g, uint64_t N) {
    double sum = 0.0;
    for (int t = 0; t < v; ++t) sum += fabs(sm.A[v][t]);
    const FixVar r = fix_scale(sm.A[v][v], sum, sm.bu[v], v);
    sm.scale[v] = r.kL;
    sm.up[v] = r.up;
    FixStep& st = sm.step[v - 1];
    st.G = fix64_ratio(g, N);
    st.nlz = fix_coef(sm.A[v][v - 1], r.kL);
    st.rdiag = r.rdiag;
    st.lim = r.lim;
    st.shift = r.shift;
}

template <int DMAX>
__device__ __forceinline__ void genz_points_fp64(const ProbDev& P,
                                                 int q, int c, int s, int64_t k_begin, int64_t k_end,
                                                 double& acc_num, double& acc_den) {
    const int lane = threadIdx.x & 31;
    // The shared memory's base as a value the compiler keeps in a register
    // (it forms the address of the array itself anew at every use).
    uint32_t base;
    asm volatile("mov.u32 %0, %1;" : "=r"(base) : "r"((uint32_t)__cvta_generic_to_shared(vk_smem)));
    const unsigned char* smem = (const unsigned char*)__builtin_assume_aligned(__cvta_shared_to_generic(base), 16);
    const GenzSmem<DMAX, false>& sm = *reinterpret_cast<const GenzSmem<DMAX, false>*>(smem);
    const fix::FixTables& tb = *reinterpret_cast<const fix::FixTables*>(smem + align16(sizeof(GenzSmem<DMAX, false>)));
    uint64_t* D = shift64_of<DMAX>(threadIdx.x >> 5);
    const uint64_t K = fix::opaque_mid();
    const double* dl = P.delta + (int64_t)s * P.dim;
    __syncwarp();
    for (int t = lane; t < q; t += 32)
        D[t] = fix_shift(dl[t]);
    __syncwarp();
    for (int64_t k = k_begin + lane; k < k_end; k += 32) {
        int64_t R[DMAX - 1];
#pragma unroll
        for (int r = 0; r < DMAX - 1; ++r) R[r] = sm.up[1 + r];
        fix::FixProb e = sm.p0;
        fix::FixFloat f = fix::prob(e), fc = f;  // c = 1: e_0
        for (int t = 0; t < q; ++t) {
            if (t + 1 == c) fc = f;  // e_0 ... e_{c-1}: the c-dim CDF sample of the leading block
            fix_step<DMAX>(sm, tb, D[t], t, q - 1 - t, (uint32_t)k, K, R, e);
            f = fix::times(f, e);  // e_0 ... e_{t+1}
        }
        acc_den += __longlong_as_double((long long)fix::to_bits(fc));
        acc_num += __longlong_as_double((long long)fix::to_bits(f));
    }
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Work items: (problem, site, shift group).  A list of segments maps a flat
// item index to them: segment k covers items [seg_prefix[k], seg_prefix[k+1])
// = sites seg_base[k].y, ... of problem seg_base[k].x, each split into
// `groups` shift groups (the group index varies fastest).  The log-space form
// takes an explicit list of (problem, site) instead, its count on the device.
//
// The last round of a launch: with items of equal size, a launch of n items
// on a grid of G CTAs leaves n mod G CTAs with one item more than the rest,
// and they finish alone at a fraction of their SMs' throughput.  So the sites
// after `whole_sites` (those whose items would form that last round) are cut
// into `tail_groups` shift groups instead of `groups`: more, smaller items
// that spread over the whole grid.  A shift's partial means are computed by
// one warp whatever the grouping, so the results do not change.
struct ItemSrc {
    const int2* items;       // the log-space form's (problem, site) list, or nullptr
    const int* dev_count;    // its device-side count
    const int* seg_prefix;   // n_segs + 1 prefix sums of items
    const int2* seg_base;    // (problem, first site) per segment
    int n_segs;
    int n_items;
    int groups;              // shift groups per site (segment mode)
    int whole_sites;         // sites [0, whole_sites) in `groups` groups, the rest in tail_groups
    int tail_groups;
    int fb_cap;              // capacity of the flagged-item list
};

__device__ __forceinline__ void item_of(const ItemSrc& src, int it, int2& ps, int& grp, int& ngroups) {
    int site_item;
    const int whole = src.whole_sites * src.groups;
    if (it < whole) {
        site_item = it / src.groups;
        grp = it - site_item * src.groups;
        ngroups = src.groups;
    } else {
        const int j = it - whole, k = j / src.tail_groups;
        site_item = src.whole_sites + k;
        grp = j - k * src.tail_groups;
        ngroups = src.tail_groups;
    }
    int lo = 0, hi = src.n_segs - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (src.seg_prefix[mid] <= site_item)
            lo = mid;
        else
            hi = mid - 1;
    }
    ps = make_int2(src.seg_base[lo].x, src.seg_base[lo].y + (site_item - src.seg_prefix[lo]));
}

// Entry and shift group of item `it` of the explicit list: the entries before `whole`
// with all shifts, the others in tail_groups.
__device__ __forceinline__ void listed_item_of(const ItemSrc& src, int whole, int tail_groups, int it, int2& ps,
                                               int& grp, int& ngroups) {
    const int j = it - whole, k = j < 0 ? 0 : j / tail_groups;
    ngroups = j < 0 ? 1 : tail_groups;
    grp = j < 0 ? 0 : j - k * tail_groups;
    ps = src.items[j < 0 ? it : whole + k];
}

// MODE: 0 = FP64, 1 = mixed fast form, 2 = mixed log-space form.
constexpr int kModeFP64 = 0, kModeFast = 1, kModeSafe = 2;

// Register cap per thread: the FP64 step at up to 13 variables runs best with
// 20 warps an SM (m = 10: 8.0 against 8.4 ms at 128 registers); from 14 on 16 warps at
// 128, spills and all (12 warps at 168 without: m = 24 18.06 against 18.12 ms, m = 27 21.97
// against 21.32, m = 30 26.9 against 24.5).  The fast mixed loop keeps DMAX - 1 partial sums per
// point in registers; capping the rest raises the number of resident warps.
// Blocks above 32 variables run one point per lane with up to 128 registers
// (fast) or 255 (FP64 and log-space forms, whose partial sums are wider), and
// at most 256 threads per CTA.
#ifndef VK_CAP_P1_SMALL
#define VK_CAP_P1_SMALL 64
#endif
#ifndef VK_CAP_P1_LARGE
#define VK_CAP_P1_LARGE 80
#endif
#ifndef VK_CAP_P2_SMALL
#define VK_CAP_P2_SMALL 96
#endif
#ifndef VK_CAP_P2_LARGE
#define VK_CAP_P2_LARGE 128
#endif
__host__ __device__ constexpr int reg_cap(int dmax, int p, int mode) {
    return dmax > 32            ? (mode == kModeFast ? 128 : 255)
           : mode != kModeFast ? (mode == kModeFP64 && dmax <= 13 ? 96 : 128)
           : p == 1            ? (dmax <= 16 ? VK_CAP_P1_SMALL : VK_CAP_P1_LARGE)
                               : (dmax <= 16 ? VK_CAP_P2_SMALL : VK_CAP_P2_LARGE);
}
__host__ __device__ constexpr int max_threads(int dmax, int p, int mode) {
    return reg_cap(dmax, p, mode) > 128 ? 256 : 512;
}

// A term of a problem: its block (the conditioning sites ascending, then the
// sites of the term) into sm.bidx, c and d; false if the row is malformed.
// Classic (group 0): term i is site i with N_i = the first min(m, i) entries
// of row i.  Group p: term k is sites k p .. min(k p + p, D) - 1 with the
// leading non-negative entries of row k (the rest must be -1).
template <int DMAX, bool MIXED>
__device__ __forceinline__ bool term_block(GenzSmem<DMAX, MIXED>& sm, const ProbDev& Pd, int64_t term,
                                           int& c, int& d, int64_t& i0) {
    const int lane = threadIdx.x & 31;
    const int m = Pd.m;
    const int32_t* row = Pd.nbr + term * (int64_t)m;
    int g;
    bool ok = true;
    if (Pd.group == 0) {
        i0 = term;
        g = 1;
        c = (int)((term < m) ? term : m);
    } else {
        i0 = term * Pd.group;
        g = (int)min((int64_t)Pd.group, Pd.D - i0);
        c = m;
        for (int base = 0; base < m; base += 32) {  // first negative entry
            const int r = base + lane;
            const unsigned neg = __ballot_sync(0xffffffffu, r < m && row[r] < 0);
            if (neg) {
                c = base + __ffs(neg) - 1;
                break;
            }
        }
        for (int r = c + lane; r < m; r += 32) ok = ok && row[r] < 0;
    }
    d = c + g;
    if (d > DMAX) ok = false;
    if (ok)
        for (int v = lane; v < d; v += 32) sm.bidx[v] = (v < c) ? row[v] : (int)(i0 + (v - c));
    __syncwarp();
    if (ok)
        for (int v = lane; v < c; v += 32) {
            const int idx = sm.bidx[v];
            ok = ok && idx >= 0 && idx < i0 && (v == 0 || idx > sm.bidx[v - 1]);  // ascending (block order)
        }
    return __all_sync(0xffffffffu, ok);
}

// Lattice slices of a shift where the tile names none, of the problem's own S and
// N alone (so a problem's sums do not depend on the batch it runs in): one in the
// mixed fast form, whose FP32 lane sums another split would round anew; FP64 as
// many as make the units (shifts x slices) a multiple of four warps; four in the
// log-space form, a unit for each of its four warps.
__host__ __device__ constexpr int auto_slices(int S, int64_t N, int mode) {
    int g = mode == kModeFast ? 1 : (mode == kModeSafe || (S & 1)) ? 4 : (S & 2) ? 2 : 1;
    while (g > 1 && (S * g > kMaxUnits || N < 256 * g)) g >>= 1;
    return g;
}

// Shift groups for the `rest` entries of the list's last round on a grid of G CTAs (all
// entries, where there are fewer than CTAs): of 1, 2, 4, ... the number whose rounds
// take the fewest steps, an item's being its factor (about 3 a variable and 20) and its
// warps' rounds of units.  Any listed problem may stand for the rest: the groups do not
// change a shift's sums.
__device__ __forceinline__ int listed_groups(const ProbDev& P, int rest, int G, int max_S, int slices, int n_warps) {
    const int64_t unit = (P.N + 32 * slices - 1) / (32 * slices) * (P.m + 1);
    int64_t best = LLONG_MAX;
    int groups = 1;
    for (int g = 1; g <= max_S; g *= 2) {
        const int units = (max_S + g - 1) / g * slices;
        const int64_t t = ((int64_t)rest * g + G - 1) / G * (3 * P.m + 20 + (units + n_warps - 1) / n_warps * unit);
        if (t < best) {
            best = t;
            groups = g;
        }
    }
    return groups;
}

template <int DMAX, int P, int MODE>
__global__ void __launch_bounds__(max_threads(DMAX, P, MODE)) __maxnreg__(reg_cap(DMAX, P, MODE))
    genz_kernel(const ProbDev* __restrict__ probs, ItemSrc src, int tile_slices, int max_S,
                ProbResult* __restrict__ results, int* __restrict__ fallback_count,
                int2* __restrict__ fallback_items) {
    constexpr bool MIXED = MODE != kModeFP64;
    GenzSmem<DMAX, MIXED>& sm = *reinterpret_cast<GenzSmem<DMAX, MIXED>*>(vk_smem);
    using T = typename GenzSmem<DMAX, MIXED>::T;
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int n_warps = blockDim.x >> 5;

    if constexpr (!MIXED) {
        load_fix_tables(fix_tables<DMAX>());
        __syncthreads();
    }
    int n_run = src.n_items, whole = 0, tail_groups = 1;
    if constexpr (MODE == kModeSafe) {
        const int n = min(*src.dev_count, src.n_items), G = (int)gridDim.x;
        whole = n / G * G;
        if (n > whole) {
            const ProbDev& P0 = probs[src.items[whole].x];
            tail_groups = listed_groups(P0, n - whole, G, max_S, auto_slices(P0.S, P0.N, MODE), n_warps);
        }
        n_run = whole + (n - whole) * tail_groups;
    }
    for (int it = blockIdx.x; it < n_run; it += gridDim.x) {
        int2 item;
        int grp, groups;
        if constexpr (MODE == kModeSafe)
            listed_item_of(src, whole, tail_groups, it, item, grp, groups);
        else
            item_of(src, it, item, grp, groups);
        const ProbDev& Pd = probs[item.x];
        const int64_t term = item.y;
        const int S = Pd.S;
        const int s_lo = (S * grp) / groups, s_hi = (S * (grp + 1)) / groups;
        const int slices = tile_slices > 0 ? tile_slices : auto_slices(S, Pd.N, MODE);

        // ---- prologue: block (warp 0), covariance and Cholesky (all warps); FP64 ----
        if (warp == 0) {
            int c = 0, d = 1;
            int64_t i0 = 0;
            const int bad = term_block<DMAX, MIXED>(sm, Pd, term, c, d, i0) ? 0 : 2;
            if (!bad)
                for (int v = lane; v < d; v += 32) {
                    const int idx = sm.bidx[v];
                    sm.bx[v] = Pd.sites[2 * (int64_t)idx];
                    sm.by[v] = Pd.sites[2 * (int64_t)idx + 1];
                    sm.bu[v] = Pd.u[idx];
                }
            if (lane == 0) {
                sm.bad = bad;
                sm.q = d - 1;
                sm.c = c;
                sm.flag = 0;
            }
        }
        __syncthreads();
        // covariance, lower triangle, entries packed over every thread (the
        // FP64 units of all the CTA's warps)
        if (!sm.bad) {
            const int d = sm.q + 1;
            for (int e = threadIdx.x; e < d * (d + 1) / 2; e += blockDim.x) {
                int r, col;
                tri_index(e, r, col);
                const double h = site_dist(Pd, __dsub_rn(sm.bx[r], sm.bx[col]), __dsub_rn(sm.by[r], sm.by[col]));
                double v = cov_fn(Pd.cov_kind, Pd.variance, Pd.range, Pd.nu, h);
                if (col == r) v += Pd.nugget;
                if (Pd.lr_k > 0) {  // conditional covariance: minus scale V_a . V_b
                    const double* Va = Pd.lr_V + (int64_t)sm.bidx[r] * Pd.lr_k;
                    const double* Vb = Pd.lr_V + (int64_t)sm.bidx[col] * Pd.lr_k;
                    double acc = 0.0;
                    for (int t = 0; t < Pd.lr_k; ++t) acc = fma(Va[t], Vb[t], acc);
                    v = v - Pd.lr_scale * acc;
                }
                sm.A[r][col] = v;
            }
        }
        __syncthreads();
        if (!sm.bad) {
            const int d = sm.q + 1;
            // Cholesky, right-looking: after column j is final, the trailing
            // triangle takes its update fma(-L_rj, L_cj, A_rc).  Each entry thus
            // receives its terms in ascending k with fma and is divided by the
            // pivot last: the operations of the row-by-row definition, in its
            // order.  Warp 0 takes the next column's entries and goes on to its
            // pivot and quotients (exact_math.h: the same values by integers, a
            // third of the FP64 chain), the other warps the rest of the triangle
            // meanwhile; one barrier a column.  (One warp for all of it: 26 us a
            // term at d = 21, 160 us at d = 51.)
            int failed = 0;
            for (int j = 0; j < d; ++j) {
                if (warp == 0) {
                    const double s = sm.A[j][j];
                    if (s > 0.0) {  // warp-uniform: every lane reads the same value
                        const exact::Pivot piv = exact::pivot(s);
                        for (int r = j + 1 + lane; r < d; r += 32) sm.A[r][j] = exact::quotient(sm.A[r][j], piv);
                        __syncwarp();
                        if (lane == 0) sm.A[j][j] = piv.piv;
                    } else {
                        failed = 1;
                    }
                }
                failed = __syncthreads_or(failed);
                if (failed) break;  // CTA-uniform
                if (warp == 0) {
                    for (int r = j + 1 + lane; r < d; r += 32)
                        sm.A[r][j + 1] = fma(-sm.A[r][j], sm.A[j + 1][j], sm.A[r][j + 1]);
                    __syncwarp();
                }
                if (warp > 0 || n_warps == 1) {
                    const int n = d - 2 - j, w = n_warps > 1 ? 32 : 0;
                    for (int e = (int)threadIdx.x - w; e < n * (n + 1) / 2; e += (int)blockDim.x - w) {
                        int a, b;
                        tri_index(e, a, b);
                        const int r = j + 2 + a, col = j + 2 + b;
                        sm.A[r][col] = fma(-sm.A[r][j], sm.A[col][j], sm.A[r][col]);
                    }
                    if (n_warps == 1) __syncwarp();
                }
            }
            if (failed && threadIdx.x == 0) sm.bad = 1;
        }
        __syncthreads();
        const int q = sm.q, c = sm.c;

        if (!sm.bad) {
            // ---- derived tables for the recursion ----
            // (mixed: one FP64 reciprocal 1/L_vv per row, each row scaled by
            // kZs/L_vv, so the recursion's conditional means arrive as the
            // kZs z that its Phi takes; FP64: integers of each row's scale)
            constexpr int LS = GenzSmem<DMAX, MIXED>::LS;
            const int d = q + 1;
            if (threadIdx.x == blockDim.x - 1) {  // e_0, beside the tables
                const double z0 = sm.bu[0] / sm.A[0][0];
                phi_pair64(z0, sm.e0, sm.ec0);
                sm.le2_0 = (sm.e0 < 0x1p-64) ? (float)log2(sm.e0) : 0.0f;
                if constexpr (!MIXED)
                    sm.p0 = fix::prob_of((uint64_t)__double_as_longlong(z0 < 0.0 ? sm.e0 : sm.ec0), z0 < 0.0);
            }
            if constexpr (MIXED) {
                for (int v = threadIdx.x; v < DMAX; v += blockDim.x)
                    sm.diag[v] = (v < d) ? special::kZsD / sm.A[v][v] : 0.0;
            } else {
                for (int v = threadIdx.x; v < DMAX; v += blockDim.x) {
                    if (v >= 1 && v < d)
                        fix_row<DMAX>(sm, v, Pd.g[v - 1], (uint64_t)Pd.N);
                    else
                        sm.up[v] = 0;
                }
            }
            __syncthreads();
            for (int x = threadIdx.x; x < DMAX * LS; x += blockDim.x) {
                const int t = x / LS, r = x % LS, v = t + 2 + r;
                T val = T();
                if (t < q && v < d) {
                    if constexpr (MIXED)
                        val = (T)(sm.A[v][t] * sm.diag[v]);
                    else
                        val = fix_coef(sm.A[v][t], sm.scale[v]);
                }
                sm.Lup[t][r] = val;
            }
            if constexpr (MIXED) {
                for (int v = threadIdx.x; v < DMAX; v += blockDim.x) {
                    T val = (T)0, lz = (T)0;
                    if (v < d) val = (T)(sm.bu[v] * sm.diag[v]);
                    if (v < q) lz = (T)(sm.A[v + 1][v] * sm.diag[v + 1]);
                    sm.up[v] = val;
                    sm.Lz[v] = lz;
                    if (v < q) sm.gl[v] = Pd.gfix[v];
                }
                for (int x = threadIdx.x; x < S * DMAX; x += blockDim.x) {
                    const int s = x / DMAX, t = x % DMAX;
                    dfix_row<DMAX>(s)[t] = (t < q) ? Pd.dfix[(int64_t)s * Pd.dim + t] : 0u;
                }
            }
        }
        __syncthreads();

        // ---- body: Genz recursion over shifts x lattice slices ----
        const int units = (s_hi - s_lo) * slices;
        if (!sm.bad && q > 0) {
            for (int un = warp; un < units; un += n_warps) {
                const int s = s_lo + un / slices, h = un % slices;
                const int64_t k0 = (Pd.N * h) / slices, k1 = (Pd.N * (h + 1)) / slices;
                double an = 0.0, ad = 0.0;
                if constexpr (MODE == kModeFast) {
                    if (c == q)  // classic term (or a group of one): no capture in the loop
                        genz_points_fast<DMAX, P, false>(sm, q, c, s, max_S, k0, k1, an, ad);
                    else
                        genz_points_fast<DMAX, P, true>(sm, q, c, s, max_S, k0, k1, an, ad);
                }
                else if constexpr (MODE == kModeSafe)
                    genz_points_safe<DMAX, P>(sm, q, c, s, k0, k1, an, ad);
                else
                    genz_points_fp64<DMAX>(Pd, q, c, s, k0, k1, an, ad);
                an = warp_sum(an);
                ad = warp_sum(ad);
                if (lane == 0) {
                    sm.part_num[un] = an;
                    sm.part_den[un] = ad;
                }
            }
        }
        __syncthreads();

        // ---- epilogue: per-shift means ----
        for (int s = s_lo + threadIdx.x; s < s_hi; s += blockDim.x) {
            const int un0 = (s - s_lo) * slices;
            double vn, vd;
            if (sm.bad) {
                vn = vd = __longlong_as_double(0x7ff8000000000000LL);
            } else if (q == 0) {
                vn = sm.e0;
                vd = 1.0;
            } else {
                double sn = 0.0, sd = 0.0;
                for (int h = 0; h < slices; ++h) {
                    sn += sm.part_num[un0 + h];
                    sd += sm.part_den[un0 + h];
                }
                vn = sn / (double)Pd.N;
                vd = sd / (double)Pd.N;
                if constexpr (MIXED) {
                    vn *= sm.e0;
                    vd *= sm.e0;
                }
                if constexpr (!MIXED) {
                    if (sm.e0 != sm.e0) vn = vd = sm.e0;  // a NaN threshold
                }
                if (c == 0) vd = 1.0;  // no conditioning set: the term is the joint CDF itself
                if constexpr (MIXED) {
                    // the fast form is exact to 2^-22 only for means >= 2^-40
                    if (MODE == kModeFast && !(vn >= 0x1p-40 && vd >= 0x1p-40 && isfinite(vn) && isfinite(vd)))
                        sm.flag = 1;
                }
            }
            Pd.num[term * S + s] = vn;
            Pd.den[term * S + s] = vd;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            if (sm.bad) {
                ProbResult* R = Pd.res ? Pd.res : &results[item.x];
                atomicMin((unsigned long long*)&R->bad_site, (unsigned long long)term);
                R->status = (sm.bad == 1) ? VECCHIA_ERR_NOT_PD : VECCHIA_ERR_ARG;
            } else if (MODE == kModeFast && sm.flag && fallback_items) {
                const int pos = atomicAdd(fallback_count, 1);
                if (pos < src.fb_cap) fallback_items[pos] = item;  // the callers size it for every item
            }
        }
        __syncthreads();
    }
}

// ------------------------------- log-sum ------------------------------------
// Two passes with a fixed reduction order, so results are bit-identical run to
// run and alone vs in a batch:
//   partial: CTA (slice, problem) takes sites slice*32 .. +31, forms each
//     term T_i = log mean_s num - log mean_s den (Sec. 3.1: every term on the
//     log scale) and the delta-method pieces num_is/numbar_i - den_is/denbar_i,
//     and writes their slice sums;
//   final: one warp per problem adds the slices in order and forms
//     log P = sum_i T_i and SE = sqrt(sum_s l_s^2 / (S (S-1))).

// The per-site work (two FP64 logarithms and the S delta-method quotients) is
// FP64-bound on GB300: 32 sites a CTA, so that a 2,500-site problem is spread over
// 79 SMs, and eight warps a CTA, the means and logarithms on two of them and the
// shifts' quotients over all (S = 10: 16.7 -> 7.9 us).
constexpr int kSliceSites = kLogsumSlice;
constexpr int kLogsumWarps = 8;
static_assert(kSliceSites == 32, "a lane a site");

__device__ __forceinline__ double warp_sum_xor(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__global__ void __launch_bounds__(32 * kLogsumWarps) logsum_partial_kernel(
    const ProbDev* __restrict__ probs, double* const* __restrict__ terms, double* __restrict__ scratch,
    const int64_t* __restrict__ scratch_off) {
    __shared__ double mean[2][kSliceSites], lg[2][kSliceSites];
    const int pi = blockIdx.y, slice = blockIdx.x;
    const ProbDev& Pd = probs[pi];
    const int64_t D = Pd.n_terms;
    const int S = Pd.S;
    if ((int64_t)slice * kSliceSites >= D) return;  // CTA-uniform
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i = (int64_t)slice * kSliceSites + lane;
    const bool valid = i < D;
    if (warp < 2) {
        double m = 1.0;
        if (valid) {
            const double* v = (warp == 0 ? Pd.num : Pd.den) + i * S;
            double sum = 0.0;
            for (int s = 0; s < S; ++s) sum += v[s];
            m = sum / (double)S;
        }
        mean[warp][lane] = m;
        lg[warp][lane] = valid ? log(m) : 0.0;
    }
    __syncthreads();
    double* out = scratch + scratch_off[pi] + (int64_t)slice * (S + 1);
    const double a = mean[0][lane], b = mean[1][lane];
    for (int c = warp; c <= S; c += kLogsumWarps) {
        double v;
        if (c == 0) {
            const double T = lg[0][lane] - lg[1][lane];
            if (valid && terms && terms[pi]) terms[pi][i] = T;
            v = valid ? T : 0.0;
        } else {  // quotients, not products by reciprocals: equal shifts give exactly 0
            v = valid ? Pd.num[i * S + c - 1] / a - Pd.den[i * S + c - 1] / b : 0.0;
        }
        v = warp_sum_xor(v);
        if (lane == 0) out[c] = v;
    }
}

// Warp w of a problem's CTA adds slices w, w + 8, ... of its lanes' columns, the
// first warp the eight sums of each column in order.
__global__ void __launch_bounds__(32 * kLogsumWarps) logsum_final_kernel(const ProbDev* __restrict__ probs,
                                                                         ProbResult* __restrict__ results,
                                                                         const double* __restrict__ scratch,
                                                                         const int64_t* __restrict__ scratch_off) {
    __shared__ double red[kLogsumWarps][kMaxS + 1];
    const int pi = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const ProbDev& Pd = probs[pi];
    const int64_t D = Pd.n_terms;
    const int S = Pd.S;
    if (D <= 0 || S < 2) return;
    const int slices = (int)((D + kSliceSites - 1) / kSliceSites);
    const double* part = scratch + scratch_off[pi];
    for (int c = lane; c <= S; c += 32) {
        double sum = 0.0;
        for (int sl = warp; sl < slices; sl += kLogsumWarps) sum += part[(int64_t)sl * (S + 1) + c];
        red[warp][c] = sum;
    }
    __syncthreads();
    if (warp != 0) return;
    double col[3] = {0.0, 0.0, 0.0};  // columns lane, lane + 32, lane + 64 (S + 1 <= 65)
    for (int k = 0; k < 3; ++k) {
        const int c = lane + 32 * k;
        if (c <= S)
            for (int w = 0; w < kLogsumWarps; ++w) col[k] += red[w][c];
    }
    const double log_p = __shfl_sync(0xffffffffu, col[0], 0);
    // sum of the squared shift columns: this lane's in order, then across lanes
    double ss = 0.0;
    for (int k = 0; k < 3; ++k) {
        const int c = lane + 32 * k;
        if (c >= 1 && c <= S) ss = fma(col[k], col[k], ss);
    }
    ss = warp_sum_xor(ss);
    if (lane == 0) {
        ProbResult& R = Pd.res ? *Pd.res : results[pi];
        R.log_p = log_p;
        R.std_err = sqrt(ss / ((double)S * (double)(S - 1)));
        if (R.status == VECCHIA_OK && !(isfinite(log_p) && isfinite(R.std_err)))
            R.status = VECCHIA_ERR_NONFINITE;
    }
}

__global__ void init_results_kernel(ProbResult* r, int n, int* fallback_count) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        r[i].log_p = 0.0;
        r[i].std_err = 0.0;
        r[i].bad_site = LLONG_MAX;
        r[i].status = VECCHIA_OK;
        r[i].pad = 0;
    }
    if (i == 0 && fallback_count) *fallback_count = 0;
}

// ------------------------------- shifts -------------------------------------

__global__ void shifts_kernel(const uint64_t* __restrict__ seeds, const int32_t* __restrict__ Ss,
                              const int64_t* __restrict__ off, int n_probs, int dim,
                              double* __restrict__ delta, uint32_t* __restrict__ dfix) {
    const int pi = blockIdx.y;
    if (pi >= n_probs) return;
    const int S = Ss[pi];
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= S * dim) return;
    const int s = x / dim, j = x % dim;
    uint32_t c[4] = {(uint32_t)s, (uint32_t)j, 0x51A7u, 0u};
    const uint64_t seed = seeds[pi];
    philox4x32_10(c, (uint32_t)(seed & 0xffffffffu), (uint32_t)(seed >> 32));
    const uint64_t M = ((uint64_t)(c[0] >> 5) << 26) | (uint64_t)(c[1] >> 6);  // 53-bit integer
    delta[off[pi] + x] = (double)M * 0x1p-53;
    dfix[off[pi] + x] = (uint32_t)(M >> 21);
}

__global__ void eval_special_kernel(int which, const float* __restrict__ x, int64_t n,
                                    float* __restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float v = x[i];
    float e, ec, le2 = 0.0f, r = 0.0f;
    bool tiny;
    switch (which) {
        case 0: special::phi_pair(v, e, ec, tiny, le2); r = e; break;
        case 1: special::phi_pair(v, e, ec, tiny, le2); r = ec; break;
        case 2: special::phi_pair(v, e, ec, tiny, le2); r = tiny ? le2 : NAN; break;
        case 3: r = special::phiinv_pq(v, 1.0f - v); break;
        case 4: r = special::phiinv_log2(v); break;
        case 5: special::phi_pair_fast_s(v, e, ec); r = e; break;
        case 6: special::phi_pair_fast_s(v, e, ec); r = ec; break;
        case 7: r = special::phiinv16_pq(__fmul_rn(16.0f, v), __fmul_rn(16.0f, __fsub_rn(1.0f, v))); break;
        default: r = NAN;
    }
    out[i] = r;
}

// FP64 forms of the FP64 path: which = 0: Phi(x); 1: 1 - Phi(x); 2: Phi^{-1}(x)
// given p = x and q = 1 - x; 3: Phi^{-1}(1 - x) given q = x and p = 1 - x, i.e.
// -Phi^{-1}(x) taken from the upper argument.
__global__ void eval_special64_kernel(int which, const double* __restrict__ x, int64_t n,
                                      double* __restrict__ out) {
    extern __shared__ __align__(16) unsigned char tb_smem[];
    special64::Tables64& tb = *reinterpret_cast<special64::Tables64*>(tb_smem);
    special64::load_tables(tb);
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double v = x[i];
    double e, ec, r;
    switch (which) {
        case 0: special64::phi_pair(tb, v, e, ec); r = e; break;
        case 1: special64::phi_pair(tb, v, e, ec); r = ec; break;
        case 2: r = special64::phiinv_pq(tb, v, 1.0 - v); break;
        case 3: r = special64::phiinv_pq(tb, 1.0 - v, v); break;
        default: r = NAN;
    }
    out[i] = r;
}

}  // namespace

cudaError_t launch_eval_special64(int which, const double* x, int64_t n, double* out, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    eval_special64_kernel<<<(int)((n + 255) / 256), 256, sizeof(special64::Tables64), st>>>(which, x, n, out);
    return cudaGetLastError();
}

cudaError_t launch_eval_special(int which, const float* x, int64_t n, float* out, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    eval_special_kernel<<<(int)((n + 255) / 256), 256, 0, st>>>(which, x, n, out);
    return cudaGetLastError();
}

// ------------------------------- launchers ----------------------------------

namespace {

template <int DMAX, int P, int MODE>
cudaError_t launch_one(const GenzTile& tile, const ProbDev* probs, const ItemSrc& src, int max_S,
                       ProbResult* results, int* fb_count, int2* fb_items, cudaStream_t st) {
    auto kern = genz_kernel<DMAX, P, MODE>;
    constexpr bool MIXED = MODE != kModeFP64;
    constexpr int kWarpCap = max_threads(DMAX, P, MODE) / 32;
    const int warps = tile.warps < 1 ? 1 : (tile.warps > kWarpCap ? kWarpCap : tile.warps);
    const size_t smem = smem_bytes<DMAX, MIXED>(max_S < 1 ? 1 : max_S, warps);
    int dev = 0;
    cudaGetDevice(&dev);
    // occupancy per (device, warps, shared bytes); the attribute once per device
    static std::mutex mu;
    static std::map<std::tuple<int, int, size_t>, int> per_sm;
    static std::map<int, size_t> attr_set;
    int blocks_per_sm = 0;
    {
        std::lock_guard<std::mutex> lk(mu);
        auto& a = attr_set[dev];
        if (smem > 48 * 1024 && a < smem) {
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
            a = smem;
        }
        auto key = std::make_tuple(dev, warps, smem);
        auto it = per_sm.find(key);
        if (it == per_sm.end()) {
            int b = 0;
            cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kern, warps * 32, smem);
            if (e != cudaSuccess) return e;
            it = per_sm.emplace(key, b > 0 ? b : 1).first;
        }
        blocks_per_sm = it->second;
    }
    const int64_t cap = (int64_t)blocks_per_sm * device_sm_count(dev);
    ItemSrc s2 = src;
    if (!src.items && src.n_items > cap) {
        // cut the sites of the last, partial round into more shift groups (as
        // long as each piece keeps a shift per warp and the pieces fit one round)
        const int g = src.groups, n_sites = src.n_items / g;
        const int whole_sites = (int)(((int64_t)(src.n_items / cap) * cap) / g);
        const int rest = n_sites - whole_sites;
        int tg = g;
        while (rest > 0 && 2 * tg * warps <= max_S && (int64_t)rest * 2 * tg <= cap) tg *= 2;
        if (tg > g) {
            s2.whole_sites = whole_sites;
            s2.tail_groups = tg;
            s2.n_items = whole_sites * g + rest * tg;
        }
    }
    const int grid = (int)((s2.n_items < cap) ? s2.n_items : cap);
    if (grid <= 0) return cudaSuccess;
    kern<<<grid, warps * 32, smem, st>>>(probs, s2, tile.slices, max_S, results, fb_count, fb_items);
    return cudaGetLastError();
}

}  // namespace

// Built-in tile (measured on the 50x50 grid): mixed blocks of up to 32
// variables run two points per lane (one vote per step for both), FP64 one.
// Warps, mixed: 4 (above 21 variables 8 where they divide the shifts: S = 16, m =
// 30 5.89 against 5.97 ms), but where 4 would leave more than a fifth of their
// rounds idle (S = 5, 6, 9) 5 or 3 if those divide S (S = 5, m = 20: 1.34 against
// 1.59 ms; S = 6 1.52 against 1.70; S = 10 stays at 4: 2.43 against 2.55 with 5;
// idle warps of one CTA leave their issue slots to the others).  FP64: of 8 down to 4
// what keeps the most warps at work, 16 resident and the units (shifts x lattice
// slices) in rounds of w: 8 for S = 16 (55.6 against 58.2 ms with 4 at m = 20),
// 4 for 12 units (S = 6, 333 terms: 0.68 against 0.77 ms with 6).  Shift groups
// (a power of two, so S = 2^k splits evenly) until a launch has ~2048 CTA items,
// never fewer shifts per item than warps (a warp without a unit idles); ~4096 items
// for blocks of up to 16 variables, which fit more CTAs per SM.  A launch whose
// units all fit the GPU's resident warps at once gives each warp one, up to 12 warps
// a CTA: its time is one unit's chain of steps (100 terms, S = 10: call 0.239 ms in
// groups of 4 warps, 0.192 so).
// Blocks above 32 variables: 8 warps, one point per lane, every shift of a term in
// one item, so the Cholesky of up to 64 variables is shared by the most work.
GenzTile default_tile(bool mixed, int64_t total_sites, int max_S, int bucket, int sms) {
    GenzTile t;
    const int dmax = kDmaxBuckets[bucket];
    t.slices = 0;
    if (dmax > 32) {
        t.warps = 8;
        t.points = 1;
        t.groups = 1;
        return t;
    }
    const int per_shift = auto_slices(max_S, 1 << 20, mixed ? kModeFast : kModeFP64);
    const int units = max_S * per_shift;
    t.points = mixed ? 2 : 1;
    if (total_sites * units <= (int64_t)sms * 16) {
        t.groups = (units + 11) / 12;
        t.warps = (max_S + t.groups - 1) / t.groups * per_shift;
        return t;
    }
    if (!mixed) {
        double best = 0.0;
        for (int w = 8; w >= 4; --w) {
            const double rate = (double)(16 / w * w) * units / (w * ((units + w - 1) / w));
            if (rate > 1.001 * best) {
                best = rate;
                t.warps = w;
            }
        }
    } else if (dmax > 21 && max_S % 8 == 0) {
        t.warps = 8;
    } else {
        const int full = (max_S + 3) / 4 * 4;
        t.warps = 5 * max_S >= 4 * full ? 4 : max_S % 5 == 0 ? 5 : max_S % 3 == 0 ? 3 : 4;
    }
    // small blocks fit more CTAs per SM: they want more items
    const int64_t target = dmax <= 16 ? 4096 : 2048;
    int g = 1;
    while (g < max_S && (int64_t)g * total_sites < target && max_S / (2 * g) >= t.warps) g *= 2;
    t.groups = g;
    return t;
}

int default_slices(bool mixed, int S, int64_t N) { return auto_slices(S, N, mixed ? kModeFast : kModeFP64); }

cudaError_t launch_genz(int bucket, bool mixed, const GenzTile& tile, const ProbDev* probs,
                        const int* seg_prefix, const int2* seg_base, int n_segs, int n_sites,
                        ProbResult* results, int* fallback_count, int2* fallback_items, int max_S,
                        int fb_capacity, cudaStream_t st) {
    if (n_sites <= 0) return cudaSuccess;
    GenzTile t = tile;
    if (t.groups < 1) t.groups = 1;
    if (t.groups > max_S) t.groups = max_S;
    const int per_group = (max_S + t.groups - 1) / t.groups;
    while (t.slices > 1 && per_group * t.slices > kMaxUnits) --t.slices;
    ItemSrc src{nullptr, nullptr, seg_prefix, seg_base, n_segs, n_sites * t.groups, t.groups, n_sites, t.groups,
                fb_capacity};
#define VK_ARGS t, probs, src, max_S, results
#define VK_CASE(IDX, DM)                                                                         \
    case IDX:                                                                                    \
        if (!mixed) return launch_one<DM, 1, kModeFP64>(VK_ARGS, nullptr, nullptr, st);           \
        if (t.points >= 2)                                                                       \
            return launch_one<DM, 2, kModeFast>(VK_ARGS, fallback_count, fallback_items, st);    \
        return launch_one<DM, 1, kModeFast>(VK_ARGS, fallback_count, fallback_items, st);
#define VK_CASE1(IDX, DM)                                                                        \
    case IDX:                                                                                    \
        if (!mixed) return launch_one<DM, 1, kModeFP64>(VK_ARGS, nullptr, nullptr, st);           \
        return launch_one<DM, 1, kModeFast>(VK_ARGS, fallback_count, fallback_items, st);
    static_assert(kNumBuckets == 9, "bucket table");
    switch (bucket) {
        VK_CASE(0, 9)
        VK_CASE(1, 13)
        VK_CASE(2, 17)
        VK_CASE(3, 21)
        VK_CASE(4, 25)
        VK_CASE(5, 29)
        VK_CASE(6, 32)
        VK_CASE1(7, 48)
        VK_CASE1(8, 64)
        default:
            return cudaErrorInvalidValue;
    }
#undef VK_CASE
#undef VK_CASE1
#undef VK_ARGS
}

// The flagged terms: four warps a CTA (eight above 32 variables), each shift in four
// slices, several CTAs an SM, so that one term's factor runs beside the others' points;
// the last round's terms (all, where few are flagged) in shift groups over the whole
// grid.  2,500 terms, all flagged, whole call in ms, against 16 warps a term, one CTA an
// SM: m = 20, N S = 256 x 8 1.04 against 1.54, 2,048 x 8 5.46 against 5.59, 4,096 x 16 21.5
// against 21.3; about 100 flagged: 0.50 both, 2.09 against 2.08, 7.70 against 7.68.
cudaError_t launch_genz_fallback(int max_bucket, const ProbDev* probs, const int* fallback_count,
                                 const int2* fallback_items, int capacity, ProbResult* results,
                                 int max_S, cudaStream_t st) {
    if (capacity <= 0) return cudaSuccess;
    ItemSrc src{fallback_items, fallback_count, nullptr, nullptr, 0, capacity, 1, 0, 1, 0};
    if (max_bucket >= 7)  // blocks of more than 32 variables in the batch
        return launch_one<64, 1, kModeSafe>(GenzTile{8, 1, 0, 1}, probs, src, max_S, results, nullptr, nullptr, st);
    return launch_one<32, 1, kModeSafe>(GenzTile{4, 1, 0, 1}, probs, src, max_S, results, nullptr, nullptr, st);
}

cudaError_t launch_logsum(const ProbDev* probs, int n_probs, int max_slices, ProbResult* results,
                          double* const* terms, double* scratch, const int64_t* scratch_off,
                          cudaStream_t st) {
    if (n_probs <= 0 || max_slices <= 0) return cudaSuccess;
    logsum_partial_kernel<<<dim3(max_slices, n_probs), 32 * kLogsumWarps, 0, st>>>(probs, terms, scratch,
                                                                               scratch_off);
    logsum_final_kernel<<<n_probs, 32 * kLogsumWarps, 0, st>>>(probs, results, scratch, scratch_off);
    return cudaGetLastError();
}

cudaError_t launch_shifts(const uint64_t* seeds, const int32_t* S, const int64_t* out_off,
                          int n_probs, int dim, double* delta, uint32_t* dfix, cudaStream_t st) {
    if (n_probs <= 0 || dim <= 0) return cudaSuccess;
    const int per = kMaxS * dim;
    dim3 grid((per + 127) / 128, n_probs);
    shifts_kernel<<<grid, 128, 0, st>>>(seeds, S, out_off, n_probs, dim, delta, dfix);
    return cudaGetLastError();
}

cudaError_t launch_init_results(ProbResult* results, int n, int* fallback_count, cudaStream_t st) {
    const int nn = n > 1 ? n : 1;
    init_results_kernel<<<(nn + 255) / 256, 256, 0, st>>>(results, n, fallback_count);
    return cudaGetLastError();
}

}  // namespace vk
