// special_fix.h -- Genz's step in 64-bit fixed point, for the FP64 path.
//
// GB300 issues an FP64 instruction at 1/64 of its FP32 rate (76 cycles a warp
// instruction and SMSP, measured), a 32 x 32 + 64-bit integer multiply-add in
// 4 cycles.  A 64 x 64-bit product kept to its high half is three of those
// and a few additions (14-16 cycles), so a step written in 64-bit fixed point
// costs a fraction of the FP64 one at the same or better accuracy: every
// quantity below carries 57 to 64 fraction bits against FP64's 53.
//
// The step's state of a point: the conditional probability e = Phi(z) as
// FixProb, the running product f = mf 2^-64 2^-ef, and the partial sums of
// the later variables as integers in each variable's own unit.
//
//   w e        W = 2 |int64(X)| (Q0.64 tent value, within 2^-64), one product;
//   Phi^{-1}   of s = min(w e, 1 - w e): s normalised by its leading zeros,
//              interval from exponent and five mantissa bits, degree-7
//              polynomial: |y| within 2^-56 (Q6.57).  Below 2^-11 (one step in
//              1,000) s is formed anew from the operands' exponents, so it
//              keeps its relative accuracy; below 2^-32 the FP64 quantile;
//   updates    acc_j -= L_j y: L_j scaled per row to 62 bits, rounded to
//              nearest at 2^-62 of the row's largest possible sum;
//   Phi(z)     z = acc / L_vv as Q6.58, interval of width 1/64, degree-7
//              polynomial of Phi(-|z|) 2^e: relative error below 2^-55 for
//              |z| < 4, 2^-51.5 for |z| < 7, 2^-49 for |z| < 9.25.  At z >= 9.25
//              the tail t is below 2^-66 and taken as 0: it enters as 1 - t and as
//              w t beside 1 - w only, where it moves the mean of the quantiles by
//              less than 2^-60; at z <= -7 the FP64 tail.
//
// The integer code compiles for the host too (tests).  Digits: a 64-bit value
// v as hi 2^32 + lo with lo a signed 32-bit integer ("balanced"), so the three
// products of a 64 x 64 high half are signed 32 x 32 ones.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define VK_FIX_FN __host__ __device__ __forceinline__
#define VK_FIX_TABLE __device__ constexpr
#else
#define VK_FIX_FN static inline
#define VK_FIX_TABLE static const
#endif

namespace vk {
namespace fix {

struct alignas(16) FixRow {
    int64_t c0, c1, c2, c3;
    int32_t c4, c5, c6, c7;
};

#include "special_fix.cuh"

// The tables as a CTA keeps them in shared memory (copied once): the
// quantile's first ten binades (s >= 2^-11); the rest is read from global memory.
constexpr int kQShared = 10;
struct FixTables {
    FixRow quant[kQShared * kQSub];
    FixRow tail[kTRows];
    uint16_t meta[kTRows];
};

// A 64-bit value as balanced digits.
struct alignas(8) Digits {
    int32_t lo, hi;
};

VK_FIX_FN Digits digits(int64_t v) {
    Digits d;
    d.lo = (int32_t)(uint32_t)(uint64_t)v;
    d.hi = (int32_t)(v >> 32) + (int32_t)((uint32_t)d.lo >> 31);
    return d;
}

// round(a b 2^-64) + c + 2^31 (the product of the low digits dropped: below
// 1/4).  The middle products carry kMid = 2^63 + 2^31, so that their high word,
// rounded, is taken as an unsigned number (one addition with carry instead of a
// sign extension too); the callers' constants hold the -kMulBias for it.  K
// is kMid, on the device from opaque_mid(): a register pair that the compiler
// keeps, where a literal is copied into each product's addend.
constexpr uint64_t kMid = (1ull << 63) + (1ull << 31);
constexpr int64_t kMulBias = 1ll << 31;

VK_FIX_FN uint64_t opaque_mid() {
#ifdef __CUDA_ARCH__
    uint64_t K;
    asm volatile("mov.b64 %0, %1;" : "=l"(K) : "l"(kMid));
    return K;
#else
    return kMid;
#endif
}

VK_FIX_FN int64_t mul_add(Digits a, Digits b, int64_t c, uint64_t K) {
#ifdef __CUDA_ARCH__
    int64_t r;
    asm("{\n\t.reg .s64 m, h;\n\t.reg .u32 ml, mh, l, u;\n\t"
        "mad.wide.s32 m, %1, %4, %6;\n\t"
        "mad.wide.s32 m, %2, %3, m;\n\t"
        "mad.wide.s32 h, %2, %4, %5;\n\t"
        "mov.b64 {ml, mh}, m;\n\t"
        "mov.b64 {l, u}, h;\n\t"
        "add.cc.u32 l, l, mh;\n\t"
        "addc.u32 u, u, 0;\n\t"
        "mov.b64 %0, {l, u};\n\t}"
        : "=l"(r)
        : "r"(a.lo), "r"(a.hi), "r"(b.lo), "r"(b.hi), "l"(c), "l"(K));
    return r;
#else
    const uint64_t mid = (uint64_t)((int64_t)a.hi * b.lo) + ((uint64_t)((int64_t)a.lo * b.hi) + K);
    return (int64_t)((uint64_t)((int64_t)a.hi * b.hi) + (uint64_t)c + (uint32_t)(mid >> 32));
#endif
}

VK_FIX_FN int32_t mul_hi32(int32_t a, int32_t b) {
#ifdef __CUDA_ARCH__
    return __mulhi(a, b);
#else
    return (int32_t)(((int64_t)a * b) >> 32);
#endif
}

// High half of an unsigned 64 x 64 product (within 2 of it, from below).
VK_FIX_FN uint64_t umul_hi(uint64_t a, uint64_t b) {
    const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32), bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
    const uint64_t m1 = (uint64_t)ah * bl, m2 = (uint64_t)al * bh;
    return (uint64_t)ah * bh + (m1 >> 32) + (m2 >> 32);
}

VK_FIX_FN int clz32(uint32_t v) {
#ifdef __CUDA_ARCH__
    return __clz((int)v);
#else
    return v ? __builtin_clz(v) : 32;
#endif
}

VK_FIX_FN int clz64(uint64_t v) {
#ifdef __CUDA_ARCH__
    return __clzll((long long)v);
#else
    return v ? __builtin_clzll(v) : 64;
#endif
}

// c0 + c1 x + ... + c7 x^7 for x = X 2^-64, |X| <= 2^62, in the row's unit;
// the top four coefficients in 32 bits of a finer unit (2^(shift3 - 32) of it);
// the table's c0 .. c2 hold -kMulBias.
VK_FIX_FN int64_t poly(const FixRow& r, Digits X, int shift3, uint64_t K) {
    int32_t H = r.c6 + mul_hi32(r.c7, X.hi);
    H = r.c5 + mul_hi32(H, X.hi);
    H = r.c4 + mul_hi32(H, X.hi);
    int64_t P = r.c3 + (((int64_t)H * X.hi) >> shift3);
    P = mul_add(digits(P), X, r.c2, K);
    P = mul_add(digits(P), X, r.c1, K);
    return mul_add(digits(P), X, r.c0, K);
}

// v >> n for n >= 0, 0 from n = 64 on (PTX's shift clamps its amount; C++'s is undefined there).
VK_FIX_FN uint64_t shr64(uint64_t v, int n) {
#ifdef __CUDA_ARCH__
    uint64_t r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
    return r;
#else
    return n < 64 ? v >> n : 0;
#endif
}

// Phi(z): E its Q0.64 value (below 2^63 exactly where it is taken as the
// tail t = Phi(-|z|), above as 1 - t), and t = mt 2^-64 2^-et (mt = 0: none)
// for the places where E's last bit is not relative accuracy enough.
struct FixProb {
    uint64_t E, mt;
    int et;
};

// A positive number m 2^-64 2^-ex, m in [2^62, 2^64).
struct FixFloat {
    uint64_t m;
    int ex;
};

VK_FIX_FN bool is_tail(const FixProb& p) { return (p.E >> 63) == 0; }

// Phi(z) as mantissa and exponent: the tail's own below 1/2, else E.  (E's bits
// below 1/2 too would leave the mantissa unnormalised, and the product of two such
// loses the bits that umul_hi drops: 5.6e-13 at z = -3.29 twice.)
VK_FIX_FN FixFloat prob(const FixProb& p) {
    FixFloat r;
    const bool t = is_tail(p);
    r.m = t ? p.mt : p.E;
    r.ex = t ? p.et : 0;
    return r;
}

// The tent value w = 1 - |2x - 1| of x = X 2^-64 in Q0.64: 2 |int64(X)|, one
// less where X is negative (so it stays below 2^64).
VK_FIX_FN uint64_t tent(uint64_t X) {
    const uint64_t s = (uint64_t)((int64_t)X >> 63);
    return ((X ^ s) << 1) | (s & 1);
}

// f e, its mantissa normalised.
VK_FIX_FN FixFloat times(FixFloat f, const FixProb& p) {
    FixFloat e = prob(p), r;
    r.m = umul_hi(f.m, e.m);
    const int k = clz32((uint32_t)(r.m >> 32));  // f.m and e.m >= 2^62 (or 0: k = 32, the product stays 0)
    r.m <<= k;
    r.ex = f.ex + e.ex + k;
    return r;
}


// s = min(w e, 1 - w e) where it is below 2^-11, from the operands' mantissas
// and exponents: s = m 2^-64 2^-lz, m >= 2^63 (0 when s is 0).
VK_FIX_FN void small_s(uint64_t W, const FixProb& p, bool lower, uint64_t& m, int& lz) {
    uint64_t v;
    int ex;
    if (lower) {  // w e
        const bool t = is_tail(p);
        const int k = clz64(W);
        v = W ? umul_hi(W << k, t ? p.mt : p.E) : 0;
        ex = k + (t ? p.et : 0);
    } else {  // (1 - w) + w t; 1 - w = 2^64 - W > 0
        const uint64_t a = 0 - W;
        const uint64_t r = umul_hi(W, p.mt);
        const int et = p.mt ? p.et : 127;
        const int ka = clz64(a) - 1;  // W >= 2^63 here: a <= 2^63
        const int sh = ka < et ? ka : et;
        v = ((a << sh) >> (sh == et ? 1 : 0)) + (sh == et ? r >> 1 : shr64(r, et - sh));
        ex = sh - (sh == et ? 1 : 0);
    }
    const int k = clz64(v);
    m = v ? v << k : 0;
    lz = ex + k;
}

// Interval of s = m 2^-64 2^-lz (m >= 2^63, 1 <= lz <= 31) and its offset.
VK_FIX_FN int quant_row(uint64_t m, int lz, Digits& X) {
    const int row = ((lz - 1) << 5) | (int)((m >> 58) & 31);
    X = digits((int64_t)((m & ((1ull << 58) - 1)) - (1ull << 57)) << 5);
    return row;
}

// Interval of A = a 2^58, a in [0, 9.25), and its offset.
VK_FIX_FN int tail_row(uint64_t A, Digits& X) {
    X = digits((int64_t)((A & ((1ull << 52) - 1)) - (1ull << 51)) << 11);
    return (int)(A >> 52);
}

// Phi(-a) = mt 2^-64 2^-et for A = a 2^58; a >= 9.25 reads the last row.
VK_FIX_FN void tail_poly(const FixRow* rows, const uint16_t* meta, uint64_t A, uint64_t& mt, int& et, uint64_t K) {
    Digits X;
    int i = tail_row(A, X);
    i = i < kTRows ? i : kTRows - 1;
    const int w = meta[i];
    mt = (uint64_t)poly(rows[i], X, w & 255, K) << 2;
    et = w >> 8;
}

// Phi of z = hi 2^(shift - 58), lim the value of |hi| at |z| = 9.25, for z > -7; true
// where z is below that and the FP64 tail takes over.
VK_FIX_FN bool phi_of(const FixRow* rows, const uint16_t* meta, int64_t hi, int64_t lim, int shift, FixProb& e,
                      uint64_t K) {
    const int64_t neg = hi >> 63;
    const int64_t a = (hi ^ neg) - neg;
    const uint64_t A = (uint64_t)a << (shift & 63);  // |z| 2^58
    const bool big = a >= lim;
    uint64_t T;
    tail_poly(rows, meta, A, e.mt, e.et, K);
    T = shr64(e.mt, e.et);
    if (big) e.mt = T = 0;  // z >= 9.25: Phi = 1 to 2^-66
    e.E = T ^ (uint64_t)~neg;
    return hi < 0 && (big || A >= (7ull << 58));
}

// A non-negative finite double below 1 as mantissa and exponent (0: m = 0).
VK_FIX_FN FixFloat from_bits(uint64_t b) {
    FixFloat r;
    const int ex = (int)(b >> 52);
    const int k = clz64(b | 1);
    r.m = ex ? ((b & 0xfffffffffffffull) | (1ull << 52)) << 11 : b << k;
    r.ex = ex ? 1022 - ex : k + 1010;
    return r;
}

// m 2^-64 2^-ex as a double's bits, rounded to nearest (also below the normal range).
VK_FIX_FN uint64_t to_bits(FixFloat f) {
    if (f.m == 0) return 0;
    const int k = clz64(f.m);
    const uint64_t m = f.m << k;
    const int e = 1022 - f.ex - k;
    if (e > 0) return ((uint64_t)e << 52) + ((m >> 11) & 0xfffffffffffffull) + ((m >> 10) & 1);
    const int sh = 12 - e;
    return sh < 64 ? (m >> sh) + ((m >> (sh - 1)) & 1) : 0;
}

// The FixProb of t = Phi(-|z|) given as a double, neg the sign of z.
VK_FIX_FN FixProb prob_of(uint64_t t_bits, bool neg) {
    const FixFloat t = from_bits(t_bits);
    const uint64_t T = shr64(t.m, t.ex);
    FixProb p;
    p.mt = t.m;
    p.et = t.ex;
    p.E = neg ? (T >> 63 ? ~T : T) : ~T;  // z = 0: t = 1/2 either way
    return p;
}

}  // namespace fix
}  // namespace vk
