// full_fix_tc.cu -- the FP64 recursion of the full D-dimensional Genz estimate
// with its contraction on the tensor cores (Sec. 2.2, Sec. 3; the step is
// fix_step.cuh's 64-bit fixed point).
//
// The conditional means of a panel of 32 variables need sum_{t < v0} L_vt y_t at
// every point: D^2/2 products of 64-bit integers a point, which bound the integer
// form (full.cu) at 25 cycles a warp product.  Here both operands are split into eight
// balanced base-256 digits (|digit| <= 128, exact in bf16; together the 64-bit
// integer itself), and the digit products of one significance,
//     G_g = sum_{i + j = g} a_i b_j,   g = 0 .. 7,
// are accumulated by tcgen05.mma (bf16, FP32 accumulators in tensor memory) over 128
// variables at a time: at most 8 x 128 products below 2^14, so every sum is an
// integer of at most 2^24, exact in FP32.  The high half of the product is then
//     G_0 2^48 + G_1 2^40 + ... + G_6 + round(G_7 2^-8)
// in 64-bit integers; the dropped significances (i + j >= 8) are of the size of the
// integer form's own rounding (below 2 units a product, 0.2 rms, at 2^-60 of the
// row's largest possible sum).
//
// A CTA takes one or two tiles of 128 lattice points (MMA rows).  Four warps a tile, one
// thread a point, run the panels: they add the accumulators of each group of 128 variables to the points'
// sums in shared memory, run the panel's variables in order, and write their y
// as digits to the history.  One lane of another warp streams history chunks of 16
// variables (32 KB of y digits, 8 KB of the panel's L digits) with cp.async.bulk
// through a ring of three stages (two tiles: two); one lane of a further one issues 36 MMAs
// (M = 128, N = 32, K = 16) a chunk.  There are two sets of accumulators (2 x 8 x 32 columns).  With one
// tile they alternate between groups, so the MMAs run up to two groups ahead, into the next
// panel during the points' pass; only the chunks of that pass wait for it.  Two tiles
// have one set each: one's MMAs run beside the other's additions, and the passes' chains,
// twice the warps an SMSP, hide each other's latency.  Operands lie in no-swizzle K-major core matrices
// (8 rows x 16 bytes): per group of 8 rows the eight digit matrices of a chunk,
// 256 bytes each (K stride 128 bytes, row-group stride 2,048).  Every wait is bounded by
// the global timer; on expiry the kernel records a timeout, waits (bounded) for
// its copies and MMAs in flight, frees its tensor memory and returns.
//
// Bound by the points' chain of D steps (1.0 us a step) up to D of about 500, then by
// the history stream (a chunk of 40 KB a us and SM, 5 to 6 TB/s over the GPU; tensor
// pipe 12 % at D = 640): D = 1,021, N S = 24,000 3.1 ms against 10.6 in integers, D =
// 2,500, N S = 65,536 31 against 134.  (One tile a CTA: 3.5 and 33; with copies and MMAs
// from one lane, which refills a stage only after the next chunk's wait: 3.8 and 38 ms.)
#include <algorithm>
#include <map>
#include <mutex>

#include "fix_step.cuh"
#include "full_fix_plan.h"
#include "vk_internal.h"

namespace vk {
namespace {

constexpr int kXGroup = 8;     // chunks per accumulation
// H halves of 128 points a CTA (1 or 2): stages of the ring, threads (point warps, the MMA
// warp, the copy warp)
template <int H>
constexpr int kXStages = H == 1 ? 3 : 2;
template <int H>
constexpr int kXThreads = H * kXP + 64;
constexpr uint32_t kXStage = kXChunkA + kXChunkB;
constexpr uint32_t kXCols = 512;                          // 2 sets x 8 significances x 32
constexpr uint64_t kXWaitNs = 2000000000ull;

// instruction descriptor: D F32, A and B BF16, both K-major, N = 32, M = 128
constexpr uint32_t kXIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kXB >> 3) << 17) |
                             ((uint32_t)(kXP >> 4) << 24);

template <int H>
struct XSmem {
    __align__(1024) unsigned char stage[kXStages<H>][kXStage];
    fix::FixTables tb;
    __align__(16) int64_t Z[kXB][H * kXP];                // conditional sums, then the panel's y (digits)
    __align__(16) fix::Digits Lp[kXB][kXB + 1];         // the panel's own triangle
    FixVar var[kXB];
    uint64_t G[kXB], Dt[kXB];                           // lattice multipliers and this shift, 64-bit fixed point
    double red[H * kXP / 32];
    __align__(8) uint64_t full[kXStages<H>], empty[kXStages<H>], done[2], freed[2], ydone[H];
    uint32_t tmem;
    int abort, nan;
};
static_assert(sizeof(XSmem<1>) <= 227 * 1024 && sizeof(XSmem<2>) <= 227 * 1024, "one CTA's shared memory");

struct XArgs {
    int D, nP, nC;              // variables, panels, chunks of 16
    int64_t N;
    int tps;                    // CTAs per shift
    int64_t first;              // the launch's first CTA
    const uint32_t* g;          // lattice vector, D - 1 entries
    const double* delta;        // S x dim shifts
    const double* u;            // thresholds (for NaN only: its result is NaN)
    int dim;
    const FixVar* var;          // per variable (its bias counts the panel's own products)
    const unsigned char* Lb;    // digits of -L, [nP][nC] blocks of 8 KB (columns before the panel)
    const fix::Digits* Lp;      // [nP][32][32]: the panel's own triangle of -L
    unsigned char* Y;           // history digits, [the launch's tiles][nC] chunks of 32 KB
    double* part;               // per shift part_stride sums, the first H tps of them ours
    int part_stride;
    int* timeout;
    uint64_t wait_ns;
    int withhold;               // tests: the copy lane issues nothing
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t n) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(n) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_u32(b)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait; with `abort`, also given up once another thread has set it.
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, uint64_t limit_ns, const int* abort) {
    if (mbar_try(b, parity)) return true;
    const uint64_t t0 = global_ns();
    for (;;) {
        for (int i = 0; i < 16; ++i)
            if (mbar_try(b, parity)) return true;
        if (abort && *(const volatile int*)abort) return false;
        if (global_ns() - t0 > limit_ns) return false;
    }
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
// Shared-memory matrix descriptors (no swizzle, K stride 128 B, row-group stride
// 2,048 B): the high word is constant, the low one the address / 16 beside the K
// stride, so a digit matrix further on is an addition (one lane issues all MMAs: its
// instructions between them count).
constexpr uint32_t kDescHi = (kRowGroup >> 4) | (1u << 14);
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr) { return (saddr >> 4) | ((128u >> 4) << 16); }
template <bool ACC>
__device__ __forceinline__ void mma_bf16(uint32_t d, uint32_t a, uint32_t b) {
    asm volatile(
        "{\n .reg .pred p;\n .reg .b64 x, y;\n setp.ne.b32 p, %4, 0;\n mov.b64 x, {%1, %5};\n mov.b64 y, {%2, %5};\n "
        "tcgen05.mma.cta_group::1.kind::f16 [%0], x, y, %3, p;\n}" ::"r"(d),
        "r"(a), "r"(b), "r"(kXIdesc), "n"(ACC ? 1 : 0), "r"(kDescHi)
        : "memory");
}
// The 36 digit products of a chunk; FIRST starts new sums.
template <bool FIRST>
__device__ __forceinline__ void mma_chunk(uint32_t d, uint32_t a, uint32_t b) {
#pragma unroll
    for (int g = 0; g < kXDig; ++g) {
        mma_bf16<!FIRST>(d + (uint32_t)(g * kXB), a, b + (uint32_t)(g * 16));
#pragma unroll
        for (int i = 1; i <= g; ++i)
            mma_bf16<true>(d + (uint32_t)(g * kXB), a + (uint32_t)(i * 16), b + (uint32_t)((g - i) * 16));
    }
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
template <int H>
__device__ __forceinline__ void points_sync() {
    asm volatile("bar.sync 1, %0;" ::"n"(H * kXP) : "memory");
}

// The eight balanced base-256 digits of X (top digit last to leave: within +-128), as bf16 bits.
__device__ __forceinline__ void digit_bits(int64_t X, uint32_t (&d)[kXDig]) {
#pragma unroll
    for (int i = kXDig - 1; i >= 1; --i) {
        const int lo = (int)(int8_t)(uint8_t)(uint64_t)X;  // in [-128, 127]
        X = (X - lo) >> 8;
        d[i] = __float_as_uint((float)lo) >> 16;
    }
    d[0] = __float_as_uint((float)(int)X) >> 16;
}

// Row v of -L: its scale, the digits of the columns before its panel (Lb) and
// the panel's own columns (Lp).  Rows beyond D fill the last panel with zeros.
__global__ void __launch_bounds__(128) fix_tc_tables_kernel(const double* __restrict__ A, const double* __restrict__ u,
                                                            int D, int nC, FixVar* __restrict__ var,
                                                            unsigned char* __restrict__ Lb,
                                                            fix::Digits* __restrict__ Lp) {
    __shared__ double red[4];
    __shared__ int s_kL;
    const int v = blockIdx.x, tid = threadIdx.x, b = v / kXB, r = v % kXB, v0 = b * kXB;
    const double* row = A + (int64_t)min(v, D - 1) * D;
    double sum = 0.0;
    if (v < D)
        for (int t = tid; t < v; t += 128) sum += fabs(row[t]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if ((tid & 31) == 0) red[tid >> 5] = sum;
    __syncthreads();
    if (tid == 0 && v < D) {
        const FixVar f = fix_scale(row[v], red[0] + red[1] + red[2] + red[3], u[v], r);
        var[v] = f;
        s_kL = f.kL;
    }
    __syncthreads();
    const int kL = s_kL;
    for (int t = tid; t < v0; t += 128) {
        uint32_t d[kXDig];
        digit_bits(v < D ? __double2ll_rn(ldexp(-row[t], kL)) : 0ll, d);
        const int c = t / kXK, k = t % kXK;
        unsigned char* blk = Lb + ((int64_t)b * nC + c) * kXChunkB + (r / 8) * kRowGroup + (k / 8) * 128 + (r % 8) * 16 +
                             (k % 8) * 2;
#pragma unroll
        for (int i = 0; i < kXDig; ++i) *(unsigned short*)(blk + i * 256) = (unsigned short)d[i];
    }
    if (tid < kXB)
        Lp[((int64_t)b * kXB + r) * kXB + tid] =
            (v < D && v0 + tid < v) ? fix_coef(row[v0 + tid], kL) : fix::Digits{0, 0};
}

template <int H>
__device__ void give_up(const XArgs& a, XSmem<H>& sm) {
    atomicExch(&sm.abort, 1);
    atomicExch(a.timeout, 1);
}

// Accumulation n of a half (its groups counted over all panels): the accumulator set,
// and how often that set was used before.  One half alternates between the two sets, two
// halves have one each.
template <int H>
__device__ __forceinline__ int acc_set(int n, int h) { return H == 1 ? n & 1 : h; }
template <int H>
__device__ __forceinline__ uint32_t acc_use(int n) { return (uint32_t)(H == 1 ? n >> 1 : n); }

// The copies of every panel, by one lane of its own (a lane that also issued the
// MMAs refilled a stage only after the next chunk's wait): chunk c < 2 p of panel p
// once the points have written the panel that it holds and its stage is free.
template <int H>
__device__ void copy_all(const XArgs& a, XSmem<H>& sm, const unsigned char* Yt) {
    constexpr int ST = kXStages<H>;
    int il = 0, seen[H] = {};  // copies issued; panels whose y a half's points have written
    bool ok = true;
    if (a.withhold) return;
    for (int p = 1; p < a.nP && ok; ++p)
        for (int c0 = 0; c0 < 2 * p && ok; c0 += kXGroup)
#pragma unroll
            for (int h = 0; h < H; ++h)
                for (int c = c0; c < min(c0 + kXGroup, 2 * p) && ok; ++c) {
                    while (ok && seen[h] <= c / 2) {
                        ok = mbar_wait(&sm.ydone[h], (uint32_t)(seen[h] & 1), a.wait_ns, &sm.abort);
                        ++seen[h];
                    }
                    const int st = il % ST;
                    ok = ok && mbar_wait(&sm.empty[st], (uint32_t)(((il / ST) & 1) ^ 1), a.wait_ns, &sm.abort);
                    if (!ok) break;
                    mbar_expect_tx(&sm.full[st], kXStage);
                    bulk_g2s(sm.stage[st], Yt + ((int64_t)h * a.nC + c) * kXChunkA, kXChunkA, &sm.full[st]);
                    bulk_g2s(sm.stage[st] + kXChunkA, a.Lb + ((int64_t)p * a.nC + c) * kXChunkB, kXChunkB, &sm.full[st]);
                    ++il;
                }
    if (!ok) give_up(a, sm);
    // the copies in flight, bounded
    for (int i = max(0, il - ST); i < il; ++i)
        mbar_wait(&sm.full[i % ST], (uint32_t)((i / ST) & 1), kXWaitNs, nullptr);
}

// The MMAs of every panel, by one lane, in the copies' order: a group of one half, then
// the same of the other, so that one's MMAs run beside the other's additions.
template <int H>
__device__ void mma_all(const XArgs& a, XSmem<H>& sm) {
    constexpr int ST = kXStages<H>;
    const uint32_t tmem = sm.tmem;
    int im = 0, n = 0;  // chunks issued; accumulations of a half
    bool ok = true;
    for (int p = 1; p < a.nP && ok; ++p)
        for (int c0 = 0; c0 < 2 * p && ok; c0 += kXGroup, ++n)
            for (int h = 0; h < H && ok; ++h) {
                const int set = acc_set<H>(n, h);
                const uint32_t d = tmem + (uint32_t)(set * kXDig * kXB);
                ok = mbar_wait(&sm.freed[set], (acc_use<H>(n) & 1) ^ 1, a.wait_ns, &sm.abort);
                for (int c = c0; c < min(c0 + kXGroup, 2 * p); ++c) {
                    const int st = im % ST;
                    ok = ok && mbar_wait(&sm.full[st], (uint32_t)((im / ST) & 1), a.wait_ns, &sm.abort);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t da = desc_lo(smem_u32(sm.stage[st])), db = desc_lo(smem_u32(sm.stage[st]) + kXChunkA);
                    if (c == c0)
                        mma_chunk<true>(d, da, db);
                    else
                        mma_chunk<false>(d, da, db);
                    mma_commit(&sm.empty[st]);
                    ++im;
                }
                if (ok) mma_commit(&sm.done[set]);
            }
    if (!ok) give_up(a, sm);
    // the last MMAs, bounded
    if (im > 0) mbar_wait(&sm.empty[(im - 1) % ST], (uint32_t)(((im - 1) / ST) & 1), kXWaitNs, nullptr);
}

template <int H>
__global__ void __launch_bounds__(kXThreads<H>, 1) full_fix_tc_kernel(XArgs a) {
    extern __shared__ __align__(1024) unsigned char x_smem[];
    XSmem<H>& sm = *reinterpret_cast<XSmem<H>*>(x_smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, D = a.D;
    const int64_t cta = a.first + blockIdx.x;
    const int s = (int)(cta / a.tps), tile = (int)(cta % a.tps);
    constexpr int kMmaWarp = H * kXP / 32, kCopyWarp = kMmaWarp + 1;
    unsigned char* Yt = a.Y + (int64_t)blockIdx.x * H * a.nC * kXChunkA;  // its halves' histories
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sm.tmem)),
                     "r"(kXCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int i = 0; i < kXStages<H>; ++i) {
            mbar_init(&sm.full[i], 1);
            mbar_init(&sm.empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sm.done[i], 1);
            mbar_init(&sm.freed[i], kXP);
        }
        for (int h = 0; h < H; ++h) mbar_init(&sm.ydone[h], kXP);
        sm.abort = *(const volatile int*)a.timeout;  // an earlier CTA gave up: so does this one
        sm.nan = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    load_fix_tables(sm.tb);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    if (warp == kMmaWarp) {
        if (lane == 0) mma_all(a, sm);
    } else if (warp == kCopyWarp) {
        if (lane == 0) copy_all(a, sm, Yt);
    } else {
        const uint64_t K = fix::opaque_mid();
        const int64_t k64 = (int64_t)tile * (H * kXP) + tid;
        const int h = tid / kXP, row = tid % kXP;
        const bool valid = k64 < a.N;
        const uint32_t k = (uint32_t)(valid ? k64 : a.N - 1);
        const uint32_t trow = sm.tmem + ((uint32_t)((warp & 3) * 32) << 16);
        fix::FixFloat f{~0ull, 0};
        int groups = 0;
        bool failed = false;
        for (int p = 0; p < a.nP; ++p) {
            const int v0 = p * kXB, nb = min(kXB, D - v0);
            points_sync<H>();  // the last panel's constants are no longer read
            if (tid < nb) {
                const int v = v0 + tid;
                sm.var[tid] = a.var[v];
                if (a.u[v] != a.u[v]) sm.nan = 1;
                sm.G[tid] = v < D - 1 ? fix64_ratio(a.g[v], (uint64_t)a.N) : 0;
                sm.Dt[tid] = v < D - 1 ? fix_shift(a.delta[(int64_t)s * a.dim + v]) : 0;
            }
            for (int x = tid; x < kXB * kXB; x += H * kXP) sm.Lp[x / kXB][x % kXB] = a.Lp[(int64_t)p * kXB * kXB + x];
            points_sync<H>();
            for (int j = 0; j < nb; ++j) sm.Z[j][tid] = sm.var[j].up;
            // add the accumulators, 128 variables of the history at a time
            const int n_groups = (2 * p + kXGroup - 1) / kXGroup;
            for (int gi = 0; gi < n_groups; ++gi, ++groups) {
                const int set = acc_set<H>(groups, h);
                if (!failed && !mbar_wait(&sm.done[set], acc_use<H>(groups) & 1, a.wait_ns, &sm.abort)) {
                    failed = true;
                    give_up(a, sm);
                }
                if (__any_sync(0xffffffffu, failed)) {  // warp-uniform: the loads below are warp-collective
                    failed = true;
                    continue;
                }
                tc_fence_after();
                const uint32_t base = trow + (uint32_t)(set * kXDig * kXB);
#pragma unroll 1
                for (int ch = 0; ch < kXB / 8; ++ch) {
                    uint32_t G[kXDig][8];
#pragma unroll
                    for (int g = 0; g < kXDig; ++g) tmem_ld8(base + (uint32_t)(g * kXB + ch * 8), G[g]);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        int n[kXDig];  // integers of at most 2^24 held as FP32
#pragma unroll
                        for (int g = 0; g < kXDig; ++g) n[g] = __float2int_rz(__uint_as_float(G[g][j]));
                        const uint32_t top = ((uint32_t)n[0] << 16) + ((uint32_t)n[1] << 8) + (uint32_t)n[2];
                        const int64_t low = (int64_t)n[3] * (1 << 24) + ((int64_t)n[4] * (1 << 16) +
                                            ((int64_t)n[5] * (1 << 8) + (n[6] + ((n[7] + 128) >> 8))));
                        sm.Z[ch * 8 + j][tid] += (int64_t)((uint64_t)low + ((uint64_t)top << 32));
                    }
                }
                tc_fence_before();
                mbar_arrive(&sm.freed[set]);
            }
            // the panel's variables in order
            fix::FixProb e;
            for (int j = 0; j < nb; ++j) {
                const int v = v0 + j;
                int64_t z0 = sm.Z[j][tid], z1 = 0;  // two chains of the panel's own terms
                int i = 0;
                for (; i + 1 < j; i += 2) {
                    z0 = fix::mul_add(sm.Lp[j][i], reinterpret_cast<const fix::Digits&>(sm.Z[i][tid]), z0, K);
                    z1 = fix::mul_add(sm.Lp[j][i + 1], reinterpret_cast<const fix::Digits&>(sm.Z[i + 1][tid]), z1, K);
                }
                if (i < j) z0 = fix::mul_add(sm.Lp[j][i], reinterpret_cast<const fix::Digits&>(sm.Z[i][tid]), z0, K);
                const FixVar& c = sm.var[j];
                const int64_t hi = fix::mul_add(c.rdiag, fix::digits(z0 + z1), -fix::kMulBias, K);
                fix_phi(sm.tb, hi, c.lim, c.shift, e, K);
                if (v == 0)
                    f = fix::prob(e);
                else
                    f = fix::times(f, e);
                if (v < D - 1)
                    reinterpret_cast<fix::Digits&>(sm.Z[j][tid]) =
                        fix_quantile(sm.tb, (uint64_t)k * sm.G[j] + sm.Dt[j], e, K);
            }
            if (p + 1 < a.nP) {  // a full panel: its y as digits, eight variables (16 bytes a digit) at a time
                unsigned char* dst =
                    Yt + ((int64_t)h * a.nC + 2 * p) * kXChunkA + (row / 8) * kRowGroup + (row % 8) * 16;
#pragma unroll 1
                for (int o = 0; o < kXB / 8; ++o) {
                    uint32_t w[kXDig][4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        uint32_t d0[kXDig], d1[kXDig];
                        const fix::Digits y0 = reinterpret_cast<const fix::Digits&>(sm.Z[o * 8 + 2 * q][tid]);
                        const fix::Digits y1 = reinterpret_cast<const fix::Digits&>(sm.Z[o * 8 + 2 * q + 1][tid]);
                        digit_bits((int64_t)((uint64_t)(int64_t)y0.hi << 32) + y0.lo, d0);
                        digit_bits((int64_t)((uint64_t)(int64_t)y1.hi << 32) + y1.lo, d1);
#pragma unroll
                        for (int i = 0; i < kXDig; ++i) w[i][q] = d0[i] | (d1[i] << 16);
                    }
                    unsigned char* at = dst + (o >> 1) * kXChunkA + (o & 1) * 128;
#pragma unroll
                    for (int i = 0; i < kXDig; ++i)
                        *reinterpret_cast<uint4*>(at + i * 256) = make_uint4(w[i][0], w[i][1], w[i][2], w[i][3]);
                }
                asm volatile("fence.proxy.async.global;" ::: "memory");
                mbar_arrive(&sm.ydone[h]);
            }
        }
        // tile sum of the point products, fixed order
        double v = valid ? __longlong_as_double((long long)fix::to_bits(f)) : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) sm.red[warp] = v;
        points_sync<H>();
        if (row == 0) {
            double t = 0.0;
            for (int w = 0; w < kXP / 32; ++w) t += sm.red[h * (kXP / 32) + w];
            a.part[(int64_t)s * a.part_stride + (int64_t)tile * H + h] = sm.nan ? __longlong_as_double(0x7ff8000000000000LL) : t;
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == kMmaWarp)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(sm.tmem), "r"(kXCols) : "memory");
}

template <int H>
cudaError_t launch_x(const XArgs& a, int ctas, cudaStream_t st) {
    static std::mutex mu;
    static std::map<int, bool> attr;
    int dev = 0;
    cudaGetDevice(&dev);
    {
        std::lock_guard<std::mutex> lk(mu);
        if (!attr[dev]) {
            const cudaError_t e = cudaFuncSetAttribute(full_fix_tc_kernel<H>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       (int)sizeof(XSmem<H>));
            if (e != cudaSuccess) return e;
            attr[dev] = true;
        }
    }
    full_fix_tc_kernel<H><<<(unsigned)ctas, kXThreads<H>, sizeof(XSmem<H>), st>>>(a);
    return cudaGetLastError();
}

int current_sms() {
    int dev = 0;
    cudaGetDevice(&dev);
    return device_sm_count(dev);
}

size_t al(size_t b) { return (b + 255) & ~(size_t)255; }

}  // namespace

size_t full_fix_tc_scratch_bytes(int64_t D, int64_t N, int S) {
    const FullFixPlan p = full_fix_plan(D, N, S, current_sms());
    const int64_t nP = (D + kXB - 1) / kXB;
    return al(p.tables) + al(sizeof(fix::Digits) * (size_t)nP * kXB * kXB) + al(sizeof(FixVar) * D) + al(p.history);
}

cudaError_t launch_full_fix_tc(const double* A, const double* u, int64_t D, int64_t N, int S, const uint32_t* g,
                               const double* delta, int dim, void* scratch, double* part, int part_stride,
                               int* timeout, uint64_t wait_ns, bool withhold, cudaEvent_t ev_begin, cudaEvent_t ev_end,
                               cudaStream_t st) {
    const int64_t nP = (D + kXB - 1) / kXB, nC = 2 * nP;
    char* p = (char*)scratch;
    unsigned char* Lb = (unsigned char*)p;
    const FullFixPlan plan = full_fix_plan(D, N, S, current_sms());
    p += al(plan.tables);
    fix::Digits* Lp = (fix::Digits*)p;
    p += al(sizeof(fix::Digits) * (size_t)nP * kXB * kXB);
    FixVar* var = (FixVar*)p;
    p += al(sizeof(FixVar) * D);
    fix_tc_tables_kernel<<<(unsigned)(nP * kXB), 128, 0, st>>>(A, u, (int)D, (int)nC, var, Lb, Lp);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    XArgs a;
    a.D = (int)D;
    a.nP = (int)nP;
    a.nC = (int)nC;
    a.N = N;
    a.tps = (int)plan.per_shift;
    a.g = g;
    a.delta = delta;
    a.u = u;
    a.dim = dim;
    a.var = var;
    a.Lb = Lb;
    a.Lp = Lp;
    a.Y = (unsigned char*)p;
    a.part = part;
    a.part_stride = part_stride;
    a.timeout = timeout;
    a.wait_ns = (wait_ns > 0 && wait_ns < kXWaitNs) ? wait_ns : kXWaitNs;
    a.withhold = withhold;
    if (ev_begin && (e = cudaEventRecord(ev_begin, st)) != cudaSuccess) return e;
    for (a.first = 0; a.first < plan.ctas && e == cudaSuccess; a.first += plan.launch) {
        const int n = (int)std::min(plan.launch, plan.ctas - a.first);
        e = plan.halves == 2 ? launch_x<2>(a, n, st) : launch_x<1>(a, n, st);
    }
    if (e == cudaSuccess && ev_end) e = cudaEventRecord(ev_end, st);
    return e;
}

}  // namespace vk
