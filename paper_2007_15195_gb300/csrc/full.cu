// full.cu -- the full D-dimensional Genz estimate of P(X < u): Genz's
// separation-of-variables recursion over all D variables at the same lattice
// points and shifts as the Vecchia terms (Sec. 2.2, Sec. 3).  It is the
// m = D - 1 limit of Eq. (vecchia-cdf) (Eq. cascading-conditional-cdf
// telescopes), the estimate the Vecchia approximation is compared against.
//
//   1. covariance Sigma (FP64, lower triangle of a D x D row-major array);
//   2. Cholesky factor, blocked right-looking in FP64: a factor of each
//      32 x 32 diagonal block, a row-wise forward substitution of the rows
//      below it, and the trailing update.  Every entry receives its terms in
//      ascending k with fma and the pivot division last: the operations of
//      the row-by-row definition in its order;
//   3. the rows of L in the recursion's form: integers of each row's scale
//      (FP64), or scaled by 1/L_vv (u likewise; mixed);
//   4. Genz's recursion.  FP64 (here), in 64-bit fixed point: CTA tiles of 64
//      lattice points, in panels of 32 variables: the panel's conditional means
//      u_v - sum_{t < v0} L_vt y_t are a register-tiled contraction of the
//      panel's rows of L with the stored y history (smem-staged chunks of 32
//      variables), then one thread per point runs the panel's variables in
//      order (the in-panel terms, Phi, the running product, Phi^{-1} of the
//      lattice-weighted probability) and appends its y values to the history.
//      Mixed: the same recursion with the contraction on the tensor cores
//      (full_tc.cu);
//   5. per-block sums of the point products, added per shift in a fixed order.
#include <climits>
#include <tuple>
#include <map>
#include <mutex>

#include "cov.cuh"
#include "exact_math.h"
#include "fix_step.cuh"
#include "full_fix_plan.h"
#include "vk_internal.h"

namespace vk {
namespace {

constexpr int kCholB = 32;   // Cholesky block
constexpr int kFullKC = 32;  // history chunk of the contraction

__global__ void full_cov_kernel(const double* __restrict__ sites, int D, CovParams cv, double* __restrict__ A) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x, r = blockIdx.y;
    if (r >= D || c > r) return;
    const double h = site_dist(cv, __dsub_rn(sites[2 * r], sites[2 * c]), __dsub_rn(sites[2 * r + 1], sites[2 * c + 1]));
    double v = cov_fn(cv.cov_kind, cv.variance, cv.range, cv.nu, h);
    if (c == r) v += cv.nugget;
    A[(int64_t)r * D + c] = v;
}

// Entry e of a packed lower triangle (e = r (r + 1) / 2 + c, c <= r).
__device__ __forceinline__ void tri_rc(int e, int& r, int& c) {
    r = (int)((sqrtf((float)(8 * e + 1)) - 1.0f) * 0.5f);
    while ((r + 1) * (r + 2) / 2 <= e) ++r;
    while (r * (r + 1) / 2 > e) --r;
    c = e - r * (r + 1) / 2;
}

// The pairs (row, column) of a packed lower triangle, in packed order: the
// pairs of an n x n triangle are the table's first n (n + 1) / 2 entries.
__device__ __forceinline__ void pair_table(unsigned short* tab) {
    for (int e = threadIdx.x; e < kCholB * (kCholB - 1) / 2; e += blockDim.x) {
        int r, c;
        tri_rc(e, r, c);
        tab[e] = (unsigned short)((r << 8) | c);
    }
}

// Factor the b x b block T in shared memory, all threads of the CTA,
// right-looking: at step j the column below the pivot is divided by it
// (exact_math.h: the same values as the FP64 square root and division by a
// shorter chain of integer instructions), then the packed trailing triangle
// takes one fma per entry, spread over the threads through the pair table.
// Warp 0 updates the next column first and goes on to its pivot while the warps of
// the other three SMSPs take the rest (an FP64 instruction holds its SMSP's pipe for
// 76 cycles, and warp 0's would queue behind theirs), so a step costs warp 0's
// chain and one barrier.  Returns the first non-positive pivot, or -1.
__device__ int factor_block(double (*T)[kCholB + 1], const unsigned short* tab, int b) {
    const int tid = threadIdx.x;
    for (int j = 0; j < b; ++j) {
        int failed = 0;
        if (tid < 32) {
            const double s = T[j][j];
            if (s > 0.0) {
                const exact::Pivot piv = exact::pivot(s);
                if (tid < b - 1 - j) T[j + 1 + tid][j] = exact::quotient(T[j + 1 + tid][j], piv);
                __syncwarp();
                if (tid == 0) T[j][j] = piv.piv;
            } else {
                failed = 1;
            }
        }
        if (__syncthreads_or(failed)) return j;  // block-uniform
        if (tid < 32) {
            if (tid < b - 1 - j) T[j + 1 + tid][j + 1] = fma(-T[j + 1 + tid][j], T[j + 1][j], T[j + 1 + tid][j + 1]);
            __syncwarp();
        } else if ((tid >> 5) & 3) {
            const int n = b - 2 - j, w = tid >> 5;
            for (int e = ((w >> 2) * 3 + (w & 3) - 1) * 32 + (tid & 31); e < n * (n + 1) / 2;
                 e += (int)blockDim.x / 4 * 3) {
                const unsigned t = tab[e];
                const int r = j + 2 + (int)(t >> 8), cc = j + 2 + (int)(t & 255u);
                T[r][cc] = fma(-T[r][j], T[cc][j], T[r][cc]);
            }
        }
    }
    __syncthreads();
    return -1;
}

// Factor the block and store it (all threads); `bad` takes its first
// non-positive pivot.
__device__ __forceinline__ void factor_store(double (*T)[kCholB + 1], const unsigned short* tab, int b,
                                             double* __restrict__ A, int D, int k0, int* __restrict__ bad) {
    const int fail = factor_block(T, tab, b);
    if (fail >= 0) {
        if (threadIdx.x == 0) atomicMin(bad, k0 + fail);
        return;
    }
    for (int e = threadIdx.x; e < b * (b + 1) / 2; e += blockDim.x) {
        int r, c;
        tri_rc(e, r, c);
        A[(int64_t)(k0 + r) * D + k0 + c] = T[r][c];
    }
}

// The diagonal block at k0, 512 threads (one trailing entry a thread at the
// first pivots, so thread 0 holds only the next pivot).  Each entry of the factor
// receives its terms in ascending order with fma and the pivot division last.
// (Tried for the
// mixed path and slower: one warp holding the block in registers and
// shuffling the columns, 49 against 26 us a block, all its FP64 work on one
// SMSP; the factor repeated by every CTA of the row solve, 70 us a block
// column, the SMs' FP64 units shared with the trailing update.)
__global__ void __launch_bounds__(512) chol_diag_kernel(double* __restrict__ A, int D, int k0,
                                                        int* __restrict__ bad) {
    __shared__ double T[kCholB][kCholB + 1];
    __shared__ unsigned short tab[kCholB * (kCholB - 1) / 2];
    const int b = min(kCholB, D - k0);
    for (int e = threadIdx.x; e < b * (b + 1) / 2; e += blockDim.x) {
        int r, c;
        tri_rc(e, r, c);
        T[r][c] = A[(int64_t)(k0 + r) * D + k0 + c];
    }
    pair_table(tab);
    __syncthreads();
    factor_store(T, tab, b, A, D, k0, bad);
}

// Mixed path, k0 >= 32: the block first takes the update by the block column
// before it (rows k0 .. k0 + 31 of that solved panel, fma in ascending column
// order), which the tensor-core update of that column leaves out, so that this
// factor waits only for the row solve of the column before and not for the
// update of its whole first tile column.  The update's 528 x 32 fma hold one SM's
// FP64 units for 6 us, so a cluster shares them: each CTA takes
// its part of the entries and leaves them in the first CTA's shared memory, and the
// first CTA factors the block.
constexpr int kDiagCluster = 4;  // (2: 7.25 ms a full estimate at D = 2,500; 4 and 8: 7.16; 1: 7.49)

__global__ void __cluster_dims__(kDiagCluster, 1, 1) __launch_bounds__(512)
    chol_diag_upd_kernel(double* __restrict__ A, int D, int k0, int* __restrict__ bad) {
    __shared__ double T[kCholB][kCholB + 1];
    __shared__ double P[kCholB][kCholB + 1];
    __shared__ unsigned short tab[kCholB * (kCholB - 1) / 2];
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    const int b = min(kCholB, D - k0), n = b * (b + 1) / 2, rank = blockIdx.x;
    // entry e: e = (warp * kDiagCluster + rank) * 32 + lane, so a rank's warps are its first ones
    const int e = ((threadIdx.x >> 5) * kDiagCluster + rank) * 32 + (threadIdx.x & 31);
    int r = 0, c = 0;
    double acc = 0.0;
    if (e < n) {
        tri_rc(e, r, c);
        acc = A[(int64_t)(k0 + r) * D + k0 + c];
    }
    for (int x = threadIdx.x; x < b * kCholB; x += blockDim.x) {
        const int pr = x / kCholB, t = x % kCholB;
        P[pr][t] = A[(int64_t)(k0 + pr) * D + k0 - kCholB + t];
    }
    if (rank == 0) pair_table(tab);
    __syncthreads();
    if (e < n) {
#pragma unroll
        for (int t = 0; t < kCholB; ++t) acc = fma(-P[r][t], P[c][t], acc);
    }
    __syncwarp();
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");  // the first CTA is resident
    if (e < n) {
        uint32_t at;
        asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(at) : "r"((uint32_t)__cvta_generic_to_shared(&T[r][c])));
        asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(at), "d"(acc) : "memory");
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (rank != 0) return;
    factor_store(T, tab, b, A, D, k0, bad);
}

// Rows r >= k0 + 32 of the block column: x L_kk^T = a by forward substitution, one
// warp per row, lane j holding x_j.  Once x_j is known it goes into every later
// lane's accumulator, so each x_k still receives its terms in ascending j with
// fma (bit for bit the row-by-row definition's sums), and each entry is divided by its
// pivot (the definition's operation: a reciprocal would change the factor's
// last bits, and with them which exactly singular block is reported; exact_math.h).
// Two warp instructions on the FP64 pipe a column instead of a thread's 528 fma:
// 7 against 41 us a block column at D = 1,021.
constexpr int kTrsmWarps = 4;
__global__ void __launch_bounds__(32 * kTrsmWarps) chol_trsm_kernel(double* __restrict__ A, int D, int k0) {
    __shared__ double T[kCholB][kCholB + 1];
    __shared__ exact::Pivot piv[kCholB];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    {  // the factored diagonal block: 8 loads a thread, issued together
        const int r = tid >> 2, c0 = (tid & 3) * 8;
        const double* src = A + (int64_t)(k0 + r) * D + k0 + c0;
        double v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = (c0 + c <= r) ? src[c] : 0.0;
#pragma unroll
        for (int c = 0; c < 8; ++c) T[r][c0 + c] = v[c];
    }
    __syncthreads();
    if (tid < kCholB) piv[tid] = exact::pivot_of(T[tid][tid]);
    __syncthreads();
    const int r = k0 + kCholB + blockIdx.x * kTrsmWarps + warp;
    if (r >= D) return;  // warp-uniform
    double* row = A + (int64_t)r * D + k0;
    double acc = row[lane];
    for (int j = 0; j < kCholB; ++j) {
        if (lane == j) acc = exact::quotient(acc, piv[j]);
        const double xj = __shfl_sync(0xffffffffu, acc, j);
        if (lane > j) acc = fma(-xj, T[lane][j], acc);
    }
    row[lane] = acc;
}

// Rows r >= k0 + 32 of the block column for the mixed path, whose trailing
// update runs on the tensor cores (chol_tc.cu): one warp per row, lane j
// holding x_j.  Step j: lane j multiplies its accumulator by the pivot's
// reciprocal, the warp shuffles x_j out and lanes k > j take fma(-x_j, L_kj, .)
// -- two FP64 warp instructions a column instead of a thread's 528 fma and 32
// divisions (GB300's FP64 unit costs the same per warp instruction however
// many lanes it carries).  The solved row then goes out for the tensor cores:
// its exponent e (|L_rt| 2^-e < 1) and the balanced base-256 digits s_0 ..
// s_6 of round(L_rt 2^(56 - e)), bf16, in the operand layout of its 8-row
// group (rel = r - k0 - 32).
constexpr int kSolveWarps = 4;
__global__ void __launch_bounds__(kSolveWarps * 32) chol_trsm_slice_kernel(double* __restrict__ A, int D, int k0,
                                                                           unsigned char* __restrict__ sl,
                                                                           int* __restrict__ ex) {
    __shared__ double T[kCholB][kCholB + 1];
    __shared__ double rinv[kCholB];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    {  // the factored diagonal block: 8 loads a thread, issued together
        const int r = tid >> 2, c0 = (tid & 3) * 8;
        const double* src = A + (int64_t)(k0 + r) * D + k0 + c0;
        double v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = (c0 + c <= r) ? src[c] : 0.0;
#pragma unroll
        for (int c = 0; c < 8; ++c) T[r][c0 + c] = v[c];
    }
    __syncthreads();
    if (tid < kCholB) rinv[tid] = 1.0 / T[tid][tid];
    __syncthreads();
    const int r = k0 + kCholB + blockIdx.x * kSolveWarps + warp;
    if (r >= D) return;  // warp-uniform
    double* row = A + (int64_t)r * D + k0;
    double acc = row[lane];
#pragma unroll
    for (int j = 0; j < kCholB; ++j) {
        if (lane == j) acc *= rinv[j];
        const double xj = __shfl_sync(0xffffffffu, acc, j);
        if (lane > j) acc = fma(-xj, T[lane][j], acc);
    }
    row[lane] = acc;
    // exponent of the row's largest entry (zeros and subnormals: the rows of
    // a zero block column, left at e = 0)
    const unsigned E = (unsigned)((__double_as_longlong(acc) >> 52) & 0x7FF);
    const unsigned Emax = __reduce_max_sync(0xffffffffu, E);
    const int e = (Emax == 0) ? 0 : max((int)Emax - 1022, -900);
    const double sc = __hiloint2double((56 - e + 1023) << 20, 0);  // 2^(56 - e)
    const int rel = r - k0 - kCholB;
    if (lane == 0) ex[rel] = e;
    long long X = __double2ll_rn(acc * sc);  // |X| <= 2^56
    int d[kCholSlices];
#pragma unroll
    for (int i = kCholSlices - 1; i >= 1; --i) {
        d[i] = (int)((X + 128) & 255) - 128;
        X = (X - d[i]) >> 8;
    }
    d[0] = (int)X;  // |d_0| <= 256
    unsigned char* grp = sl + (size_t)(rel >> 3) * kCholSliceGroupBytes + (rel & 7) * 16 + (lane >> 3) * 128 +
                         (lane & 7) * 2;
#pragma unroll
    for (int i = 0; i < kCholSlices; ++i) {
        const uint32_t h = __float_as_uint((float)d[i]) >> 16;  // exact in bf16
        const uint32_t hn = __shfl_down_sync(0xffffffffu, h, 1);
        if (!(lane & 1)) *reinterpret_cast<uint32_t*>(grp + i * 512) = h | (hn << 16);
    }
}

// Trailing update of the lower triangle below block column k0, 256 threads.
// part 0: the first tile column (the next block column, on the factor's
// critical path) in chunks of 8 rows x 32 columns, one entry per thread, so
// that it spreads over 4x more SMs; part 1: the 32 x 32 tiles (tile rows >=
// tile columns) of the tile columns after it, 4 entries per thread.
__global__ void chol_update_kernel(double* __restrict__ A, int D, int k0, int part) {
    __shared__ double Lr[kCholB][kCholB + 1], Lc[kCholB][kCholB + 1];
    const int base = k0 + kCholB;
    // rows r0 .. r0 + rows - 1 against the columns c0 .. c0 + 31
    int r0, c0, rows;
    if (part == 0) {
        r0 = base + blockIdx.x * 8;
        c0 = base;
        rows = 8;
    } else {  // tile pair (tr, tc), tc <= tr, from the linear block index
        int tr, tc;
        tri_rc(blockIdx.x, tr, tc);
        r0 = base + (tr + 1) * kCholB;
        c0 = base + (tc + 1) * kCholB;
        rows = kCholB;
    }
    for (int x = threadIdx.x; x < kCholB * kCholB; x += blockDim.x) {
        const int i = x / kCholB, t = x % kCholB;
        if (i < rows) Lr[i][t] = (r0 + i < D) ? A[(int64_t)(r0 + i) * D + k0 + t] : 0.0;
        Lc[i][t] = (c0 + i < D) ? A[(int64_t)(c0 + i) * D + k0 + t] : 0.0;
    }
    __syncthreads();
    const int j = threadIdx.x & 31;
    for (int i = threadIdx.x >> 5; i < rows; i += blockDim.x >> 5) {
        const int r = r0 + i, c = c0 + j;
        if (r >= D || c > r) continue;
        double acc = A[(int64_t)r * D + c];
#pragma unroll
        for (int t = 0; t < kCholB; ++t) acc = fma(-Lr[i][t], Lc[j][t], acc);
        A[(int64_t)r * D + c] = acc;
    }
}

// ---- the FP64 recursion, in 64-bit fixed point (fix_step.cuh) ----------------

constexpr int kFullB = 32;         // panel width
constexpr int kFullThreads = 128;
constexpr int kFullT = 4;          // per-thread tile of the contraction: 4 variables x 4 points
static_assert((kFullB / kFullT) * (kFullP / kFullT) == kFullThreads, "thread tile");

// Row v: its scale and coefficients -L_vt as digits (t < v).
__global__ void __launch_bounds__(128) full_tables_kernel(const double* __restrict__ A, const double* __restrict__ u,
                                                          int D, fix::Digits* __restrict__ Ld,
                                                          FixVar* __restrict__ var) {
    __shared__ double red[4];
    __shared__ int kL;
    const int v = blockIdx.x, tid = threadIdx.x;
    const double* row = A + (int64_t)v * D;
    double sum = 0.0;
    for (int t = tid; t < v; t += 128) sum += fabs(row[t]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if ((tid & 31) == 0) red[tid >> 5] = sum;
    __syncthreads();
    if (tid == 0) {
        const FixVar r = fix_scale(row[v], red[0] + red[1] + red[2] + red[3], u[v], v);
        var[v] = r;
        kL = r.kL;
    }
    __syncthreads();
    for (int t = tid; t < D; t += 128) Ld[(int64_t)v * D + t] = fix_coef(t < v ? row[t] : 0.0, kL);
}

struct FullArgs {
    int D;
    int64_t N;
    int S;
    int blocks_per_shift;
    const uint32_t* g;     // lattice vector, D - 1 entries
    const double* delta;   // S x dim shifts
    const double* u;       // thresholds (for NaN only: its result is NaN)
    int dim;               // row stride of delta
};

struct FullSmem {
    fix::FixTables tb;
    __align__(16) fix::Digits Ych[kFullKC][kFullP];      // chunk of the y history
    __align__(16) fix::Digits Lch[kFullB][kFullKC + 1];  // the panel's rows of L against it
    __align__(16) fix::Digits Lp[kFullB][kFullB + 1];    // the panel's own triangle
    __align__(16) int64_t Z[kFullB][kFullP];             // conditional means, then the panel's y (digits)
    FixVar var[kFullB];
    uint64_t G[kFullB], Dt[kFullB];                      // lattice multipliers and this shift, 64-bit fixed point
    double red[kFullP / 32];
    int nan;
};

// A CTA takes 64 lattice points: 192 KB of shared memory hold two CTAs an SM,
// one in its point pass (two warps, a chain of D steps) beside the other's
// contraction (four warps, 16 independent products a thread and variable).
// The contraction's D^2/2 products a point cost 25 cycles a warp instruction
// triple against the FP64 fma's 76.  (Tiles of 128 points left 152 SMs with 1 or 2
// tiles each at N S = 24,000.)  D = 1,021, N S = 24,000: 10.6 ms, D = 2,500, N S =
// 65,536: 134 ms (490 in FP64); the tensor-core form takes 3.1 and 31 ms, so this one serves the
// smallest problems and those for which the other's scratch cannot be had.
__global__ void __launch_bounds__(kFullThreads) full_genz_kernel(const fix::Digits* __restrict__ Ld,
                                                                 const FixVar* __restrict__ var, FullArgs a,
                                                                 fix::Digits* __restrict__ Y,
                                                                 double* __restrict__ part) {
    extern __shared__ __align__(16) unsigned char full_smem[];
    FullSmem& sm = *reinterpret_cast<FullSmem*>(full_smem);
    constexpr int B = kFullB, P = kFullP, KC = kFullKC, T = kFullT;
    const int tid = threadIdx.x, D = a.D;
    const uint64_t K = fix::opaque_mid();
    load_fix_tables(sm.tb);
    const int s = blockIdx.x / a.blocks_per_shift;
    const int64_t k64 = (int64_t)(blockIdx.x % a.blocks_per_shift) * P + tid;
    const bool valid = tid < P && k64 < a.N;
    const uint32_t k = (uint32_t)(valid ? k64 : a.N - 1);
    fix::Digits* Yb = Y + (int64_t)blockIdx.x * D * P;  // this tile's y history [D][P]
    const int tj = tid / (P / T), tp = tid % (P / T);   // thread tile (variables tj T.., points tp T..)
    fix::FixFloat f{~0ull, 0};
    if (tid == 0) sm.nan = 0;
    __syncthreads();
    for (int v0 = 0; v0 < D; v0 += B) {
        const int nb = min(B, D - v0);
        // the panel's constants and triangle
        for (int j = tid; j < nb; j += kFullThreads) {
            const int v = v0 + j;
            sm.var[j] = var[v];
            if (a.u[v] != a.u[v]) sm.nan = 1;
            sm.G[j] = v < D - 1 ? fix64_ratio(a.g[v], (uint64_t)a.N) : 0;
            sm.Dt[j] = v < D - 1 ? fix_shift(a.delta[(int64_t)s * a.dim + v]) : 0;
        }
        for (int x = tid; x < B * B; x += kFullThreads) {
            const int j = x / B, i = x % B;
            sm.Lp[j][i] = (j < nb && i < j) ? Ld[(int64_t)(v0 + j) * D + v0 + i] : fix::Digits{0, 0};
        }
        // conditional means from the history: Z[j][p] = u_v - sum_{t < v0} L_vt y_t[p]
        int64_t acc[T][T];
#pragma unroll
        for (int i = 0; i < T; ++i)
#pragma unroll
            for (int q = 0; q < T; ++q) acc[i][q] = 0;
        for (int t0 = 0; t0 < v0; t0 += KC) {
            __syncthreads();  // previous chunk consumed
            for (int x = tid; x < KC * P; x += kFullThreads) sm.Ych[x / P][x % P] = Yb[(int64_t)t0 * P + x];
            for (int x = tid; x < B * KC; x += kFullThreads) {
                const int j = x / KC, tt = x % KC;
                sm.Lch[j][tt] = (j < nb) ? Ld[(int64_t)(v0 + j) * D + t0 + tt] : fix::Digits{0, 0};
            }
            __syncthreads();
#pragma unroll 2
            for (int tt = 0; tt < KC; ++tt) {
                fix::Digits lv[T], yv[T];
#pragma unroll
                for (int i = 0; i < T; ++i) lv[i] = sm.Lch[tj * T + i][tt];
#pragma unroll
                for (int q = 0; q < T; ++q) yv[q] = sm.Ych[tt][tp * T + q];
#pragma unroll
                for (int i = 0; i < T; ++i)
#pragma unroll
                    for (int q = 0; q < T; ++q) acc[i][q] = fix::mul_add(lv[i], yv[q], acc[i][q], K);
            }
        }
        __syncthreads();  // the constants are in place
#pragma unroll
        for (int i = 0; i < T; ++i) {
            const int j = tj * T + i;
            const int64_t uv = (j < nb) ? sm.var[j].up : 0;
#pragma unroll
            for (int q = 0; q < T; ++q) sm.Z[j][tp * T + q] = uv + acc[i][q];
        }
        __syncthreads();
        // the panel's variables in order, one thread per point
        if (tid < P) {
            const int p = tid;
            fix::FixProb e;
            for (int j = 0; j < nb; ++j) {
                const int v = v0 + j;
                int64_t z0 = sm.Z[j][p], z1 = 0;  // two chains of the panel's own terms
                int i = 0;
                for (; i + 1 < j; i += 2) {
                    z0 = fix::mul_add(sm.Lp[j][i], reinterpret_cast<const fix::Digits&>(sm.Z[i][p]), z0, K);
                    z1 = fix::mul_add(sm.Lp[j][i + 1], reinterpret_cast<const fix::Digits&>(sm.Z[i + 1][p]), z1, K);
                }
                if (i < j) z0 = fix::mul_add(sm.Lp[j][i], reinterpret_cast<const fix::Digits&>(sm.Z[i][p]), z0, K);
                const FixVar& c = sm.var[j];
                const int64_t hi = fix::mul_add(c.rdiag, fix::digits(z0 + z1), -fix::kMulBias, K);
                fix_phi(sm.tb, hi, c.lim, c.shift, e, K);
                if (v == 0)
                    f = fix::prob(e);
                else
                    f = fix::times(f, e);
                if (v < D - 1)
                    reinterpret_cast<fix::Digits&>(sm.Z[j][p]) =
                        fix_quantile(sm.tb, (uint64_t)k * sm.G[j] + sm.Dt[j], e, K);
            }
            for (int j = 0; j < nb; ++j)
                if (v0 + j < D - 1) Yb[(int64_t)(v0 + j) * P + p] = reinterpret_cast<const fix::Digits&>(sm.Z[j][p]);
        }
        __syncthreads();  // Z and Lp reused by the next panel
    }
    // tile sum of the point products, fixed order
    double v = valid ? __longlong_as_double((long long)fix::to_bits(f)) : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (tid < P && (tid & 31) == 0) sm.red[tid >> 5] = v;
    __syncthreads();
    if (tid == 0) {
        double t = 0.0;
        for (int w = 0; w < P / 32; ++w) t += sm.red[w];
        part[blockIdx.x] = sm.nan ? __longlong_as_double(0x7ff8000000000000LL) : t;
    }
}

cudaError_t launch_full_genz_fix(const double* A, const double* u, const FullArgs& a, void* Ld, void* var, void* Y,
                                 double* part, cudaEvent_t ev_begin, cudaEvent_t ev_end, cudaStream_t st) {
    full_tables_kernel<<<a.D, 128, 0, st>>>(A, u, a.D, (fix::Digits*)Ld, (FixVar*)var);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    static std::mutex mu;
    static std::map<int, bool> attr;
    int dev = 0;
    cudaGetDevice(&dev);
    {
        std::lock_guard<std::mutex> lk(mu);
        if (!attr[dev]) {
            e = cudaFuncSetAttribute(full_genz_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sizeof(FullSmem));
            if (e != cudaSuccess) return e;
            attr[dev] = true;
        }
    }
    const int blocks = a.S * a.blocks_per_shift;
    if (ev_begin && (e = cudaEventRecord(ev_begin, st)) != cudaSuccess) return e;
    full_genz_kernel<<<blocks, kFullThreads, sizeof(FullSmem), st>>>((const fix::Digits*)Ld, (const FixVar*)var, a,
                                                                     (fix::Digits*)Y, part);
    e = cudaGetLastError();
    if (e == cudaSuccess && ev_end) e = cudaEventRecord(ev_end, st);
    return e;
}

}  // namespace

// Row solve of block column k0 (a warp a row).
void launch_trsm(double* A, int64_t D, int64_t k0, cudaStream_t st) {
    const int64_t rows = D - k0 - kCholB;
    chol_trsm_kernel<<<(unsigned)((rows + kTrsmWarps - 1) / kTrsmWarps), 32 * kTrsmWarps, 0, st>>>(A, (int)D, (int)k0);
}

// Blocked Cholesky with a one-block lookahead on two streams.  The caller's
// stream st carries the critical path: update of block column k by step k-1,
// then its diagonal factor and the rows below it; a second stream applies the
// rest of step k's trailing update meanwhile.  Every entry still receives the
// steps' terms in ascending order: the rest of step k-1 finishes before the
// first-column update of step k, and each stream keeps its own order.
size_t chol_tc_scratch_bytes(int64_t D) {
    auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
    return 2 * (al(chol_tc_slice_bytes(D)) + al(sizeof(int) * (size_t)(D + 128)));
}

// The side streams and events of one factorization (created per call, so
// that concurrent calls on other streams share nothing).
struct CholStreams {
    cudaStream_t side = nullptr, side2 = nullptr;
    cudaEvent_t ev_panel = nullptr, ev_rest[2] = {nullptr, nullptr}, ev_p0[2] = {nullptr, nullptr};
    cudaError_t create(bool tc) {
        cudaError_t e = cudaStreamCreateWithFlags(&side, cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev_panel, cudaEventDisableTiming);
        for (int i = 0; i < 2 && e == cudaSuccess; ++i) e = cudaEventCreateWithFlags(&ev_rest[i], cudaEventDisableTiming);
        if (tc) {
            if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&side2, cudaStreamNonBlocking);
            for (int i = 0; i < 2 && e == cudaSuccess; ++i) e = cudaEventCreateWithFlags(&ev_p0[i], cudaEventDisableTiming);
        }
        return e;
    }
    ~CholStreams() {  // work still queued completes first (the runtime defers the release)
        if (ev_panel) cudaEventDestroy(ev_panel);
        for (int i = 0; i < 2; ++i) {
            if (ev_rest[i]) cudaEventDestroy(ev_rest[i]);
            if (ev_p0[i]) cudaEventDestroy(ev_p0[i]);
        }
        if (side) cudaStreamDestroy(side);
        if (side2) cudaStreamDestroy(side2);
    }
};

// The blocked factor of the covariance in A (see launch_cov_chol), queued on st.
cudaError_t enqueue_chol(double* A, int64_t D, int* bad, cudaStream_t st, void* tc_scratch, int* timeout,
                         uint64_t wait_ns, CholStreams& cs) {
    cudaError_t e = cudaSuccess;
    const int64_t nblk = (D + kCholB - 1) / kCholB;
    if (nblk <= 2 || e != cudaSuccess) {  // nothing to overlap
        for (int64_t k0 = 0; k0 < D && e == cudaSuccess; k0 += kCholB) {
            chol_diag_kernel<<<1, 512, 0, st>>>(A, (int)D, (int)k0, bad);
            const int64_t rows = D - k0 - kCholB;
            if (rows > 0) {
                launch_trsm(A, D, k0, st);
                chol_update_kernel<<<(unsigned)((rows + 7) / 8), 256, 0, st>>>(A, (int)D, (int)k0, 0);
            }
            e = cudaGetLastError();
        }
        return e;
    }
    // tensor-core updates: slice buffers and exponents, one pair per parity of
    // the block column (the side stream's update of column k still reads its
    // slices while the row solve of column k + 1 writes the other pair)
    const bool tc = tc_scratch != nullptr;
    unsigned char* slb[2] = {nullptr, nullptr};
    int* exb[2] = {nullptr, nullptr};
    if (tc) {
        auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
        char* q = (char*)tc_scratch;
        for (int i = 0; i < 2; ++i) {
            slb[i] = (unsigned char*)q;
            q += al(chol_tc_slice_bytes(D));
            exb[i] = (int*)q;
            q += al(sizeof(int) * (size_t)(D + 128));
        }
    }
    cudaStream_t side = cs.side, side2 = cs.side2;
    cudaEvent_t ev_panel = cs.ev_panel;
    cudaEvent_t* ev_rest = cs.ev_rest;
    cudaEvent_t* ev_p0 = cs.ev_p0;
    if (tc && e == cudaSuccess) {
        // Critical stream: row solve of column k, then the factor of block
        // k + 1 (which applies column k's update to its own block), then the
        // solve of column k + 1 once the tensor-core update of column k + 1's
        // other rows (side2) is in.  side: the rest of the trailing update.
        chol_diag_kernel<<<1, 512, 0, st>>>(A, (int)D, 0, bad);
        for (int64_t k = 0; k < nblk && e == cudaSuccess; ++k) {
            const int64_t k0 = k * kCholB, rows = D - k0 - kCholB;
            if (rows <= 0) break;
            chol_trsm_slice_kernel<<<(unsigned)((rows + kSolveWarps - 1) / kSolveWarps), kSolveWarps * 32, 0, st>>>(
                A, (int)D, (int)k0, slb[k & 1], exb[k & 1]);
            e = cudaGetLastError();
            if (e == cudaSuccess) e = cudaEventRecord(ev_panel, st);
            const int64_t tiles = (rows + kCholB - 1) / kCholB;
            if (tiles > 1) {
                if (e == cudaSuccess) e = cudaStreamWaitEvent(side, ev_panel, 0);
                if (e == cudaSuccess)
                    e = launch_chol_update_tc(slb[k & 1], exb[k & 1], A, D, k0 + kCholB, 1, timeout, wait_ns, side);
                if (e == cudaSuccess) e = cudaEventRecord(ev_rest[k & 1], side);
            }
            // column k + 1 below its diagonal block: after the solve of k and
            // the rest of step k - 1 (launched whenever this step has rows)
            if (e == cudaSuccess) e = cudaStreamWaitEvent(side2, ev_panel, 0);
            if (k > 0 && e == cudaSuccess) e = cudaStreamWaitEvent(side2, ev_rest[(k - 1) & 1], 0);
            if (e == cudaSuccess)
                e = launch_chol_update_tc(slb[k & 1], exb[k & 1], A, D, k0 + kCholB, 0, timeout, wait_ns, side2);
            if (e == cudaSuccess) e = cudaEventRecord(ev_p0[k & 1], side2);
            // block k + 1, which the rest of step k - 1 has updated
            if (k > 0 && e == cudaSuccess) e = cudaStreamWaitEvent(st, ev_rest[(k - 1) & 1], 0);
            if (e == cudaSuccess) {
                chol_diag_upd_kernel<<<kDiagCluster, 512, 0, st>>>(A, (int)D, (int)(k0 + kCholB), bad);
                e = cudaGetLastError();
            }
            if (e == cudaSuccess) e = cudaStreamWaitEvent(st, ev_p0[k & 1], 0);
        }
    }
    for (int64_t k = 0; !tc && k < nblk && e == cudaSuccess; ++k) {
        const int64_t k0 = k * kCholB, rows = D - k0 - kCholB;
        chol_diag_kernel<<<1, 512, 0, st>>>(A, (int)D, (int)k0, bad);
        if (rows <= 0) {
            e = cudaGetLastError();
            break;
        }
        launch_trsm(A, D, k0, st);
        const int64_t tiles = (rows + kCholB - 1) / kCholB;
        if (tiles > 1) {  // the rest of step k on the side stream
            if (e == cudaSuccess) e = cudaEventRecord(ev_panel, st);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(side, ev_panel, 0);
            if (e == cudaSuccess) {
                chol_update_kernel<<<(unsigned)(tiles * (tiles - 1) / 2), 256, 0, side>>>(A, (int)D, (int)k0, 1);
                e = cudaEventRecord(ev_rest[k & 1], side);
            }
        }
        // the first column of step k needs the rest of step k - 1
        if (k > 0 && e == cudaSuccess) e = cudaStreamWaitEvent(st, ev_rest[(k - 1) & 1], 0);
        if (e == cudaSuccess) {
            chol_update_kernel<<<(unsigned)((rows + 7) / 8), 256, 0, st>>>(A, (int)D, (int)k0, 0);
            e = cudaGetLastError();
        }
    }
    // the last rest update joins the caller's stream
    if (e == cudaSuccess) {
        const int64_t last = nblk - 2;  // the last step with a trailing matrix of more than one tile
        for (int64_t k = last; k >= 0; --k)
            if ((D - k * kCholB - kCholB + kCholB - 1) / kCholB > 1) {
                e = cudaStreamWaitEvent(st, ev_rest[k & 1], 0);
                break;
            }
    }
    return e;
}

// The mixed factor's few hundred small launches and stream waits per call
// are replayed from a CUDA graph captured once per (device, D, buffers):
// queued one by one, the host needs about as long per block column as the
// GPU.  The graph is captured on a private stream (after the tensor-core
// kernel's attributes are set, outside the capture) and launched on the
// caller's, which may be the legacy default stream; on a stream the caller
// is itself capturing, the factor is queued eagerly.
namespace {
struct CholGraphKey {
    int dev;
    int64_t D;
    const void *A, *bad, *scratch, *timeout;
    uint64_t wait_ns;
    bool operator<(const CholGraphKey& o) const {
        return std::tie(dev, D, A, bad, scratch, timeout, wait_ns) <
               std::tie(o.dev, o.D, o.A, o.bad, o.scratch, o.timeout, o.wait_ns);
    }
};
std::mutex g_chol_mu;
std::map<CholGraphKey, cudaGraphExec_t> g_chol_graphs;
constexpr size_t kMaxCholGraphs = 32;
}  // namespace

cudaError_t launch_cov_chol(const double* sites, int64_t D, const vecchia_cov& cov, double* A, int* bad,
                            cudaStream_t st, void* tc_scratch, int* timeout, uint64_t wait_ns) {
    if (D <= 0) return cudaSuccess;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) dev = 0;
    full_cov_kernel<<<dim3((unsigned)((D + 127) / 128), (unsigned)D), 128, 0, st>>>(sites, (int)D, cov_params(cov), A);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const bool tc = tc_scratch != nullptr;
    const int64_t nblk = (D + kCholB - 1) / kCholB;
    bool graph = tc && nblk > 2;
    if (graph) {
        cudaStreamCaptureStatus cst = cudaStreamCaptureStatusNone;
        graph = cudaStreamIsCapturing(st, &cst) == cudaSuccess && cst == cudaStreamCaptureStatusNone;
    }
    const CholGraphKey key{dev, D, A, bad, tc_scratch, timeout, wait_ns};
    if (graph) {
        std::lock_guard<std::mutex> lk(g_chol_mu);
        auto it = g_chol_graphs.find(key);
        if (it != g_chol_graphs.end()) return cudaGraphLaunch(it->second, st);
    }
    if (tc) {
        e = chol_tc_prepare();
        if (e != cudaSuccess) return e;
    }
    CholStreams cs;
    e = cs.create(tc);
    if (e != cudaSuccess) return e;
    if (!graph) return enqueue_chol(A, D, bad, st, tc_scratch, timeout, wait_ns, cs);
    cudaGraph_t g = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaStream_t cap = nullptr;  // capture only: nothing runs on it
    e = cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        const cudaError_t eq = enqueue_chol(A, D, bad, cap, tc_scratch, timeout, wait_ns, cs);
        e = cudaStreamEndCapture(cap, &g);
        if (eq != cudaSuccess) e = eq;
    }
    if (cap) cudaStreamDestroy(cap);
    if (e == cudaSuccess) e = cudaGraphInstantiate(&exec, g, 0);
    if (g) cudaGraphDestroy(g);
    if (e != cudaSuccess) {  // not capturable here: queue it eagerly
        cudaGetLastError();
        if (exec) cudaGraphExecDestroy(exec);
        return enqueue_chol(A, D, bad, st, tc_scratch, timeout, wait_ns, cs);
    }
    {
        std::lock_guard<std::mutex> lk(g_chol_mu);
        if (g_chol_graphs.size() >= kMaxCholGraphs) {
            for (auto& kv : g_chol_graphs) cudaGraphExecDestroy(kv.second);
            g_chol_graphs.clear();
        }
        g_chol_graphs[key] = exec;
    }
    return cudaGraphLaunch(exec, st);
}

int64_t full_genz_blocks_per_shift(int64_t N, bool mixed) {
    return mixed ? full_tc_blocks_per_shift(N) : (N + kFullP - 1) / kFullP;
}

// Scratch: the shared part (factor, lattice and shift tables, block sums,
// status words) followed by the precision's own tables and y history.
// FP64 recursion: the tensor cores' contraction from kFixTcMin variables on (N S =
// 24,000: D = 64 0.08 against 0.16 ms, D = 256 0.39 against 0.94, D = 1,021 3.1
// against 10.6); the caller takes the integer form, too, where this one's scratch
// cannot be allocated.
constexpr int64_t kFixTcMin = 64;
bool full_fix_tc_pays(int64_t D) { return D >= kFixTcMin; }

size_t full_genz_scratch_bytes(int64_t D, int64_t N, int S, bool mixed, bool tc64) {
    const int64_t bps = (N + kFullP - 1) / kFullP, nblk = full_genz_blocks_per_shift(N, mixed);
    const int64_t dim = D > 1 ? D - 1 : 1;
    auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const size_t shared = al(sizeof(double) * D * D) + al(sizeof(uint32_t) * dim * 2) + al(sizeof(double) * S * dim) +
                          al(sizeof(uint32_t) * S * dim) + al(sizeof(double) * S * nblk) + al(2 * sizeof(int)) +
                          al(sizeof(uint64_t) + 2 * sizeof(int64_t) + sizeof(int32_t));
    if (mixed) return shared + al(chol_tc_scratch_bytes(D)) + full_tc_scratch_bytes(D, N, S);
    if (tc64) return shared + full_fix_tc_scratch_bytes(D, N, S);
    return shared + al(sizeof(fix::Digits) * D * D) + al(sizeof(FixVar) * D) +
           al(sizeof(fix::Digits) * (size_t)S * bps * D * kFullP);
}

cudaError_t launch_full_genz(const double* sites, const double* u, int64_t D, const vecchia_cov& cov, int64_t N,
                             int S, bool mixed, bool tc64, const uint32_t* g_host, const uint32_t* gfix_host,
                             uint64_t seed, void* scratch, double* part_host, int* bad_host, int* timeout_host,
                             uint64_t wait_ns, int withhold, cudaEvent_t ev_begin, cudaEvent_t ev_end,
                             cudaStream_t st) {
    auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
    const int64_t bps = (N + kFullP - 1) / kFullP, nblk = full_genz_blocks_per_shift(N, mixed);
    const int64_t dim = D > 1 ? D - 1 : 1;
    char* p = (char*)scratch;
    double* A = (double*)p;
    p += al(sizeof(double) * D * D);
    uint32_t* gdev = (uint32_t*)p;
    p += al(sizeof(uint32_t) * dim * 2);
    double* delta = (double*)p;
    p += al(sizeof(double) * S * dim);
    uint32_t* dfix = (uint32_t*)p;
    p += al(sizeof(uint32_t) * S * dim);
    double* part = (double*)p;
    p += al(sizeof(double) * S * nblk);
    int* bad = (int*)p;  // bad[0]: first failing pivot; bad[1]: a device wait timed out
    p += al(2 * sizeof(int));
    char* small = p;  // seed, offset, S for the shift kernel
    p += al(sizeof(uint64_t) + 2 * sizeof(int64_t) + sizeof(int32_t));
    uint64_t* seed_d = (uint64_t*)small;
    int64_t* off_d = (int64_t*)(small + sizeof(uint64_t));
    int32_t* S_d = (int32_t*)(small + sizeof(uint64_t) + 2 * sizeof(int64_t));

    const int status_init[2] = {INT_MAX, 0};
    cudaError_t e = cudaMemcpyAsync(bad, status_init, sizeof(status_init), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(gdev, g_host, sizeof(uint32_t) * dim, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(gdev + dim, gfix_host, sizeof(uint32_t) * dim, cudaMemcpyHostToDevice, st);
    const int64_t zero = 0;
    const int32_t S32 = S;
    if (e == cudaSuccess) e = cudaMemcpyAsync(seed_d, &seed, sizeof(uint64_t), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(off_d, &zero, sizeof(int64_t), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(S_d, &S32, sizeof(int32_t), cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return e;
    e = launch_shifts(seed_d, S_d, off_d, 1, (int)dim, delta, dfix, st);
    if (e != cudaSuccess) return e;
    if (mixed) {  // the factor's trailing updates on the tensor cores
        e = launch_cov_chol(sites, D, cov, A, bad, st, p, bad + 1, wait_ns);
        p += al(chol_tc_scratch_bytes(D));
    } else {
        e = launch_cov_chol(sites, D, cov, A, bad, st);
    }
    if (e != cudaSuccess) return e;
    if (mixed) {
        e = launch_full_genz_tc(A, u, D, N, S, gdev + dim, dfix, (int)dim, p, part, bad + 1, wait_ns, withhold,
                                ev_begin, ev_end, st);
    } else if (tc64) {
        e = cudaMemsetAsync(part, 0, sizeof(double) * S * nblk, st);
        if (e == cudaSuccess)
            e = launch_full_fix_tc(A, u, D, N, S, gdev, delta, (int)dim, p, part, (int)nblk, bad + 1,
                                   (withhold & 2) ? wait_ns : 0, (withhold & 2) != 0, ev_begin, ev_end, st);
    } else {
        void* Ld = p;
        p += al(sizeof(fix::Digits) * D * D);
        void* var = p;
        p += al(sizeof(FixVar) * D);
        void* Y = p;
        FullArgs fa;
        fa.D = (int)D;
        fa.N = N;
        fa.S = S;
        fa.blocks_per_shift = (int)bps;
        fa.g = gdev;
        fa.delta = delta;
        fa.u = u;
        fa.dim = (int)dim;
        e = launch_full_genz_fix(A, u, fa, Ld, var, Y, part, ev_begin, ev_end, st);
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(part_host, part, sizeof(double) * S * nblk, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(bad_host, bad, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(timeout_host, bad + 1, sizeof(int), cudaMemcpyDeviceToHost, st);
    return e;
}

}  // namespace vk
