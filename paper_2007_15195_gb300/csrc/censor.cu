// censor.cu -- the conditional law of censored sites given observed ones, for
// the censored likelihood G_I of Sec. 4 (Eq. model05): with L the Cholesky
// factor of Sigma_II (observed sites I),
//   V_a = L^-1 Sigma_{I a}  (each censored site a),   w = L^-1 x_I,
//   mean_a = Sigma_{a I} Sigma_II^-1 x_I = V_a . w,
//   (Sigma_{c|I})_{ab} = Sigma_ab - V_a . V_b,
// so the Vecchia terms of the censored sites need only V (the Genz kernel
// subtracts V_a . V_b from each block entry) and the thresholds x_c - mean.
#include "cov.cuh"
#include "exact_math.h"
#include "vk_internal.h"

namespace vk {
namespace {

// Forward substitution, one warp per row: rows a < nc solve L v = Sigma_{I a},
// row nc solves L w = x_I.  Lane j holds entry 32 b + j of block b: it takes the
// earlier blocks' terms, then the block's own as they become final, so each
// entry still takes its terms in ascending order with fma and the pivot division
// last.  Bound by the chain of k divisions (475 rows, k = 53: 225 us with one
// thread a row, 45 us so).
constexpr int kSolveRows = 4;  // warps per CTA

__global__ void __launch_bounds__(32 * kSolveRows) cond_solve_kernel(const double* __restrict__ L, int k,
                                                                     const double* __restrict__ sites_i,
                                                                     const double* __restrict__ x_i,
                                                                     const double* __restrict__ sites_c, int nc,
                                                                     CovParams cv, double* __restrict__ V) {
    const int lane = threadIdx.x & 31;
    const int a = blockIdx.x * kSolveRows + (threadIdx.x >> 5);
    if (a > nc) return;  // warp-uniform
    double* row = V + (int64_t)a * k;
    for (int b0 = 0; b0 < k; b0 += 32) {
        const int t = b0 + lane;
        double acc = 0.0;
        if (t < k) {
            if (a < nc) {
                const double h = site_dist(cv, __dsub_rn(sites_i[2 * t], sites_c[2 * a]),
                                           __dsub_rn(sites_i[2 * t + 1], sites_c[2 * a + 1]));
                acc = cov_fn(cv.cov_kind, cv.variance, cv.range, cv.nu, h);
            } else {
                acc = x_i[t];
            }
        }
        const double* Lt = L + (int64_t)min(t, k - 1) * k;
        for (int s = 0; s < b0; ++s) acc = fma(-Lt[s], row[s], acc);
        const exact::Pivot piv = exact::pivot_of(Lt[min(t, k - 1)]);  // this lane's
        const int n = min(32, k - b0);
        for (int j = 0; j < n; ++j) {
            if (lane == j) acc = exact::quotient(acc, piv);
            const double xj = __shfl_sync(0xffffffffu, acc, j);
            if (lane > j) acc = fma(-Lt[b0 + j], xj, acc);
        }
        if (t < k) row[t] = acc;
        __syncwarp();
    }
}

__global__ void cond_mean_kernel(const double* __restrict__ V, int k, int nc, const double* __restrict__ x_c,
                                 double* __restrict__ u_out) {
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= nc) return;
    const double* va = V + (int64_t)a * k;
    const double* w = V + (int64_t)nc * k;
    double mu = 0.0;
    for (int t = 0; t < k; ++t) mu = fma(va[t], w[t], mu);
    u_out[a] = x_c[a] - mu;
}

}  // namespace

cudaError_t launch_conditioning(const double* L, int k, const double* sites_i, const double* x_i,
                                const double* sites_c, const double* x_c, int64_t nc, const vecchia_cov& cov,
                                double* V, double* u_out, cudaStream_t st) {
    if (k <= 0) return cudaSuccess;
    cond_solve_kernel<<<(unsigned)((nc + kSolveRows) / kSolveRows), 32 * kSolveRows, 0, st>>>(
        L, k, sites_i, x_i, sites_c, (int)nc, cov_params(cov), V);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess && nc > 0) {
        cond_mean_kernel<<<(unsigned)((nc + 127) / 128), 128, 0, st>>>(V, k, (int)nc, x_c, u_out);
        e = cudaGetLastError();
    }
    return e;
}

}  // namespace vk
