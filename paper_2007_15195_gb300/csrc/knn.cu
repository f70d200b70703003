// knn.cu -- conditioning sets N(i): the min(m, i) nearest previously ordered
// sites of every ordered site i (Sec. 2.1; Eq. vecchia-pdf / vecchia-cdf use
// |N_i| = min(m, i-1) in 1-based indexing).
//
// Integer work throughout, so the result is exact and reproducible:
//   - quantise: q = floor((x - xmin) * c), c = 2^30 / max extent (FP64, no
//     contraction), giving coordinates in [0, 2^30];
//   - key of a candidate j for site i: (squared quantised distance, j), so
//     distance ties go to the smaller index;
//   - bucket the sites into a (G+1) x (G+1) grid of square cells of side
//     2^(30 - log2 G) by a counting sort;
//   - one warp per site visits rings of cells of growing Chebyshev radius r
//     around the site's cell, keeping the best q keys among sites j < i in a
//     warp-wide sorted list; after ring r every unvisited site is at least
//     r*cell + 1 away in one coordinate, so the search stops once the q-th
//     best squared distance is below (r*cell + 1)^2;
//   - sites with a small index are searched by brute force over j < i.
#include <climits>
#include <map>
#include <mutex>

#include "vk_internal.h"

namespace vk {
namespace {

constexpr int kBruteLimit = 512;

struct Grid {
    double xmin, ymin, c;
    int shift;  // cell = q >> shift
    int G;      // cells per axis minus one (q = 2^30 lands in cell G)
    int zero;   // all sites equal: every coordinate quantises to 0
};

int grid_bits(int64_t D) {
    int k = 0;
    while (k < 10 && (int64_t)(2 << k) * (2 << k) <= D / 2) ++k;  // (2^(k+1))^2 <= D/2
    return k;
}

// Order-preserving integer image of a double (-0 taken as +0, as the
// comparison x < y treats them): integer compares instead of FP64 ones, which
// GB300 runs at 1/64 of its FP32 rate.
__device__ __forceinline__ unsigned long long ord_key(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x == 0.0 ? 0.0 : x);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ULL);
}
__device__ __forceinline__ double ord_value(unsigned long long k) {
    return __longlong_as_double((long long)((k >> 63) ? (k & 0x7FFFFFFFFFFFFFFFULL) : ~k));
}
__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
        v = w > v ? w : v;
    }
    return v;
}

// The grid of a bounding box given as keys: max ~x, max ~y, max x, max y.
__device__ __forceinline__ Grid box_grid(const unsigned long long (&k)[4], int gbits) {
    const double xmin = ord_value(~k[0]), ymin = ord_value(~k[1]);
    const double xmax = ord_value(k[2]), ymax = ord_value(k[3]);
    const double ex = xmax - xmin, ey = ymax - ymin;
    const double s = (ex > ey) ? ex : ey;
    Grid g;
    g.xmin = xmin;
    g.ymin = ymin;
    g.zero = !(s > 0.0);
    g.c = g.zero ? 0.0 : 1073741824.0 / s;
    g.shift = 30 - gbits;
    g.G = 1 << gbits;
    return g;
}

// Coordinates index cells, so they are kept in [0, 2^30] where the box does not
// bound them: a NaN leaves its axis out of the extent, and an extent below 2^-994
// makes c infinite.  (The host ordering's rule, too.)
__device__ __forceinline__ int2 quantise(const Grid& g, double x, double y) {
    if (g.zero) return make_int2(0, 0);
    const int qx = __double2int_rd(__dmul_rn(__dsub_rn(x, g.xmin), g.c));
    const int qy = __double2int_rd(__dmul_rn(__dsub_rn(y, g.ymin), g.c));
    return make_int2(min(max(qx, 0), 1 << 30), min(max(qy, 0), 1 << 30));
}

// Bounding box of the sites: maxima of the keys of x, y and of their
// complements (the minima), warp shuffles, then one atomic a warp and quantity;
// the last CTA to finish writes the grid.  box: four keys and a counter, all
// zero at the start.  (One CTA alone took 119 us at D = 100,000, against 10 us.)
__global__ void __launch_bounds__(256) bbox_kernel(const double* __restrict__ sites, int64_t D, int gbits,
                                                   unsigned long long* box, Grid* out) {
    unsigned long long k[4] = {0, 0, 0, 0};  // max ~x, max ~y, max x, max y
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < D; i += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long kx = ord_key(sites[2 * i]), ky = ord_key(sites[2 * i + 1]);
        k[0] = max(k[0], ~kx);
        k[1] = max(k[1], ~ky);
        k[2] = max(k[2], kx);
        k[3] = max(k[3], ky);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        k[q] = warp_max_u64(k[q]);
        if ((threadIdx.x & 31) == 0) atomicMax(&box[q], k[q]);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd((unsigned int*)(box + 4), 1u) == gridDim.x - 1) {
        __threadfence();
#pragma unroll
        for (int q = 0; q < 4; ++q) k[q] = atomicMax(&box[q], 0ULL);
        *out = box_grid(k, gbits);
    }
}

__global__ void quantize_kernel(const double* __restrict__ sites, int64_t D,
                                const Grid* __restrict__ grid, int2* __restrict__ qxy,
                                int* __restrict__ counts) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= D) return;
    const Grid g = *grid;
    const int2 q = quantise(g, sites[2 * i], sites[2 * i + 1]);
    qxy[i] = q;
    const int cell = (q.y >> g.shift) * (g.G + 1) + (q.x >> g.shift);
    atomicAdd(&counts[cell], 1);
}

// Exclusive scan of the cell counts (one CTA of 1,024 threads; the grid has at
// most 1025^2 cells): a run of cells a thread, the threads' sums by warp shuffles
// (one thread adding the 1,024 sums took 16 of the kernel's 25 us).
__global__ void __launch_bounds__(1024) scan_kernel(const int* __restrict__ counts, int n, int* __restrict__ offsets,
                                                    int* __restrict__ cursor) {
    __shared__ int part[32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int per = (n + 1023) / 1024;
    const int lo = min(n, t * per), hi = min(n, lo + per);
    int s = 0;
    for (int i = lo; i < hi; ++i) s += counts[i];
    int run = s;  // inclusive over the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, run, o);
        if (lane >= o) run += v;
    }
    if (lane == 31) part[warp] = run;
    __syncthreads();
    if (warp == 0) {
        int w = part[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += v;
        }
        part[lane] = w;
    }
    __syncthreads();
    run += (warp > 0 ? part[warp - 1] : 0) - s;  // exclusive
    if (t == 0) offsets[n] = part[31];
    for (int i = lo; i < hi; ++i) {
        offsets[i] = run;
        cursor[i] = run;
        run += counts[i];
    }
}

__global__ void scatter_kernel(const int2* __restrict__ qxy, int64_t D, const Grid* __restrict__ grid,
                               int* __restrict__ cursor, int4* __restrict__ cell_pts) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= D) return;
    const Grid g = *grid;
    const int2 q = qxy[i];
    const int cell = (q.y >> g.shift) * (g.G + 1) + (q.x >> g.shift);
    const int pos = atomicAdd(&cursor[cell], 1);
    cell_pts[pos] = make_int4(q.x, q.y, (int)i, 0);
}

// ---- warp-wide top-q list -------------------------------------------------
// A key is (squared quantised distance, index), compared lexicographically.
// The list holds the 32 K smallest keys seen so far (K = 1 or 2 keys per
// lane): element e = h 32 + lane lives in register h of that lane.
// Candidates arrive in chunks of up to 32 (one per lane): a chunk is sorted
// across lanes by a bitonic network, reversed and merged into the top of the
// list by an element-wise minimum (the 32 K smallest of the union form a
// bitonic sequence), which a bitonic clean-up sorts again.

struct Key {
    unsigned long long d2;
    int j;
};

constexpr unsigned long long kInfD2 = ~0ULL;

__device__ __forceinline__ bool key_less(const Key& a, const Key& b) {
    return a.d2 < b.d2 || (a.d2 == b.d2 && a.j < b.j);
}

__device__ __forceinline__ Key inf_key() {
    Key k;
    k.d2 = kInfD2;
    k.j = INT_MAX;
    return k;
}

__device__ __forceinline__ Key shfl_key(const Key& k, int src) {
    Key o;
    o.d2 = __shfl_sync(0xffffffffu, k.d2, src);
    o.j = __shfl_sync(0xffffffffu, k.j, src);
    return o;
}

__device__ __forceinline__ Key shfl_xor_key(const Key& k, int m) {
    Key o;
    o.d2 = __shfl_xor_sync(0xffffffffu, k.d2, m);
    o.j = __shfl_xor_sync(0xffffffffu, k.j, m);
    return o;
}

// one compare-exchange stage across lanes: partner element e ^ jm (jm < 32);
// blocks of size kb ascending (kb >= 64 * K: the whole list ascending)
__device__ __forceinline__ void cx(Key& k, int e, int kb, int jm) {
    const Key o = shfl_xor_key(k, jm);
    const bool up = (e & kb) == 0;
    const bool lower = (e & jm) == 0;
    const bool keep_min = (lower == up);
    const bool mine_less = key_less(k, o);
    if (keep_min != mine_less) k = o;
}

// the compare-exchange of elements lane and lane + 32, both in this lane
__device__ __forceinline__ void cx_in(Key& lo, Key& hi, bool ascending) {
    if (key_less(hi, lo) == ascending) {
        const Key t = lo;
        lo = hi;
        hi = t;
    }
}

__device__ __forceinline__ void bitonic_sort32(Key& k, int lane) {
#pragma unroll
    for (int kb = 2; kb <= 32; kb <<= 1)
#pragma unroll
        for (int jm = kb >> 1; jm > 0; jm >>= 1) cx(k, lane, kb, jm);
}

// ascending sort of the 64 elements (L[0] at e = lane, L[1] at e = lane + 32)
__device__ __forceinline__ void bitonic_sort64(Key (&L)[2], int lane) {
    bitonic_sort32(L[0], lane);  // first half ascending,
#pragma unroll
    for (int kb = 2; kb <= 32; kb <<= 1)  // second half descending (e & 32 set flips `up`)
#pragma unroll
        for (int jm = kb >> 1; jm > 0; jm >>= 1) cx(L[1], lane | 32, kb, jm);
    cx_in(L[0], L[1], true);  // then one bitonic merge of 64
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int jm = 16; jm > 0; jm >>= 1) cx(L[h], lane + 32 * h, 64, jm);
}

// list (ascending, 32 K elements) <- the 32 K smallest of list and chunk
template <int K>
__device__ __forceinline__ void merge_chunk(Key (&L)[K], Key c, int lane) {
    bitonic_sort32(c, lane);
    const Key rev = shfl_key(c, 31 - lane);  // descending chunk against the top 32 of the list
    if (key_less(rev, L[K - 1])) L[K - 1] = rev;
    if constexpr (K == 2) cx_in(L[0], L[1], true);
#pragma unroll
    for (int h = 0; h < K; ++h)
#pragma unroll
        for (int jm = 16; jm > 0; jm >>= 1) cx(L[h], lane + 32 * h, 128, jm);
}

__device__ __forceinline__ unsigned long long qdist2(int ax, int ay, int bx, int by) {
    const long long dx = (long long)ax - bx, dy = (long long)ay - by;
    return (unsigned long long)(dx * dx + dy * dy);
}

constexpr int kSearchWarps = 4;
// An own cell of more sites is searched by itself: 100,000 sites on a line, m = 30, 0.92 ->
// 0.71 ms; without the rule for m > 32 1.24 -> 1.31, with it 0.91.  (24 to 256 alike;
// cells of an even spread hold 2 to 8.)
constexpr int kCrowdedCell = 64;

// One warp per site i: the min(m, lim) nearest sites j < lim, lim = i
// (group 0) or the first site of i's group of `group` sites.
template <int K>
__global__ void __launch_bounds__(32 * kSearchWarps) search_kernel(
    const int2* __restrict__ qxy, int64_t D, int m, int group, const Grid* __restrict__ grid,
    const int* __restrict__ offsets, const int4* __restrict__ cell_pts, int32_t* __restrict__ nbr) {
    __shared__ Key stage[kSearchWarps][64];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t i64 = (int64_t)blockIdx.x * kSearchWarps + wid;
    if (i64 >= D) return;  // warp-uniform
    const int i = (int)i64;
    const int lim = group > 0 ? (i / group) * group : i;
    const int q = (lim < m) ? lim : m;
    int32_t* out = nbr + i64 * m;
    if (q == lim) {  // every earlier site is a neighbour
        for (int r = lane; r < m; r += 32) out[r] = (r < lim) ? r : -1;
        return;
    }
    Key L[K];
#pragma unroll
    for (int h = 0; h < K; ++h) L[h] = inf_key();
    const int2 me = qxy[i];
    Key* st = stage[wid];
    int n = 0;  // staged candidates (warp-uniform)
    auto worst = [&]() {  // element q - 1 (q is warp-uniform: no dynamic register index)
        Key src = L[0];
        if (K == 2 && q > 32) src = L[K - 1];
        return shfl_key(src, (q - 1) & 31);
    };
    Key w = inf_key();  // the current q-th best (it changes with a merge only)
    // stage the lanes' candidates that beat it; merge full chunks
    auto offer = [&](bool valid, Key k) {
        valid = valid && key_less(k, w);
        const unsigned mask = __ballot_sync(0xffffffffu, valid);
        if (valid) st[n + __popc(mask & ((1u << lane) - 1u))] = k;
        n += __popc(mask);
        __syncwarp();
        if (n >= 32) {
            merge_chunk<K>(L, st[lane], lane);
            __syncwarp();
            if (lane < n - 32) st[lane] = st[32 + lane];
            n -= 32;
            w = worst();
            __syncwarp();
        }
    };
    auto flush = [&]() {
        if (n > 0) {
            const Key c = (lane < n) ? st[lane] : inf_key();
            merge_chunk<K>(L, c, lane);
            n = 0;
            w = worst();
            __syncwarp();
        }
    };
    if (lim < kBruteLimit) {
        for (int base = 0; base < lim; base += 32) {
            const int j = base + lane;
            Key k = inf_key();
            if (j < lim) {
                const int2 o = qxy[j];
                k.d2 = qdist2(me.x, me.y, o.x, o.y);
                k.j = j;
            }
            offer(j < lim, k);
        }
        flush();
    } else {
        const Grid g = *grid;
        const int G = g.G, W = G + 1;
        const long long cs = 1LL << g.shift;
        const int cx0 = me.x >> g.shift, cy0 = me.y >> g.shift;
        // the sites of cells [xa, xb] of row cy (contiguous in cell_pts)
        auto cells = [&](int cy, int xa, int xb) {
            xa = max(xa, 0);
            xb = min(xb, G);
            if (cy < 0 || cy > G || xa > xb) return;
            const int b = offsets[cy * W + xa], e = offsets[cy * W + xb + 1];
            for (int base = b; base < e; base += 32) {
                const int p = base + lane;
                Key k = inf_key();
                bool valid = false;
                if (p < e) {
                    const int4 o = cell_pts[p];
                    valid = o.z < lim;
                    k.d2 = qdist2(me.x, me.y, o.x, o.y);
                    k.j = o.z;
                }
                offer(valid, k);
            }
        };
        // Rings 0 and 1 together (few cells hold q sites, and a merge of a part
        // chunk costs as much as a full one), a crowded own cell by itself, whose sites
        // bound the list before the others are offered; then ring by ring, each row of
        // cells as one run of candidates (100,000 sites in maxmin order, m = 30: 657 -> 400 us).
        const int own = cy0 * W + cx0;
        const bool crowded = offsets[own + 1] - offsets[own] > kCrowdedCell;
        for (int r = crowded ? 0 : 1;; ++r) {
            const bool rows = r == 0 || (r == 1 && !crowded);  // whole rows, or the ring alone
            if constexpr (K == 1) {
                if (rows) {
                    for (int cy = cy0 - r; cy <= cy0 + r; ++cy) cells(cy, cx0 - r, cx0 + r);
                } else {
                    cells(cy0 - r, cx0 - r, cx0 + r);
                    for (int cy = cy0 - r + 1; cy < cy0 + r; ++cy) {
                        cells(cy, cx0 - r, cx0 - r);
                        cells(cy, cx0 + r, cx0 + r);
                    }
                    cells(cy0 + r, cx0 - r, cx0 + r);
                }
            } else {
                // one call site, whose body is inlined once, for every run (100,000 normal sites,
                // m = 50: 0.88 ms, 1.29 with the five above; m = 30 0.70 against 0.55)
                const int runs = rows ? 2 * r + 1 : 4 * r;
                for (int t = 0; t < runs; ++t) {
                    int cy = cy0 - r + t, xa = cx0 - r, xb = cx0 + r;
                    if (!rows) {  // top and bottom, then the two ends of each row between
                        cy = t == 0 ? cy0 - r : t == 1 ? cy0 + r : cy0 - r + (t >> 1);
                        if (t > 1) xa = xb = (t & 1) ? xb : xa;
                    }
                    cells(cy, xa, xb);
                }
            }
            flush();
            if (w.d2 != kInfD2) {
                const long long bound = (long long)r * cs + 1;
                if (w.d2 < (unsigned long long)(bound * bound)) break;
            }
            if (cx0 - r <= 0 && cy0 - r <= 0 && cx0 + r >= G && cy0 + r >= G) break;
        }
    }
    // elements < q hold the q nearest; list them ascending by index (Sec. 2.2 block order)
    Key byj[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        byj[h].d2 = 0;
        byj[h].j = INT_MAX;
    }
#pragma unroll
    for (int h = 0; h < K; ++h)
        if (lane + 32 * h < q) byj[h].j = L[h].j;
    if constexpr (K == 1) {
        bitonic_sort32(byj[0], lane);
    } else {
        bitonic_sort64(byj, lane);
    }
#pragma unroll
    for (int h = 0; h < K; ++h) {
        const int r = lane + 32 * h;
        if (r < m) out[r] = (r < q) ? byj[h].j : -1;
    }
}

// Group k's conditioning row: the union of its members' rows (each ascending),
// merged by one thread with a p-way merge that drops repeats.
__global__ void group_union_kernel(const int32_t* __restrict__ per_site, int64_t D, int m, int p, int cmax,
                                   int32_t* __restrict__ cond, int32_t* __restrict__ count,
                                   int* __restrict__ overflow) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t G = (D + p - 1) / p;
    if (k >= G) return;
    const int64_t i0 = k * p;
    const int g = (int)((i0 + p < D) ? p : D - i0);
    int pos[64];
    for (int a = 0; a < g; ++a) pos[a] = 0;
    int32_t* row = cond + k * (int64_t)cmax;
    int n = 0, last = -1;
    bool over = false;
    for (;;) {
        int best = INT_MAX;
        for (int a = 0; a < g; ++a) {
            if (pos[a] < m) {
                const int v = per_site[(i0 + a) * m + pos[a]];
                if (v >= 0 && v < best) best = v;
            }
        }
        if (best == INT_MAX) break;
        for (int a = 0; a < g; ++a)  // consume every head equal to best
            if (pos[a] < m && per_site[(i0 + a) * m + pos[a]] == best) ++pos[a];
        if (best != last) {
            if (n < cmax)
                row[n] = best;
            else
                over = true;
            ++n;
            last = best;
        }
    }
    for (int r = n; r < cmax; ++r) row[r] = -1;
    if (count) count[k] = n < cmax ? n : cmax;
    if (over) atomicExch(overflow, 1);
}

// Random conditioning: Floyd's algorithm per group (one thread), then an
// insertion sort of the at most 63 indices.
__global__ void group_random_kernel(int64_t D, int p, int kk, uint64_t seed, int cmax,
                                    int32_t* __restrict__ cond, int32_t* __restrict__ count) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t G = (D + p - 1) / p;
    if (k >= G) return;
    const int64_t n = k * p;
    const int take = (int)((kk < n) ? kk : n);
    int set[64];
    int have = 0;
    for (int r = 0; r < take; ++r) {
        const int64_t j = n - take + r;
        uint32_t c[4] = {(uint32_t)k, (uint32_t)r, 0x52C5u, (uint32_t)((uint64_t)k >> 32)};
        philox4x32_10(c, (uint32_t)(seed & 0xffffffffu), (uint32_t)(seed >> 32));
        const int t = (int)(((uint64_t)c[0] * (uint64_t)(j + 1)) >> 32);
        bool dup = false;
        for (int a = 0; a < have; ++a) dup = dup || set[a] == t;
        set[have++] = dup ? (int)j : t;
    }
    for (int a = 1; a < have; ++a) {
        const int v = set[a];
        int b = a - 1;
        while (b >= 0 && set[b] > v) {
            set[b + 1] = set[b];
            --b;
        }
        set[b + 1] = v;
    }
    int32_t* row = cond + k * (int64_t)cmax;
    for (int r = 0; r < cmax; ++r) row[r] = (r < have) ? set[r] : -1;
    if (count) count[k] = have;
}

size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

__global__ void gather_kernel(const int32_t* __restrict__ perm, const double* __restrict__ sites,
                              const double* __restrict__ u, int64_t D, double* __restrict__ sites_out,
                              double* __restrict__ u_out, int* __restrict__ bad) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= D) return;
    const int32_t j = perm[k];
    if (j < 0 || j >= D) {
        atomicExch(bad, 1);
        return;
    }
    sites_out[2 * k] = sites[2 * (int64_t)j];
    sites_out[2 * k + 1] = sites[2 * (int64_t)j + 1];
    if (u) u_out[k] = u[j];
}

}  // namespace

cudaError_t launch_gather(const int32_t* perm, const double* sites, const double* u, int64_t D,
                          double* sites_out, double* u_out, int* bad, cudaStream_t st) {
    if (D <= 0) return cudaSuccess;
    gather_kernel<<<(int)((D + 255) / 256), 256, 0, st>>>(perm, sites, u, D, sites_out, u_out, bad);
    return cudaGetLastError();
}

constexpr size_t kBoxBytes = 64;  // bounding-box keys and counter

size_t knn_scratch_bytes(int64_t D) {
    const int k = grid_bits(D);
    const int64_t cells = (int64_t)((1 << k) + 1) * ((1 << k) + 1);
    return align256(sizeof(Grid)) + align256(sizeof(int2) * (size_t)D) +
           align256(kBoxBytes + sizeof(int) * (size_t)(cells + 1)) + 2 * align256(sizeof(int) * (size_t)(cells + 1)) +
           align256(sizeof(int4) * (size_t)D);
}

// The cell grid of a problem in the caller's scratch (knn_scratch_bytes(D)):
// bounding box, quantised coordinates, cell offsets and the sites sorted by cell.
struct Cells {
    Grid* grid;
    int2* qxy;
    int* offsets;
    int4* cell_pts;
};

cudaError_t build_cells(const double* sites, int64_t D, void* scratch, cudaStream_t st, Cells& out) {
    const int k = grid_bits(D);
    const int64_t cells = (int64_t)((1 << k) + 1) * ((1 << k) + 1);
    char* p = (char*)scratch;
    Grid* grid = (Grid*)p;
    p += align256(sizeof(Grid));
    int2* qxy = (int2*)p;
    p += align256(sizeof(int2) * (size_t)D);
    unsigned long long* box = (unsigned long long*)p;  // zeroed together with the counts
    int* counts = (int*)(p + kBoxBytes);
    p += align256(kBoxBytes + sizeof(int) * (size_t)(cells + 1));
    int* offsets = (int*)p;
    p += align256(sizeof(int) * (size_t)(cells + 1));
    int* cursor = (int*)p;
    p += align256(sizeof(int) * (size_t)(cells + 1));
    int4* cell_pts = (int4*)p;
    out = Cells{grid, qxy, offsets, cell_pts};
    cudaError_t e = cudaMemsetAsync(box, 0, kBoxBytes + sizeof(int) * (size_t)cells, st);
    if (e != cudaSuccess) return e;
    const int blocks = (int)((D + 255) / 256);
    bbox_kernel<<<blocks < 128 ? blocks : 128, 256, 0, st>>>(sites, D, k, box, grid);
    quantize_kernel<<<blocks, 256, 0, st>>>(sites, D, grid, qxy, counts);
    scan_kernel<<<1, 1024, 0, st>>>(counts, (int)cells, offsets, cursor);
    scatter_kernel<<<blocks, 256, 0, st>>>(qxy, D, grid, cursor, cell_pts);
    return cudaGetLastError();
}

// Up to kSmallMax sites, one CTA, a thread a site: bounding box and quantised
// coordinates (to qxy) and, with ORDER, first the XY order (each site's rank
// counts the smaller keys) and the gather of sites and thresholds.  Every search
// of such a problem is by brute force, so the cell grid is not built: one launch
// of 9 us in place of four to ten (100 sites: 35 us of kernels, and their gaps).
static_assert(kSmallMax <= kBruteLimit, "small problems need no cell grid");

template <bool ORDER>
__global__ void __launch_bounds__((int)kSmallMax) small_kernel(const double* __restrict__ sites,
                                                               const double* __restrict__ u, int D,
                                                               int32_t* __restrict__ perm,
                                                               double* __restrict__ sites_out,
                                                               double* __restrict__ u_out, int2* __restrict__ qxy) {
    __shared__ unsigned long long kx[kSmallMax], ky[kSmallMax];
    __shared__ unsigned long long part[4][kSmallMax / 32];
    __shared__ Grid grid;
    const int i = threadIdx.x, lane = i & 31, warp = i >> 5, nw = blockDim.x >> 5;
    const bool in = i < D;
    const double x = in ? sites[2 * i] : 0.0, y = in ? sites[2 * i + 1] : 0.0;
    const unsigned long long mx = ord_key(x), my = ord_key(y);
    unsigned long long k[4] = {in ? ~mx : 0, in ? ~my : 0, in ? mx : 0, in ? my : 0};
    if (ORDER && in) {
        kx[i] = mx;
        ky[i] = my;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        k[q] = warp_max_u64(k[q]);
        if (lane == 0) part[q][warp] = k[q];
    }
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int q = 0; q < 4; ++q) k[q] = warp_max_u64(lane < nw ? part[q][lane] : 0ULL);
        if (lane == 0) grid = box_grid(k, 0);
    }
    int rank = i;
    if (ORDER && in) {
        rank = 0;
        for (int j = 0; j < D; ++j) {
            const unsigned long long xj = kx[j], yj = ky[j];
            rank += (xj < mx) || (xj == mx && (yj < my || (yj == my && j < i)));
        }
        perm[rank] = i;
        sites_out[2 * rank] = x;
        sites_out[2 * rank + 1] = y;
        if (u) u_out[rank] = u[i];
    }
    __syncthreads();
    if (in) qxy[rank] = quantise(grid, x, y);
}

int small_threads(int64_t D) { return (int)((D + 31) / 32 * 32); }

template <int K>
void run_search(const Cells& c, int64_t D, int m, int group, int32_t* nbr, cudaStream_t st) {
    const int blocks = (int)((D + kSearchWarps - 1) / kSearchWarps);
    search_kernel<K><<<blocks, 32 * kSearchWarps, 0, st>>>(c.qxy, D, m, group, c.grid, c.offsets, c.cell_pts, nbr);
}

cudaError_t launch_order_small(const double* sites, const double* u, int64_t D, int32_t* perm, double* sites_out,
                               double* u_out, void* scratch, cudaStream_t st) {
    small_kernel<true><<<1, small_threads(D), 0, st>>>(sites, u, (int)D, perm, sites_out, u_out, (int2*)scratch);
    return cudaGetLastError();
}

cudaError_t launch_knn_small(int64_t D, int m, int32_t* nbr, void* scratch, cudaStream_t st) {
    const Cells c{nullptr, (int2*)scratch, nullptr, nullptr};
    m <= 32 ? run_search<1>(c, D, m, 0, nbr, st) : run_search<2>(c, D, m, 0, nbr, st);
    return cudaGetLastError();
}

cudaError_t launch_knn(const double* sites, int64_t D, int m, int32_t* nbr, void* scratch,
                       cudaStream_t st, int group) {
    if (D <= 0 || m <= 0) return cudaSuccess;
    Cells c{nullptr, (int2*)scratch, nullptr, nullptr};
    if (D <= kSmallMax) {
        small_kernel<false><<<1, small_threads(D), 0, st>>>(sites, nullptr, (int)D, nullptr, nullptr, nullptr, c.qxy);
    } else {
        const cudaError_t e = build_cells(sites, D, scratch, st, c);
        if (e != cudaSuccess) return e;
    }
    m <= 32 ? run_search<1>(c, D, m, group, nbr, st) : run_search<2>(c, D, m, group, nbr, st);
    return cudaGetLastError();
}

// ---- device sort of unique keys (ordering) ----------------------------------
// Ascending by (a, b, idx): tiles of 2,048 by a bitonic network in shared
// memory, then passes that merge pairs of runs, each element finding its place
// by a binary search in the sibling run (keys are unique through idx, so every
// place is taken once).  A pass moves 12-20 bytes an element and is bound by
// the 11-17 dependent loads of its search: 3 us a pass at D = 100,000.

constexpr int kSortTile = 2048;

struct SortRun {
    unsigned long long* a;
    unsigned long long* b;  // nullptr: keys of one word
    int* idx;
};

template <bool TWO>
__device__ __forceinline__ bool sort_less(unsigned long long a0, unsigned long long b0, int i0,
                                          unsigned long long a1, unsigned long long b1, int i1) {
    if (a0 != a1) return a0 < a1;
    if (TWO && b0 != b1) return b0 < b1;
    return i0 < i1;
}

// Sorts tile blockIdx.x of keys loaded by KEYS; writes to out, or (a single tile) the indices to perm.
template <bool TWO, class KEYS>
__global__ void __launch_bounds__(kSortTile / 2) sort_tile_kernel(KEYS keys, int D, SortRun out, int32_t* perm) {
    __shared__ unsigned long long sa[kSortTile], sb[TWO ? kSortTile : 1];
    __shared__ int si[kSortTile];
    const int base = blockIdx.x * kSortTile;
    for (int t = threadIdx.x; t < kSortTile; t += blockDim.x) {
        unsigned long long a = ~0ull, b = ~0ull;
        int i = INT_MAX;  // beyond the end: after every key
        if (base + t < D) keys.load(base + t, a, b, i);
        sa[t] = a;
        if (TWO) sb[t] = b;
        si[t] = i;
    }
    for (int kb = 2; kb <= kSortTile; kb <<= 1)
        for (int jm = kb >> 1; jm > 0; jm >>= 1) {
            __syncthreads();
            const int t = threadIdx.x, lo = ((t & ~(jm - 1)) << 1) | (t & (jm - 1)), hi = lo | jm;
            const bool up = (lo & kb) == 0;
            const unsigned long long a0 = sa[lo], a1 = sa[hi], b0 = TWO ? sb[lo] : 0, b1 = TWO ? sb[hi] : 0;
            const int i0 = si[lo], i1 = si[hi];
            if (sort_less<TWO>(a1, b1, i1, a0, b0, i0) == up) {
                sa[lo] = a1;
                sa[hi] = a0;
                if (TWO) {
                    sb[lo] = b1;
                    sb[hi] = b0;
                }
                si[lo] = i1;
                si[hi] = i0;
            }
        }
    __syncthreads();
    for (int t = threadIdx.x; t < kSortTile && base + t < D; t += blockDim.x) {
        if (perm) {
            perm[base + t] = si[t];
        } else {
            out.a[base + t] = sa[t];
            if (TWO) out.b[base + t] = sb[t];
            out.idx[base + t] = si[t];
        }
    }
}

// Merges runs of length w in pairs; the last pass writes the indices to perm.
template <bool TWO>
__global__ void sort_merge_kernel(SortRun in, SortRun out, int D, int64_t w, int32_t* perm) {
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= D) return;
    const int64_t run = g / w, mine = run * w, other = (run ^ 1) * w;
    const unsigned long long a = in.a[g], b = TWO ? in.b[g] : 0;
    const int i = in.idx[g];
    int64_t lo = other < D ? other : D, hi = other + w < D ? other + w : D;
    const int64_t o0 = lo;
    while (lo < hi) {  // first element of the sibling run that is not before this key
        const int64_t mid = (lo + hi) >> 1;
        if (sort_less<TWO>(in.a[mid], TWO ? in.b[mid] : 0, in.idx[mid], a, b, i))
            lo = mid + 1;
        else
            hi = mid;
    }
    const int64_t dst = (mine < other ? mine : other) + (g - mine) + (lo - o0);
    if (perm) {
        perm[dst] = i;
    } else {
        out.a[dst] = a;
        if (TWO) out.b[dst] = b;
        out.idx[dst] = i;
    }
}

// r: two sets of D entries, the first of which may lie where KEYS reads its own
// (a tile is read whole before it is written).
template <bool TWO, class KEYS>
cudaError_t launch_sort(KEYS keys, int64_t D, int32_t* perm, const SortRun (&r)[2], cudaStream_t st) {
    const int tiles = (int)((D + kSortTile - 1) / kSortTile);
    sort_tile_kernel<TWO><<<tiles, kSortTile / 2, 0, st>>>(keys, (int)D, r[0], tiles == 1 ? perm : nullptr);
    int cur = 0;
    for (int64_t w = kSortTile; w < D; w *= 2, cur ^= 1)
        sort_merge_kernel<TWO><<<(unsigned)((D + 255) / 256), 256, 0, st>>>(r[cur], r[cur ^ 1], (int)D, w,
                                                                         2 * w >= D ? perm : nullptr);
    return cudaGetLastError();
}

// ---- exact maxmin ordering (one thread-block cluster, or grid-wide rounds) ------
// Same rule as the host ordering: first the site nearest the centre of the
// quantised bounding box (2q - qmax, smallest squared distance, ties to the
// smaller index), then repeatedly the unchosen site whose squared distance to
// the chosen set is largest (ties to the smaller index).
//
// The picks need not be made one at a time.  Let mind_i be site i's squared
// distance to the chosen set and key_i = (mind_i, -i).  Picking a site only
// lowers keys, so the picks' keys decrease strictly, and the ordering is the
// sites sorted by the key each has when it is picked.  Site i's key is final as
// soon as no unchosen site of larger key lies closer than mind_i to it: only a
// site picked before i, hence of larger key now, could lower mind_i, and only
// from within that distance.  So each round takes every site whose key is final
// (the locally dominant ones), records the key, and lowers mind in their
// surroundings; about 15 to 20 rounds order any even spread of sites (n sites in
// a round allow a fixed fraction of n in the next).  A pick p lowers mind_j only
// where key_j < key_p: a j of larger key comes before p in the ordering (and
// whenever that holds, d(j, p) >= mind_p, so p is no nearer to j than what j has
// by the time its key falls below p's).  The first kMmSerial picks, whose reach
// spans most sites, are made one at a time by all threads; a sort of the
// recorded keys ends it.  Each unchosen site keeps a witness (a site that
// dominates it) from round to round and searches anew only once that one no
// longer does; the search is per thread over the 3 x 3 cells around the site,
// where it nearly always ends, and by the whole warp over the reach otherwise.
//
// Below kMmGridWide sites one cluster of up to 16 CTAs runs it all: a round's two
// barriers are the hardware's cluster barrier, and there are no spin-waits.  From
// there on (0.53 against 0.75 ms at 6,000 sites, 0.95 against 2.8 ms at 100,000)
// the first kMmRounds rounds are launches over the whole GPU, which do nothing
// once every site is taken, and the cluster does what rounds remain.  Bound by
// the latency of the dependent L2 loads (witness, its mind; cell, its sites,
// their minds): a late round of 20 us moves a few MB.  A
// serial pick took 5 to 7 us (one CTA: scan, tournament tree).  Whole call: D =
// 100,000 705 -> 0.95 ms, 20,011 116 -> 0.60 ms, 2,048 9.7 -> 0.53 ms, 100
// 0.47 -> 0.16 ms; 8,000 sites crowded about a point 127 -> 16 ms.

constexpr int kMmThreads = 1024;
constexpr int kMmSerial = 32;  // (D = 100,000: 1.07 ms with 16, 0.96 with 32, 1.05 with 64)
constexpr int kMmMaxCluster = 16;
constexpr int kMmRounds = 16;        // grid-wide rounds
constexpr int64_t kMmGridWide = 6000;  // from this many sites on

struct MmSlot {
    long long v, w;
    int s, pad;
};

struct MmState {
    const int4* pts;     // sites sorted by cell: (qx, qy, index, -); the arrays below go by that position
    const int* offsets;  // cell starts
    long long* mind;     // squared distance to the chosen set, -1 once chosen
    long long* key;      // mind when chosen
    int* wit;            // witness, or -1
    int* list;           // the round's picks
    int* count;          // their number: rounds of the cluster mod 3, then the grid-wide rounds
    MmSlot* slot;        // per CTA (two sets, alternating)
};

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ bool mm_better(long long va, int ia, long long vb, int ib) {
    return va > vb || (va == vb && ia < ib);
}

// Cells within reach of a site: |dx|, |dy| < rr for d^2 < m.
struct MmReach {
    int xl, xh, yl, yh;
};
__device__ __forceinline__ MmReach mm_reach(const Grid& g, int x, int y, long long m) {
    // sqrt from above: FP32 rounding is below 1e-6 relative
    const long long rr = m == LLONG_MAX ? (1LL << 31) : (long long)(sqrtf((float)m) * 1.000001f) + 2;
    MmReach r;
    r.xl = (int)(max(0LL, (long long)x - rr) >> g.shift);
    r.yl = (int)(max(0LL, (long long)y - rr) >> g.shift);
    r.xh = (int)min((long long)g.G, ((long long)x + rr) >> g.shift);
    r.yh = (int)min((long long)g.G, ((long long)y + rr) >> g.shift);
    return r;
}

__device__ __forceinline__ long long mm_d2(const int4& a, const int4& b) {
    const long long dx = (long long)a.x - b.x, dy = (long long)a.y - b.y;
    return dx * dx + dy * dy;
}

// Site q (mind mq) keeps site p's key open: larger key, closer than mind_p.
__device__ __forceinline__ bool mm_dominates(const int4& q, long long mq, const int4& p, long long mp) {
    return mm_better(mq, q.z, mp, p.z) && mm_d2(q, p) < mp;
}

// Best (largest v, then smallest i) over the CTA; valid in warp 0.
__device__ __forceinline__ void mm_block_best(long long& v, int& i, int& s, long long* rv, int* ri, int* rs) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int pass = 0; pass < 2; ++pass) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const long long ov = __shfl_xor_sync(0xffffffffu, v, o);
            const int oi = __shfl_xor_sync(0xffffffffu, i, o), os = __shfl_xor_sync(0xffffffffu, s, o);
            if (mm_better(ov, oi, v, i)) {
                v = ov;
                i = oi;
                s = os;
            }
        }
        if (pass == 1) return;
        if (lane == 0) {
            rv[warp] = v;
            ri[warp] = i;
            rs[warp] = s;
        }
        __syncthreads();
        if (warp != 0) return;
        v = rv[lane];  // kMmThreads = 32 warps
        i = ri[lane];
        s = rs[lane];
    }
}

// Warp gw of GW: the sites whose keys are final go to the round's list (cnt).
__device__ __forceinline__ void mm_check(const Grid& g, const MmState& S, int D, int* cnt, int gw, int GW) {
    const int lane = threadIdx.x & 31, W = g.G + 1;
    auto take = [&](int s, long long m) {
        S.key[s] = m;
        S.list[atomicAdd(cnt, 1)] = s;
    };
    for (int base = gw * 32; base < D; base += GW * 32) {
        const int s = base + lane;
        const long long m = s < D ? __ldcg(&S.mind[s]) : -1;
        bool open = m >= 0;
        int4 p = make_int4(0, 0, 0, 0);
        if (open) {
            p = S.pts[s];
            const int w = S.wit[s];
            if (w >= 0 && mm_dominates(S.pts[w], __ldcg(&S.mind[w]), p, m)) open = false;
        }
        MmReach R{0, 0, 0, 0};
        if (open && m == 0) {  // a duplicate of a chosen site: nothing is closer
            take(s, m);
            open = false;
        }
        if (open) {  // the 3 x 3 cells around the site, its own row first
            R = mm_reach(g, p.x, p.y, m);
            const int cx = p.x >> g.shift, cy = p.y >> g.shift;
            const int xa = max(R.xl, cx - 1), xb = min(R.xh, cx + 1);
            int found = -1;
            bool cut = false;  // rows of crowded cells are left to the warp
            for (int t = 0; t < 3 && found < 0; ++t) {
                const int row = cy + (t == 0 ? 0 : t == 1 ? -1 : 1);
                if (row < R.yl || row > R.yh) continue;
                const int b = S.offsets[row * W + xa], end = S.offsets[row * W + xb + 1];
                const int e = min(end, b + 64);
                cut = cut || e < end;
                for (int x = b; x < e && found < 0; x += 4) {
                    int4 q[4];
                    long long mq[4];
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        const int y = min(x + h, e - 1);
                        q[h] = S.pts[y];
                        mq[h] = __ldcg(&S.mind[y]);
                    }
#pragma unroll
                    for (int h = 0; h < 4; ++h)
                        if (mm_dominates(q[h], mq[h], p, m)) found = min(x + h, e - 1);
                }
            }
            if (found >= 0) {
                S.wit[s] = found;
                open = false;
            } else if (!cut && R.xl >= cx - 1 && R.xh <= cx + 1 && R.yl >= cy - 1 && R.yh <= cy + 1) {
                take(s, m);
                open = false;
            }
        }
        unsigned todo = __ballot_sync(0xffffffffu, open);
        while (todo) {  // the whole reach, by the warp, rows from the site's own outwards
            const int b = __ffs(todo) - 1;
            todo &= todo - 1;
            const int4 c = make_int4(__shfl_sync(0xffffffffu, p.x, b), __shfl_sync(0xffffffffu, p.y, b),
                                     __shfl_sync(0xffffffffu, p.z, b), 0);
            const long long mc = __shfl_sync(0xffffffffu, m, b);
            const MmReach Q = mm_reach(g, c.x, c.y, mc);
            const int cy = c.y >> g.shift, far = max(cy - Q.yl, Q.yh - cy);
            int found = -1;
            for (int t0 = 0; t0 <= 2 * far && found < 0; t0 += 32) {
                // lane t holds the bounds of row t0 + t of that order
                const int t = t0 + lane, row = cy + ((t & 1) ? -((t + 1) >> 1) : (t >> 1));
                const bool in = row >= Q.yl && row <= Q.yh;
                const int rlo = in ? S.offsets[row * W + Q.xl] : 0, rhi = in ? S.offsets[row * W + Q.xh + 1] : 0;
                for (unsigned rows = __ballot_sync(0xffffffffu, rlo < rhi); rows && found < 0; rows &= rows - 1) {
                    const int h = __ffs(rows) - 1;
                    const int lo = __shfl_sync(0xffffffffu, rlo, h), hi = __shfl_sync(0xffffffffu, rhi, h);
                    for (int x0 = lo; x0 < hi && found < 0; x0 += 64) {  // two sites a lane
                        const int x = x0 + lane, y = min(x + 32, hi - 1);
                        bool d = false;
                        if (x < hi) {
                            const int4 p0 = S.pts[x], p1 = S.pts[y];
                            const long long m0 = __ldcg(&S.mind[x]), m1 = __ldcg(&S.mind[y]);
                            d = mm_dominates(p0, m0, c, mc);
                            const bool d1 = mm_dominates(p1, m1, c, mc);
                            if (d || d1) found = d ? x : y;
                            d = d || d1;
                        }
                        const unsigned hit = __ballot_sync(0xffffffffu, d);
                        if (hit) found = __shfl_sync(0xffffffffu, found, __ffs(hit) - 1);
                    }
                }
            }
            if (lane == b) {
                if (found >= 0)
                    S.wit[s] = found;
                else
                    take(s, m);
            }
        }
    }
}

// Warp gw of GW: the round's n picks leave the open sites and lower mind around them.
__device__ __forceinline__ void mm_update(const Grid& g, const MmState& S, int n, int gw, int GW) {
    const int lane = threadIdx.x & 31, W = g.G + 1;
    // warps to spare take a pick's rows side by side (the first rounds: few picks of wide reach)
    const int per = n > 0 ? max(1, min(GW / n, 64)) : 1;
    for (int64_t e = gw; e < (int64_t)n * per; e += GW) {
        const int s = __ldcg(&S.list[e / per]), r0 = (int)(e % per);
        const int4 p = S.pts[s];
        const long long K = __ldcg(&S.key[s]);
        if (r0 == 0 && lane == 0) S.mind[s] = -1;
        const MmReach R = mm_reach(g, p.x, p.y, K);
        for (int row = R.yl + r0; row <= R.yh; row += per) {
            const int lo = S.offsets[row * W + R.xl], hi = S.offsets[row * W + R.xh + 1];
            for (int x = lo + lane; x < hi; x += 32) {
                const long long m = __ldcg(&S.mind[x]);
                if (m < 0) continue;
                const int4 q = S.pts[x];
                const long long d2 = mm_d2(p, q);
                if (d2 < m && mm_better(K, p.z, m, q.z)) atomicMin(&S.mind[x], d2);
            }
        }
    }
}

__global__ void __launch_bounds__(256) maxmin_check_kernel(const Grid* __restrict__ grid, MmState S, int D, int r) {
    int done = kMmSerial;
    for (int k = 0; k < r; ++k) done += S.count[3 + k];
    if (done >= D) return;
    mm_check(*grid, S, D, S.count + 3 + r, (blockIdx.x * blockDim.x + threadIdx.x) >> 5, (gridDim.x * blockDim.x) >> 5);
}

__global__ void __launch_bounds__(256) maxmin_update_kernel(const Grid* __restrict__ grid, MmState S, int r) {
    mm_update(*grid, S, S.count[3 + r], (blockIdx.x * blockDim.x + threadIdx.x) >> 5, (gridDim.x * blockDim.x) >> 5);
}

__global__ void __launch_bounds__(kMmThreads) maxmin_kernel(const Grid* __restrict__ grid, MmState S, int D,
                                                            bool serial, bool finish, int rounds) {
    __shared__ long long red_v[32];
    __shared__ int red_i[32], red_s[32];
    __shared__ long long s_v;
    __shared__ int s_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = blockIdx.x, C = gridDim.x;  // one cluster
    const int gt = rank * kMmThreads + tid, GT = C * kMmThreads;
    const Grid g = *grid;

    if (serial) {
        // the first site: nearest the centre of the quantised bounding box
        long long qx = 0, qy = 0;
        for (int s = gt; s < D; s += GT) {
            const int4 p = S.pts[s];
            qx = max(qx, (long long)p.x);
            qy = max(qy, (long long)p.y);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            qx = max(qx, __shfl_xor_sync(0xffffffffu, qx, o));
            qy = max(qy, __shfl_xor_sync(0xffffffffu, qy, o));
        }
        if (lane == 0) {
            red_v[warp] = qx;
            red_i[warp] = (int)qy;
        }
        __syncthreads();
        if (tid == 0) {
            for (int w = 1; w < kMmThreads / 32; ++w) {
                qx = max(qx, red_v[w]);
                qy = max(qy, (long long)red_i[w]);
            }
            S.slot[rank].v = qx;
            S.slot[rank].w = qy;
        }
        cluster_sync();
        for (int c = 0; c < C; ++c) {
            qx = max(qx, __ldcg(&S.slot[c].v));
            qy = max(qy, __ldcg(&S.slot[c].w));
        }
        long long bv = LLONG_MIN;  // minus the distance: the largest is the nearest
        int bi = INT_MAX, bs = -1;
        for (int s = gt; s < D; s += GT) {
            const int4 p = S.pts[s];
            const long long dx = 2LL * p.x - qx, dy = 2LL * p.y - qy, v = -(dx * dx + dy * dy);
            if (mm_better(v, p.z, bv, bi)) {
                bv = v;
                bi = p.z;
                bs = s;
            }
        }
        // one pick at a time; the first iteration only finds the first site
        const int n_serial = min(kMmSerial, D);
        for (int k = 0; k <= n_serial; ++k) {
            mm_block_best(bv, bi, bs, red_v, red_i, red_s);
            MmSlot* sl = S.slot + kMmMaxCluster * (1 + (k & 1));
            if (tid == 0) {
                sl[rank].v = bv;
                sl[rank].w = bi;
                sl[rank].s = bs;
            }
            cluster_sync();
            if (warp == 0) {
                bv = lane < C ? __ldcg(&sl[lane].v) : LLONG_MIN;
                bi = lane < C ? (int)__ldcg(&sl[lane].w) : INT_MAX;
                bs = lane < C ? __ldcg(&sl[lane].s) : -1;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const long long ov = __shfl_xor_sync(0xffffffffu, bv, o);
                    const int oi = __shfl_xor_sync(0xffffffffu, bi, o), os = __shfl_xor_sync(0xffffffffu, bs, o);
                    if (mm_better(ov, oi, bv, bi)) {
                        bv = ov;
                        bi = oi;
                        bs = os;
                    }
                }
                if (lane == 0) {
                    s_v = bv;
                    s_s = bs;
                }
            }
            __syncthreads();
            if (k == n_serial) break;
            const int ps = s_s;  // this pick (k < D: there is one)
            const int4 p = S.pts[ps];
            if (gt == 0) S.key[ps] = k == 0 ? LLONG_MAX : s_v;
            bv = LLONG_MIN;
            bi = INT_MAX;
            bs = -1;
            for (int s = gt; s < D; s += GT) {
                const int4 q = S.pts[s];
                long long m = k == 0 ? LLONG_MAX : S.mind[s];  // this thread's own value
                if (s == ps) {
                    m = -1;
                } else if (m >= 0) {
                    m = min(m, mm_d2(p, q));
                    if (mm_better(m, q.z, bv, bi)) {
                        bv = m;
                        bi = q.z;
                        bs = s;
                    }
                }
                S.mind[s] = m;
                if (k == 0) S.wit[s] = -1;
            }
        }
        cluster_sync();
    }

    if (!finish) return;

    // rounds of locally dominant picks
    const int gw = rank * (kMmThreads / 32) + warp, GW = C * (kMmThreads / 32);
    int left = D - kMmSerial;
    for (int k = 0; k < rounds; ++k) left -= __ldcg(&S.count[3 + k]);  // what the grid-wide rounds took
    for (int r = 0; left > 0; ++r) {
        int* cnt = S.count + r % 3;
        mm_check(g, S, D, cnt, gw, GW);
        cluster_sync();
        const int n = __ldcg(cnt);
        if (n <= 0) break;  // never: the largest key of all is final
        left -= n;
        if (gt == 0) S.count[(r + 1) % 3] = 0;  // last read two rounds ago
        mm_update(g, S, n, gw, GW);
        cluster_sync();
    }
}

struct MmKeys {  // descending key, then ascending index
    const long long* key;
    const int4* pts;
    __device__ void load(int s, unsigned long long& a, unsigned long long& b, int& i) const {
        a = ~(unsigned long long)key[s];
        b = 0;
        i = pts[s].z;
    }
};

size_t maxmin_scratch_bytes(int64_t D) {
    return knn_scratch_bytes(D) + 2 * align256(sizeof(long long) * (size_t)D) + 2 * align256(sizeof(int) * (size_t)D) +
           align256(sizeof(MmSlot) * 3 * kMmMaxCluster + (3 + kMmRounds) * sizeof(int));
}

// The largest cluster that the device schedules (16 is beyond the portable 8).
int maxmin_cluster(int dev) {
    static std::mutex mu;
    static std::map<int, int> best;
    std::lock_guard<std::mutex> lk(mu);
    auto it = best.find(dev);
    if (it != best.end()) return it->second;
    int c = 8;
    if (cudaFuncSetAttribute(maxmin_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(kMmMaxCluster);
        cfg.blockDim = dim3(kMmThreads);
        cudaLaunchAttribute at;
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = kMmMaxCluster;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, maxmin_kernel, &cfg) == cudaSuccess && n > 0) c = kMmMaxCluster;
    }
    cudaGetLastError();
    return best[dev] = c;
}

cudaError_t launch_maxmin(const double* sites, int64_t D, int32_t* perm, void* scratch, cudaStream_t st) {
    if (D <= 0) return cudaSuccess;
    if (D > INT_MAX / 2) return cudaErrorInvalidValue;
    Cells c;
    cudaError_t e = build_cells(sites, D, scratch, st, c);
    if (e != cudaSuccess) return e;
    char* p = (char*)scratch + knn_scratch_bytes(D);
    MmState S;
    S.pts = c.cell_pts;
    S.offsets = c.offsets;
    S.mind = (long long*)p;
    p += align256(sizeof(long long) * (size_t)D);
    S.key = (long long*)p;
    p += align256(sizeof(long long) * (size_t)D);
    S.wit = (int*)p;
    p += align256(sizeof(int) * (size_t)D);
    S.list = (int*)p;
    p += align256(sizeof(int) * (size_t)D);
    S.slot = (MmSlot*)p;
    S.count = (int*)(p + sizeof(MmSlot) * 3 * kMmMaxCluster);
    e = cudaMemsetAsync(S.count, 0, (3 + kMmRounds) * sizeof(int), st);
    if (e != cudaSuccess) return e;
    int dev = 0;
    cudaGetDevice(&dev);
    const int most = maxmin_cluster(dev);
    int cl = 1;  // about four sites a thread: fewer CTAs make cheaper barriers
    while (cl < most && (int64_t)cl * kMmThreads * 4 < D) cl *= 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cl);
    cfg.blockDim = dim3(kMmThreads);
    cfg.stream = st;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = cl;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    const int rounds = D >= kMmGridWide ? kMmRounds : 0;
    if (rounds) {
        e = cudaLaunchKernelEx(&cfg, maxmin_kernel, (const Grid*)c.grid, S, (int)D, true, false, 0);
        if (e != cudaSuccess) return e;
        for (int r = 0; r < rounds; ++r) {
            maxmin_check_kernel<<<(unsigned)((D + 255) / 256), 256, 0, st>>>(c.grid, S, (int)D, r);
            maxmin_update_kernel<<<8 * device_sm_count(dev), 256, 0, st>>>(c.grid, S, r);
        }
    }
    e = cudaLaunchKernelEx(&cfg, maxmin_kernel, (const Grid*)c.grid, S, (int)D, rounds == 0, true, rounds);
    if (e != cudaSuccess) return e;
    // the sort's runs take the place of what the rounds leave behind (keys in place)
    const SortRun runs[2] = {{(unsigned long long*)S.key, nullptr, S.list}, {(unsigned long long*)S.mind, nullptr, S.wit}};
    return launch_sort<false>(MmKeys{S.key, S.pts}, D, perm, runs, st);
}

// ---- XY ordering on the device ------------------------------------------------
// The rank of site i in the (x, y, index) order is the number of sites whose
// key is smaller (the host's XY rule; keys are unique through the index);
// perm[rank_i] = i.  Up to kXyMax sites by counting (D^2 compares, but two
// launches: 12 us at D = 2,500), beyond by the sort above.

constexpr int kXyMax = 8192;
constexpr int kXyThreads = 256;

// Grid (site blocks x chunks of the other sites): each thread counts, for its
// site, the smaller keys of one chunk and adds the count to rank[i] (integer
// adds: the total does not depend on their order).
constexpr int kXyChunk = 128;  // 20 chunks at D = 2,500: a CTA for every SM

__global__ void __launch_bounds__(kXyThreads) order_xy_rank_kernel(const double* __restrict__ sites, int D,
                                                                   int* __restrict__ rank) {
    __shared__ unsigned long long tx[kXyChunk], ty[kXyChunk];
    const int i = blockIdx.x * kXyThreads + threadIdx.x;
    const int j0 = blockIdx.y * kXyChunk;
    const int n = min(kXyChunk, D - j0);
    for (int t = threadIdx.x; t < n; t += kXyThreads) {
        tx[t] = ord_key(sites[2 * (j0 + t)]);
        ty[t] = ord_key(sites[2 * (j0 + t) + 1]);
    }
    __syncthreads();
    if (i >= D) return;
    const unsigned long long xi = ord_key(sites[2 * i]), yi = ord_key(sites[2 * i + 1]);
    int cnt = 0;
    for (int t = 0; t < n; ++t) {
        const unsigned long long xj = tx[t], yj = ty[t];
        cnt += (xj < xi) || (xj == xi && (yj < yi || (yj == yi && j0 + t < i)));
    }
    if (cnt) atomicAdd(&rank[i], cnt);
}

__global__ void order_xy_scatter_kernel(const int* __restrict__ rank, int D, int32_t* __restrict__ perm) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < D) perm[rank[i]] = i;
}

struct XyKeys {
    const double* sites;
    __device__ void load(int s, unsigned long long& a, unsigned long long& b, int& i) const {
        a = ord_key(sites[2 * (int64_t)s]);
        b = ord_key(sites[2 * (int64_t)s + 1]);
        i = s;
    }
};

size_t order_xy_scratch_bytes(int64_t D) {
    return D > kXyMax ? 2 * (2 * align256(8 * (size_t)D) + align256(4 * (size_t)D)) : sizeof(int) * (size_t)(D > 0 ? D : 1);
}

cudaError_t launch_order_xy(const double* sites, int64_t D, int32_t* perm, void* scratch, cudaStream_t st) {
    if (D <= 0 || D > INT_MAX / 2) return cudaErrorInvalidValue;
    if (D > kXyMax) {
        SortRun r[2];
        char* p = (char*)scratch;
        for (SortRun& k : r) {
            k.a = (unsigned long long*)p;
            k.b = (unsigned long long*)(p + align256(8 * (size_t)D));
            k.idx = (int*)(p + 2 * align256(8 * (size_t)D));
            p += 2 * align256(8 * (size_t)D) + align256(4 * (size_t)D);
        }
        return launch_sort<true>(XyKeys{sites}, D, perm, r, st);
    }
    int* rank = (int*)scratch;
    cudaError_t e = cudaMemsetAsync(rank, 0, sizeof(int) * (size_t)D, st);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)((D + kXyThreads - 1) / kXyThreads), (unsigned)((D + kXyChunk - 1) / kXyChunk));
    order_xy_rank_kernel<<<grid, kXyThreads, 0, st>>>(sites, (int)D, rank);
    order_xy_scatter_kernel<<<(unsigned)((D + 255) / 256), 256, 0, st>>>(rank, (int)D, perm);
    return cudaGetLastError();
}

cudaError_t launch_group_union(const int32_t* per_site, int64_t D, int m, int p, int cmax, int32_t* cond,
                               int32_t* count, int* overflow, cudaStream_t st) {
    const int64_t G = (D + p - 1) / p;
    if (G <= 0) return cudaSuccess;
    group_union_kernel<<<(int)((G + 127) / 128), 128, 0, st>>>(per_site, D, m, p, cmax, cond, count, overflow);
    return cudaGetLastError();
}

// The largest number of leading non-negative entries over G rows of width m.
__global__ void rows_max_kernel(const int32_t* __restrict__ rows, int64_t G, int m, int* __restrict__ out) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= G) return;
    const int32_t* row = rows + k * (int64_t)m;
    int c = 0;
    while (c < m && row[c] >= 0) ++c;
    atomicMax(out, c);
}

cudaError_t launch_rows_max(const int32_t* rows, int64_t G, int m, int* out, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(int), st);
    if (e != cudaSuccess || G <= 0 || m <= 0) return e;
    rows_max_kernel<<<(int)((G + 255) / 256), 256, 0, st>>>(rows, G, m, out);
    return cudaGetLastError();
}

cudaError_t launch_group_random(int64_t D, int p, int kk, uint64_t seed, int cmax, int32_t* cond,
                                int32_t* count, cudaStream_t st) {
    const int64_t G = (D + p - 1) / p;
    if (G <= 0) return cudaSuccess;
    group_random_kernel<<<(int)((G + 127) / 128), 128, 0, st>>>(D, p, kk, seed, cmax, cond, count);
    return cudaGetLastError();
}

}  // namespace vk
