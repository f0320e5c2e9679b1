// a1: stencil selection -- the n nearest nodes of every centre (Sec. 6 uses
// n = 37, complete rings on Cartesian and hexagonal lattices, Appendix A).
//
// GPU design: nodes are binned into a uniform grid (about two nodes per cell,
// counting sort by cell).  One warp serves one centre: it takes the nodes of
// a (2R+1)^2 window of cells that lie strictly inside the radius the window
// is guaranteed to cover, ranks them by (squared distance, node index) and
// keeps the first n; with fewer than n inside, R grows.  The result equals a
// brute-force sort over all nodes.
//
// What bounds it: instruction issue and the latency of the window's loads.
// FP64 compares run at 2 per SM and clock here, so the ranking compares the
// high words of the squared distances (non-negative doubles order as their
// bits do) and settles equal high words by the full (distance, index) key.
// The candidates of a warp take 16 bytes each, so that 32 to 56 warps fit one
// SM; centres with more candidates than that space go to knn_kernel, which
// holds up to 2048.  Measured on 77,235 scattered nodes, n = 56:
// the whole window ranked in FP64 by 8 warps per SM 16.1 ms, this form about
// 0.45 ms (stencils and weights together 58.6 -> 42.9 ms).
#include <cfloat>
#include <cmath>

#include "common.cuh"

namespace rbf {

namespace {

constexpr int kMaxCand = 2048;   // candidates per window held in shared memory
constexpr int kWarpsPerBlock = 4;
constexpr int kMaxStencil = 128;   // largest n of a search

struct Grid {
    double x0, z0, cw, ch;   // origin and cell size
    int ncx, ncz;
    double period;           // > 0: periodic in x
};

__global__ void bbox_kernel(const double *x, const double *z, int64_t n, double *out, int *bad) {
    // out: [xmin, xmax, zmin, zmax] reduced with atomics on the ordered-int image
    __shared__ double s[4][256];
    double v[4] = {DBL_MAX, -DBL_MAX, DBL_MAX, -DBL_MAX};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double a = x[i], b = z[i];
        if (!isfinite(a) || !isfinite(b)) atomicExch(bad, 1);
        v[0] = fmin(v[0], a); v[1] = fmax(v[1], a);
        v[2] = fmin(v[2], b); v[3] = fmax(v[3], b);
    }
    for (int k = 0; k < 4; ++k) s[k][threadIdx.x] = v[k];
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            s[0][threadIdx.x] = fmin(s[0][threadIdx.x], s[0][threadIdx.x + w]);
            s[1][threadIdx.x] = fmax(s[1][threadIdx.x], s[1][threadIdx.x + w]);
            s[2][threadIdx.x] = fmin(s[2][threadIdx.x], s[2][threadIdx.x + w]);
            s[3][threadIdx.x] = fmax(s[3][threadIdx.x], s[3][threadIdx.x + w]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) out[blockIdx.x * 4 + 0] = s[0][0], out[blockIdx.x * 4 + 1] = s[1][0],
                          out[blockIdx.x * 4 + 2] = s[2][0], out[blockIdx.x * 4 + 3] = s[3][0];
}

__device__ __forceinline__ int cell_x(const Grid &g, double x) {
    int c = (int)floor((x - g.x0) / g.cw);
    if (g.period > 0.0) {
        c %= g.ncx;
        if (c < 0) c += g.ncx;
    } else {
        c = min(max(c, 0), g.ncx - 1);
    }
    return c;
}
__device__ __forceinline__ int cell_z(const Grid &g, double z) {
    int c = (int)floor((z - g.z0) / g.ch);
    return min(max(c, 0), g.ncz - 1);
}

__global__ void count_kernel(const double *x, const double *z, int64_t n, Grid g, int *cell, int *count) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    int c = cell_z(g, z[i]) * g.ncx + cell_x(g, x[i]);
    cell[i] = c;
    atomicAdd(&count[c], 1);
}

// Exclusive scan of count[0..m) into start[0..m] by one block of 1024 threads,
// tile by tile (coalesced; a thread's serial chunk took 37 us for 38,600 cells).
__global__ void __launch_bounds__(1024) scan_kernel(const int *count, int m, int *start) {
    __shared__ int part[33];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    int base = 0;
    for (int i0 = 0; i0 < m; i0 += 4096) {
        const int i = i0 + 4 * t;
        int v[4], sum = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k] = i + k < m ? count[i + k] : 0;
            sum += v[k];
        }
        int inc = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += u;
        }
        if (lane == 31) part[warp] = inc;
        __syncthreads();
        if (warp == 0) {
            const int w = part[lane];
            int winc = w;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, winc, o);
                if (lane >= o) winc += u;
            }
            part[lane] = winc - w;
            if (lane == 31) part[32] = winc;
        }
        __syncthreads();
        int run = base + part[warp] + inc - sum;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (i + k < m) start[i + k] = run;
            run += v[k];
        }
        base += part[32];
        __syncthreads();
    }
    if (t == 0) start[m] = base;
}

__global__ void scatter_kernel(const int *cell, int64_t n, const int *start, int *cursor, int *sorted) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    int c = cell[i];
    int pos = start[c] + atomicAdd(&cursor[c], 1);
    sorted[pos] = (int)i;
}

// Squared distance as the oracle defines it: minimum image in x, then
// dx*dx + dz*dz with each operation rounded (no contraction into FMA).
__device__ __forceinline__ double sqdist(double xc, double zc, double xj, double zj, double period) {
    double dx = __dsub_rn(xj, xc);
    if (period > 0.0) {
        double half = 0.5 * period;
        if (dx > half) dx = __dsub_rn(dx, period);
        else if (dx < -half) dx = __dadd_rn(dx, period);
    }
    double dz = __dsub_rn(zj, zc);
    return __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dz, dz));
}

// Columns [xa, xb] and rows [za, zb] of the (2R+1)^2 window around cell (cx, cz),
// whether it holds every column or row, and the radius it is guaranteed to cover.
struct Window {
    int xa, xb, za, zb;
    bool all_x, all_z;
    double guard;
};
__device__ __forceinline__ Window window_of(const Grid &g, int cx, int cz, int R) {
    Window w;
    w.all_x = (2 * R + 1 >= g.ncx);
    w.xa = w.all_x ? 0 : cx - R;
    w.xb = w.all_x ? g.ncx - 1 : cx + R;
    w.za = max(cz - R, 0);
    w.zb = min(cz + R, g.ncz - 1);
    w.all_z = (cz - R <= 0) && (cz + R >= g.ncz - 1);
    if (g.period <= 0.0) {
        w.all_x = w.all_x || ((cx - R <= 0) && (cx + R >= g.ncx - 1));
        w.xa = max(w.xa, 0);
        w.xb = min(w.xb, g.ncx - 1);
    }
    w.guard = DBL_MAX;
    if (!w.all_x) w.guard = fmin(w.guard, R * g.cw);
    if (!w.all_z) w.guard = fmin(w.guard, R * g.ch);
    w.guard *= (1.0 - 1e-9);
    return w;
}

// Positions [p0, p1) in `sorted` of the window's nodes in row rz; a periodic
// window that wraps has a second range [q0, q1), which comes first.
struct RowRange {
    int p0, p1, q0, q1;
};
__device__ __forceinline__ RowRange row_range(const Grid &g, const Window &w, const int *start, int rz) {
    RowRange r = {0, 0, 0, 0};
    int a = w.xa, b = w.xb;
    const int *s = start + rz * g.ncx;
    if (g.period > 0.0 && !w.all_x) {
        if (a < 0) { r.q0 = s[a + g.ncx]; r.q1 = s[g.ncx]; a = 0; }
        if (b >= g.ncx) { r.q0 = s[0]; r.q1 = s[b - g.ncx + 1]; b = g.ncx - 1; }
    }
    r.p0 = s[a];
    r.p1 = s[b + 1];
    return r;
}

constexpr int kFastWarps = 8;

// ranks of the NC candidates lane + 32 (k0 + c) of a warp's m: those with a
// smaller high word
template <int NC>
__device__ __forceinline__ void count_smaller(const unsigned *hi2, int m, int k0, int lane, int *rank) {
    unsigned own[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        const int i = lane + 32 * (k0 + c);
        own[c] = i < m ? hi2[2 * i + 1] : 0u;
        rank[c] = 0;
    }
    const uint4 *pair = reinterpret_cast<const uint4 *>(hi2);
#pragma unroll 4
    for (int j = 0; j < (m + 1) / 2; ++j) {   // an odd m is padded with the largest key
        const uint4 v = pair[j];
#pragma unroll
        for (int c = 0; c < NC; ++c) rank[c] += (int)(v.y < own[c]) + (int)(v.w < own[c]);
    }
}

// One warp per centre.  Centres whose window holds more than `cap` candidates
// inside the guaranteed radius are listed in slow (n_slow of them).
__global__ void __launch_bounds__(kFastWarps * 32)
knn_ranked_kernel(const double *__restrict__ x, const double *__restrict__ z, int64_t n_centers, int n, Grid g,
                  const int *__restrict__ start, const int *__restrict__ sorted, int R0, int Rmax, int cap,
                  int32_t *__restrict__ idx, int *__restrict__ status, int *__restrict__ slow,
                  int *__restrict__ n_slow) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double *cd2 = reinterpret_cast<double *>(smem) + (size_t)warp * cap;
    int *cid = reinterpret_cast<int *>(smem + (size_t)kFastWarps * cap * 8) + warp * cap;
    int *mark = reinterpret_cast<int *>(smem + (size_t)kFastWarps * cap * 12) + warp * cap;
    const int64_t c = blockIdx.x * (int64_t)kFastWarps + warp;
    if (c >= n_centers) return;
    const double xc = x[c], zc = z[c];
    const int cx = cell_x(g, xc), cz = cell_z(g, zc);
    for (int R = R0; R <= Rmax; ++R) {
        const Window w = window_of(g, cx, cz, R);
        const double r2 = w.guard * w.guard;
        int m = 0, total = 0;
        bool over = false;
        for (int rb = w.za; rb <= w.zb; rb += 32) {
            // the ranges of up to 32 rows at once, one per lane
            RowRange rr = {0, 0, 0, 0};
            if (rb + lane <= w.zb) rr = row_range(g, w, start, rb + lane);
            int rows = rr.p1 - rr.p0 + rr.q1 - rr.q0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) rows += __shfl_xor_sync(0xffffffffu, rows, o);
            total += rows;
            const int nr = min(32, w.zb - rb + 1);
            for (int r = 0; r < nr && !over; ++r)
                for (int part = 0; part < 2 && !over; ++part) {
                    const int a = __shfl_sync(0xffffffffu, part ? rr.p0 : rr.q0, r);
                    const int b = __shfl_sync(0xffffffffu, part ? rr.p1 : rr.q1, r);
                    for (int base = a; base < b; base += 32) {
                        const int p = base + lane;
                        int j = 0;
                        double d2 = DBL_MAX;
                        bool in = false;
                        if (p < b) {
                            j = sorted[p];
                            d2 = sqdist(xc, zc, x[j], z[j], g.period);
                            in = d2 < r2;
                        }
                        const unsigned mask = __ballot_sync(0xffffffffu, in);
                        if (m + __popc(mask) > cap - 1) { over = true; break; }   // one slot pads an odd count
                        if (in) {
                            const int pos = m + __popc(mask & ((1u << lane) - 1u));
                            cd2[pos] = d2;
                            cid[pos] = j;
                            mark[pos] = 0;
                        }
                        m += __popc(mask);
                    }
                }
        }
        if (total > kMaxCand) {
            if (lane == 0) atomicCAS(status, 0, 2);
            return;
        }
        if (over) {
            if (lane == 0) slow[atomicAdd(n_slow, 1)] = (int)c;
            return;
        }
        if (m < n) {
            __syncwarp();
            continue;   // fewer than n nodes strictly inside the guaranteed radius
        }
        if (lane == 0) cd2[m] = __longlong_as_double(-1LL);   // pads the last pair with the largest key
        __syncwarp();
        // mark[i] holds candidate i's rank (high half), and how many candidates
        // have rank i (low half)
        const unsigned *hi2 = reinterpret_cast<const unsigned *>(cd2);
        const int need = (m + 31) / 32;
        for (int k0 = 0; k0 < need; k0 += 6) {
            int rank[6];
            if (need - k0 > 4) count_smaller<6>(hi2, m, k0, lane, rank);
            else count_smaller<4>(hi2, m, k0, lane, rank);
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                const int i = lane + 32 * (k0 + q);
                if (i < m && q < need - k0) {
                    atomicAdd(&mark[i], rank[q] << 16);
                    atomicAdd(&mark[rank[q]], 1);
                }
            }
        }
        __syncwarp();
        for (int i = lane; i < m; i += 32) {
            int at = mark[i] >> 16;
            if (at >= n) continue;
            const int ii = cid[i];
            if ((mark[at] & 0xffff) > 1) {   // equal high words: the full key decides
                const double di = cd2[i];
                const unsigned hi = hi2[2 * i + 1];
                for (int j = 0; j < m; ++j)
                    if (hi2[2 * j + 1] == hi) {
                        const double dj = cd2[j];
                        at += (dj < di) || (dj == di && cid[j] < ii);
                    }
            }
            if (at < n) idx[c * n + at] = ii;
        }
        return;
    }
    if (lane == 0) atomicCAS(status, 0, 3);
}

// The general form: up to kMaxCand candidates per window in shared memory, the
// whole window ranked.  Takes the centres that knn_ranked_kernel listed.
__global__ void __launch_bounds__(kWarpsPerBlock * 32)
knn_kernel(const double *__restrict__ x, const double *__restrict__ z, const int *__restrict__ list, int n_list, int n,
           Grid g, const int *__restrict__ start, const int *__restrict__ sorted, int R0, int Rmax,
           int32_t *__restrict__ idx, int *__restrict__ status) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double *cd2 = reinterpret_cast<double *>(smem) + warp * kMaxCand;
    int *cid = reinterpret_cast<int *>(reinterpret_cast<double *>(smem) + kWarpsPerBlock * kMaxCand) + warp * kMaxCand;
    __shared__ double nth_d2[kWarpsPerBlock];

    const int64_t q = blockIdx.x * (int64_t)kWarpsPerBlock + warp;
    if (q >= n_list) return;
    const int64_t c = list[q];
    const double xc = x[c], zc = z[c];
    const int cx = cell_x(g, xc), cz = cell_z(g, zc);

    for (int R = R0; R <= Rmax; ++R) {
        const Window w = window_of(g, cx, cz, R);
        int m = 0;
        for (int rz = w.za; rz <= w.zb; ++rz) {
            const RowRange rr = row_range(g, w, start, rz);
            for (int part = 0; part < 2; ++part) {
                const int p0 = part ? rr.p0 : rr.q0, p1 = part ? rr.p1 : rr.q1;
                if (m + p1 - p0 > kMaxCand) {
                    if (lane == 0) atomicCAS(status, 0, 2);
                    return;
                }
                for (int p = p0 + lane; p < p1; p += 32) {
                    const int j = sorted[p];
                    cd2[m + p - p0] = sqdist(xc, zc, x[j], z[j], g.period);
                    cid[m + p - p0] = j;
                }
                m += p1 - p0;
            }
        }
        __syncwarp();
        if (m < n) continue;
        // rank every candidate by (d2, index); ranks are a permutation
        for (int i = lane; i < m; i += 32) {
            double di = cd2[i];
            int ii = cid[i];
            int rank = 0;
            for (int j = 0; j < m; ++j) {
                double dj = cd2[j];
                rank += (dj < di) || (dj == di && cid[j] < ii);
            }
            if (rank < n) idx[c * n + rank] = ii;
            if (rank == n - 1) nth_d2[warp] = di;
        }
        __syncwarp();
        if (nth_d2[warp] < w.guard * w.guard) return;   // the window provably holds the n nearest
        __syncwarp();
    }
    if (lane == 0) atomicCAS(status, 0, 3);
}

// First window of a search for n neighbours: about 2.5 n candidates at two nodes per cell.
int first_window(int n) {
    const int R0 = (int)std::ceil(std::sqrt(2.5 * n / (4.0 * 2.0)));
    return R0 < 1 ? 1 : R0;
}
// Room for the candidates inside that window's radius (2 pi R0^2 on average),
// half as many again and a margin, in whole warps.
int ranked_room(int n) {
    const int R0 = first_window(n);
    return std::min(kMaxCand, ((int)(1.5 * 6.2832 * R0 * R0) + 64 + 31) / 32 * 32);
}
size_t ranked_smem(int n) { return (size_t)kFastWarps * ranked_room(n) * (sizeof(double) + 2 * sizeof(int)); }

// Searches the stencils of every centre on a binned grid: knn_ranked_kernel,
// then knn_kernel for the centres it listed.  `slow` takes n_centers entries;
// counts[0] is the status and counts[1] the number listed (both cleared here).
// Synchronises the stream.
void search(const double *x, const double *z, int64_t n_centers, int n, const Grid &g, const int *start,
            const int *sorted, int *slow, int *counts, int32_t *idx, cudaStream_t st) {
    const int R0 = first_window(n), Rmax = std::max(g.ncx, g.ncz), cap = ranked_room(n);
    const size_t fast = ranked_smem(n);
    // the largest search's need: the limit is the kernel's, and another thread's
    // launch may lie between this call and the one below
    RBF_CUDA(cudaFuncSetAttribute(knn_ranked_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)ranked_smem(kMaxStencil)));
    RBF_CUDA(cudaMemsetAsync(counts, 0, 2 * sizeof(int), st));
    knn_ranked_kernel<<<div_up(n_centers, kFastWarps), kFastWarps * 32, fast, st>>>(
        x, z, n_centers, n, g, start, sorted, R0, Rmax, cap, idx, counts, slow, counts + 1);
    RBF_CHECK_LAUNCH();
    int h[2] = {0, 0};
    RBF_CUDA(cudaMemcpyAsync(h, counts, sizeof(h), cudaMemcpyDeviceToHost, st));
    RBF_CUDA(cudaStreamSynchronize(st));
    if (h[0] == 0 && h[1] > 0) {
        const size_t smem = (size_t)kWarpsPerBlock * kMaxCand * (sizeof(double) + sizeof(int));
        RBF_CUDA(cudaFuncSetAttribute(knn_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        knn_kernel<<<div_up(h[1], kWarpsPerBlock), kWarpsPerBlock * 32, smem, st>>>(x, z, slow, h[1], n, g, start, sorted,
                                                                                    R0, Rmax, idx, counts);
        RBF_CHECK_LAUNCH();
        RBF_CUDA(cudaMemcpyAsync(h, counts, sizeof(int), cudaMemcpyDeviceToHost, st));
        RBF_CUDA(cudaStreamSynchronize(st));
    }
    RBF_REQUIRE(h[0] == 0, "stencil search failed (%s)",
                h[0] == 2 ? "more than 2048 candidates in a search window: node density too uneven"
                          : "no window holds n nodes");
}

}  // namespace

void build_stencils(const double *x, const double *z, int64_t n_all, int64_t n_centers, int n,
                    double period_x, int32_t *idx, cudaStream_t st) {
    RBF_REQUIRE(n >= 1 && n <= kMaxStencil, "stencil size n=%d must be in [1, %d]", n, kMaxStencil);
    RBF_REQUIRE(n_all >= n, "n_all=%lld smaller than the stencil size %d", (long long)n_all, n);
    RBF_REQUIRE(n_centers >= 0 && n_centers <= n_all, "n_centers=%lld out of range", (long long)n_centers);
    RBF_REQUIRE(n_all < (int64_t)1 << 31, "n_all=%lld exceeds int32 indexing", (long long)n_all);
    RBF_REQUIRE(period_x >= 0.0 && std::isfinite(period_x), "period_x must be finite and >= 0");
    if (n_centers == 0) return;
    RBF_REQUIRE(x && z && idx, "null pointer argument");

    const int nb = 64;
    DevBuf<double> part(nb * 4);
    DevBuf<int> bad(1);
    RBF_CUDA(cudaMemsetAsync(bad.p, 0, sizeof(int), st));
    bbox_kernel<<<nb, 256, 0, st>>>(x, z, n_all, part.p, bad.p);
    RBF_CHECK_LAUNCH();
    std::vector<double> hp(nb * 4);
    int hbad = 0;
    RBF_CUDA(cudaMemcpyAsync(hp.data(), part.p, part.bytes(), cudaMemcpyDeviceToHost, st));
    RBF_CUDA(cudaMemcpyAsync(&hbad, bad.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    RBF_CUDA(cudaStreamSynchronize(st));
    RBF_REQUIRE(!hbad, "non-finite node coordinates");
    double xmin = DBL_MAX, xmax = -DBL_MAX, zmin = DBL_MAX, zmax = -DBL_MAX;
    for (int b = 0; b < nb; ++b) {
        xmin = std::fmin(xmin, hp[b * 4 + 0]); xmax = std::fmax(xmax, hp[b * 4 + 1]);
        zmin = std::fmin(zmin, hp[b * 4 + 2]); zmax = std::fmax(zmax, hp[b * 4 + 3]);
    }
    Grid g;
    g.period = period_x;
    double W = period_x > 0.0 ? period_x : (xmax - xmin);
    double H = zmax - zmin;
    double area = std::fmax(W, 1e-300) * std::fmax(H, 1e-300);
    if (W <= 0.0 || H <= 0.0) area = std::fmax(W, H) * std::fmax(W, H) / (double)n_all;
    double cell = std::sqrt(2.0 * area / (double)n_all);
    if (!(cell > 0.0)) cell = 1.0;
    g.x0 = xmin;
    g.z0 = zmin;
    g.ncx = (int)std::fmax(1.0, std::fmin(std::floor(W / cell), 1e6));
    g.ncz = (int)std::fmax(1.0, std::fmin(std::ceil(H / cell), 1e6));
    if (period_x <= 0.0 && W / g.ncx > 0) g.ncx = (int)std::fmax(1.0, std::ceil(W / cell));
    g.cw = W > 0.0 ? W / g.ncx : cell;
    g.ch = H > 0.0 ? H / g.ncz : cell;
    int64_t ncell = (int64_t)g.ncx * g.ncz;
    RBF_REQUIRE(ncell < ((int64_t)1 << 30), "binning grid too large");

    DevBuf<int> cellof(n_all), count(ncell), start(ncell + 1), cursor(ncell), sorted(n_all);
    DevBuf<int> counts(2);
    RBF_CUDA(cudaMemsetAsync(count.p, 0, count.bytes(), st));
    RBF_CUDA(cudaMemsetAsync(cursor.p, 0, cursor.bytes(), st));
    count_kernel<<<div_up(n_all, 256), 256, 0, st>>>(x, z, n_all, g, cellof.p, count.p);
    RBF_CHECK_LAUNCH();
    scan_kernel<<<1, 1024, 0, st>>>(count.p, (int)ncell, start.p);
    RBF_CHECK_LAUNCH();
    scatter_kernel<<<div_up(n_all, 256), 256, 0, st>>>(cellof.p, n_all, start.p, cursor.p, sorted.p);
    RBF_CHECK_LAUNCH();

    search(x, z, n_centers, n, g, start.p, sorted.p, cellof.p, counts.p, idx, st);   // cellof is free by now
}

// ---- allocation-free variant (rbf_build_stencils_static) --------------------
// The same kernels as rbf_build_stencils, with every scratch buffer carved out
// of one file-scope device array instead of cudaMalloc.  The array lives on
// every GPU that loads this library until the process exits.
namespace {

constexpr int64_t kStaticMaxNodes = 262144;   // n_all limit of the static variant
constexpr int64_t kStaticMaxCells = 262144;   // binning cells limit
constexpr int kBboxBlocks = 64;

constexpr size_t align256(size_t b) { return (b + 255) & ~size_t(255); }
constexpr size_t kOffPart = 0;
constexpr size_t kOffBad = kOffPart + align256(kBboxBlocks * 4 * sizeof(double));
constexpr size_t kOffStatus = kOffBad + 256;
constexpr size_t kOffCellOf = kOffStatus + 256;
constexpr size_t kOffSorted = kOffCellOf + align256(kStaticMaxNodes * sizeof(int));
constexpr size_t kOffCount = kOffSorted + align256(kStaticMaxNodes * sizeof(int));
constexpr size_t kOffCursor = kOffCount + align256(kStaticMaxCells * sizeof(int));
constexpr size_t kOffStart = kOffCursor + align256(kStaticMaxCells * sizeof(int));
constexpr size_t kStaticScratchBytes = kOffStart + align256((kStaticMaxCells + 1) * sizeof(int));  // ~5 MB

static __device__ __align__(256) unsigned char g_stencil_scratch[kStaticScratchBytes];

// Device address of the scratch array on the current device.  In host code
// the symbol is only a stand-in, so the address is looked up with the device
// current -- on every call, not cached: after a device reset or in a new
// context the module is loaded again and the array moves.  The lookup is
// cheap next to the call's own two stream synchronisations.
unsigned char *static_scratch() {
    void *ptr = nullptr;
    RBF_CUDA(cudaGetSymbolAddress(&ptr, g_stencil_scratch));
    return static_cast<unsigned char *>(ptr);
}

}  // namespace

void build_stencils_static(const double *x, const double *z, int64_t n_all, int64_t n_centers, int n,
                           double period_x, int32_t *idx, cudaStream_t st) {
    RBF_REQUIRE(n >= 1 && n <= kMaxStencil, "stencil size n=%d must be in [1, %d]", n, kMaxStencil);
    RBF_REQUIRE(n_all >= n, "n_all=%lld smaller than the stencil size %d", (long long)n_all, n);
    RBF_REQUIRE(n_all <= kStaticMaxNodes, "n_all=%lld exceeds the static scratch limit of %lld nodes",
                (long long)n_all, (long long)kStaticMaxNodes);
    RBF_REQUIRE(n_centers >= 0 && n_centers <= n_all, "n_centers=%lld out of range", (long long)n_centers);
    RBF_REQUIRE(period_x >= 0.0 && std::isfinite(period_x), "period_x must be finite and >= 0");
    if (n_centers == 0) return;
    RBF_REQUIRE(x && z && idx, "null pointer argument");
    unsigned char *base = static_scratch();
    double *part = reinterpret_cast<double *>(base + kOffPart);
    int *bad = reinterpret_cast<int *>(base + kOffBad);
    int *status = reinterpret_cast<int *>(base + kOffStatus);
    int *cellof = reinterpret_cast<int *>(base + kOffCellOf);
    int *sorted = reinterpret_cast<int *>(base + kOffSorted);
    int *count = reinterpret_cast<int *>(base + kOffCount);
    int *cursor = reinterpret_cast<int *>(base + kOffCursor);
    int *start = reinterpret_cast<int *>(base + kOffStart);

    // bounding box (the array keeps the previous call's contents: clear flags)
    RBF_CUDA(cudaMemsetAsync(bad, 0, sizeof(int), st));
    bbox_kernel<<<kBboxBlocks, 256, 0, st>>>(x, z, n_all, part, bad);
    RBF_CHECK_LAUNCH();
    double hp[kBboxBlocks * 4];
    int hbad = 0;
    RBF_CUDA(cudaMemcpyAsync(hp, part, sizeof(hp), cudaMemcpyDeviceToHost, st));
    RBF_CUDA(cudaMemcpyAsync(&hbad, bad, sizeof(int), cudaMemcpyDeviceToHost, st));
    RBF_CUDA(cudaStreamSynchronize(st));
    RBF_REQUIRE(!hbad, "non-finite node coordinates");
    double xmin = DBL_MAX, xmax = -DBL_MAX, zmin = DBL_MAX, zmax = -DBL_MAX;
    for (int b = 0; b < kBboxBlocks; ++b) {
        xmin = std::fmin(xmin, hp[b * 4 + 0]); xmax = std::fmax(xmax, hp[b * 4 + 1]);
        zmin = std::fmin(zmin, hp[b * 4 + 2]); zmax = std::fmax(zmax, hp[b * 4 + 3]);
    }
    // binning grid: the same rule as the allocating entry point
    Grid g;
    g.period = period_x;
    double W = period_x > 0.0 ? period_x : (xmax - xmin);
    double H = zmax - zmin;
    double area = std::fmax(W, 1e-300) * std::fmax(H, 1e-300);
    if (W <= 0.0 || H <= 0.0) area = std::fmax(W, H) * std::fmax(W, H) / (double)n_all;
    double cell = std::sqrt(2.0 * area / (double)n_all);
    if (!(cell > 0.0)) cell = 1.0;
    g.x0 = xmin;
    g.z0 = zmin;
    g.ncx = (int)std::fmax(1.0, std::fmin(std::floor(W / cell), 1e6));
    g.ncz = (int)std::fmax(1.0, std::fmin(std::ceil(H / cell), 1e6));
    if (period_x <= 0.0 && W / g.ncx > 0) g.ncx = (int)std::fmax(1.0, std::ceil(W / cell));
    g.cw = W > 0.0 ? W / g.ncx : cell;
    g.ch = H > 0.0 ? H / g.ncz : cell;
    const int64_t ncell = (int64_t)g.ncx * g.ncz;
    RBF_REQUIRE(ncell <= kStaticMaxCells, "binning grid of %lld cells exceeds the static scratch limit of %lld",
                (long long)ncell, (long long)kStaticMaxCells);

    RBF_CUDA(cudaMemsetAsync(count, 0, ncell * sizeof(int), st));
    RBF_CUDA(cudaMemsetAsync(cursor, 0, ncell * sizeof(int), st));
    count_kernel<<<div_up(n_all, 256), 256, 0, st>>>(x, z, n_all, g, cellof, count);
    RBF_CHECK_LAUNCH();
    scan_kernel<<<1, 1024, 0, st>>>(count, (int)ncell, start);
    RBF_CHECK_LAUNCH();
    scatter_kernel<<<div_up(n_all, 256), 256, 0, st>>>(cellof, n_all, start, cursor, sorted);
    RBF_CHECK_LAUNCH();
    search(x, z, n_centers, n, g, start, sorted, cellof, status, idx, st);   // cellof is free by now
}

}  // namespace rbf

extern "C" int rbf_build_stencils(const double *x, const double *z, int64_t n_all, int64_t n_centers,
                                  int32_t n, double period_x, int32_t *idx, void *stream) {
    return rbf::guarded([&] {
        rbf::build_stencils(x, z, n_all, n_centers, n, period_x, idx, rbf::as_stream(stream));
    });
}

extern "C" int rbf_build_stencils_static(const double *x, const double *z, int64_t n_all, int64_t n_centers,
                                         int32_t n, double period_x, int32_t *idx, void *stream) {
    return rbf::guarded([&] {
        rbf::build_stencils_static(x, z, n_all, n_centers, n, period_x, idx, rbf::as_stream(stream));
    });
}
