// a9: learned tendency correction for coarse runs (no counterpart in the
// paper; the paper's method is the solver it corrects).
//
// Per coarse node: features = the stencil differences of the four fields,
// scaled per field (4 (n-1) values, the node's own RBF-FD stencil); a 3-layer
// MLP f (width 64, tanh, BF16 weights, FP32 accumulation) gives the tendency
// correction delta = (f(x) - f(0)) s_out, added as dt * delta after each
// coarse RK4 step.  Subtracting f(0) makes a locally uniform state (all
// differences zero), where fine and coarse steps agree, uncorrected.
//
// Kernels (CUDA cores: the per-node contraction is ~14k MACs on a few
// thousand nodes, latency-bound, not a tensor-core sized GEMM):
//   mlp_infer_kernel  fused gather + forward, one thread per node, weights in
//                     shared memory as BF16
//   mlp_train_kernel  fused gather + forward + backward for 31 samples per
//                     block; the block's weight gradients (H^T dH products
//                     over its samples) go to its own FP32 partials
//   mlp_reduce_kernel sums the partials in block order, then Adam on the FP32
//                     master weights and the refresh of the BF16 copy
#include <cuda_bf16.h>

#include <cmath>
#include <vector>
#include <cstring>

#include "problem.cuh"
#include "records.cuh"

namespace rbf {

constexpr int kWidth = 64;
constexpr int kTrainRows = 32;               // rows of a training block: 31 samples and the all-zero row
constexpr int kTrainSamples = kTrainRows - 1;
constexpr int kTrainSets = 608;               // most blocks of a training launch (their partials: 34 MB for n = 37)
constexpr int kTrainThreads = 320;           // 10 warps: two passes over the 592 tiles of dW1 (n = 37)
constexpr int kScaleWarps = 2048;   // warps of the scale-sum launch (256 blocks of 256 threads)
constexpr float kClip = 4.f;   // |y| <= 4 (in output-scale units) when the correction is applied

struct Mlp {
    int n = 0, slots = 0, n_in = 0;
    int64_t n_params = 0;
    int64_t oW1 = 0, ob1 = 0, oW2 = 0, ob2 = 0, oW3 = 0, ob3 = 0;
    cudaStream_t st = nullptr;
    DevBuf<float> P, Gr, M, V, scales, loss;
    DevBuf<float> Gp, Lp;     // per-block gradient and loss partials of a training launch
    DevBuf<__nv_bfloat16> Pb;
    DevBuf<double> acc;       // scale sums
    DevBuf<unsigned long long> bad;
    int64_t t = 0;
};

namespace {

struct Offs {   // parameter offsets: W1 [n_in][64], b1, W2 [64][64], b2, W3 [64][4], b3
    int64_t oW1, ob1, oW2, ob2, oW3, ob3;
};

Offs offs_of(const Mlp &m) { return {m.oW1, m.ob1, m.oW2, m.ob2, m.oW3, m.ob3}; }

// state of target sample k: runs hold n_snap states and n_snap - 1 targets
__device__ __forceinline__ int64_t state_of(int64_t k, int64_t n_snap) {
    return (k / (n_snap - 1)) * n_snap + k % (n_snap - 1);
}

struct Net {
    const __nv_bfloat16 *W1, *W2, *W3;
    const float *b1, *b2, *b3;
};

__device__ __forceinline__ float bf(const __nv_bfloat16 v) { return __bfloat162float(v); }

// shared-memory image of the network: BF16 weights, FP32 biases
__device__ Net load_net(unsigned char *sm, const __nv_bfloat16 *Pb, const float *P, int n_in, const Offs o) {
    const int64_t oW1 = o.oW1, ob1 = o.ob1, oW2 = o.oW2, ob2 = o.ob2, oW3 = o.oW3, ob3 = o.ob3;
    __nv_bfloat16 *w1 = reinterpret_cast<__nv_bfloat16 *>(sm);
    __nv_bfloat16 *w2 = w1 + n_in * kWidth;
    __nv_bfloat16 *w3 = w2 + kWidth * kWidth;
    float *b = reinterpret_cast<float *>(w3 + kWidth * 4);
    for (int e = threadIdx.x; e < n_in * kWidth; e += blockDim.x) w1[e] = Pb[oW1 + e];
    for (int e = threadIdx.x; e < kWidth * kWidth; e += blockDim.x) w2[e] = Pb[oW2 + e];
    for (int e = threadIdx.x; e < kWidth * 4; e += blockDim.x) w3[e] = Pb[oW3 + e];
    for (int e = threadIdx.x; e < kWidth; e += blockDim.x) {
        b[e] = P[ob1 + e];
        b[kWidth + e] = P[ob2 + e];
    }
    if (threadIdx.x < 4) b[2 * kWidth + threadIdx.x] = P[ob3 + threadIdx.x];
    __syncthreads();
    return {w1, w2, w3, b, b + kWidth, b + 2 * kWidth};
}

// f(0) of the network (the output for all-zero features), and its hidden
// activations, computed by the first 64 threads of the block into z1, z2, y0.
__device__ void zero_branch(const Net &net, float *z1, float *z2, float *y0) {
    const int t = threadIdx.x;
    if (t < kWidth) z1[t] = tanhf(net.b1[t]);
    __syncthreads();
    if (t < kWidth) {
        float a = net.b2[t];
        for (int m = 0; m < kWidth; ++m) a += z1[m] * bf(net.W2[m * kWidth + t]);
        z2[t] = tanhf(a);
    }
    __syncthreads();
    if (t < 4) {
        float a = net.b3[t];
        for (int m = 0; m < kWidth; ++m) a += z2[m] * bf(net.W3[m * 4 + t]);
        y0[t] = a;
    }
    __syncthreads();
}

__host__ __device__ __forceinline__ size_t net_bytes(int n_in) {
    return (size_t)(n_in * kWidth + kWidth * kWidth + kWidth * 4) * 2 + (2 * kWidth + 4) * 4;
}

// h1 += x (row r of W1) for the features of one neighbour (4 fields)
__device__ __forceinline__ void layer1_row(float *h, const __nv_bfloat16 *w1, int row, float x) {
    const __nv_bfloat162 *w = reinterpret_cast<const __nv_bfloat162 *>(w1 + row * kWidth);
#pragma unroll
    for (int j = 0; j < kWidth / 2; ++j) {
        const float2 v = __bfloat1622float2(w[j]);
        h[2 * j] += x * v.x;
        h[2 * j + 1] += x * v.y;
    }
}

// out = tanh(in W + b), 64 x 64
__device__ __forceinline__ void layer2(const float *in, const __nv_bfloat16 *w2, const float *b, float *out) {
#pragma unroll
    for (int j = 0; j < kWidth; ++j) out[j] = b[j];
    for (int m = 0; m < kWidth; ++m) {
        const float x = in[m];
        const __nv_bfloat162 *w = reinterpret_cast<const __nv_bfloat162 *>(w2 + m * kWidth);
#pragma unroll
        for (int j = 0; j < kWidth / 2; ++j) {
            const float2 v = __bfloat1622float2(w[j]);
            out[2 * j] += x * v.x;
            out[2 * j + 1] += x * v.y;
        }
    }
#pragma unroll
    for (int j = 0; j < kWidth; ++j) out[j] = tanhf(out[j]);
}

// Fused gather + forward pass: delta[i] = MLP(features of node i) * s_out.
template <class T>
__global__ void __launch_bounds__(128) mlp_infer_kernel(const T *__restrict__ U, const int32_t *__restrict__ idx, int n,
                                                        int64_t n_prog, const __nv_bfloat16 *__restrict__ Pb,
                                                        const float *__restrict__ P, Offs m_off, const float *scales,
                                                        const unsigned char *__restrict__ flags, T *__restrict__ delta) {
    extern __shared__ unsigned char sm[];
    const int n_in = 4 * (n - 1) + 4;
    const Net net = load_net(sm, Pb, P, n_in, m_off);
    __shared__ float z1[kWidth], z2[kWidth], y0[4];
    zero_branch(net, z1, z2, y0);
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n_prog) return;
    const float is0 = 1.f / scales[0], is1 = 1.f / scales[1], is2 = 1.f / scales[2], is3 = 1.f / scales[3];
    const Rec<T> own = load_rec(U, i);
    float h[kWidth];
#pragma unroll
    for (int j = 0; j < kWidth; ++j) h[j] = net.b1[j];
    const int slots = n - 1;
    for (int k = 1; k < n; ++k) {
        const Rec<T> r = load_rec(U, idx[i * n + k]);
        layer1_row(h, net.W1, 0 * slots + k - 1, (float)(r.u - own.u) * is0);
        layer1_row(h, net.W1, 1 * slots + k - 1, (float)(r.w - own.w) * is1);
        layer1_row(h, net.W1, 2 * slots + k - 1, (float)(r.t - own.t) * is2);
        layer1_row(h, net.W1, 3 * slots + k - 1, (float)(r.p - own.p) * is3);
    }
    // the node's own values
    layer1_row(h, net.W1, 4 * slots + 0, (float)own.u / scales[8]);
    layer1_row(h, net.W1, 4 * slots + 1, (float)own.w / scales[9]);
    layer1_row(h, net.W1, 4 * slots + 2, (float)own.t / scales[10]);
    layer1_row(h, net.W1, 4 * slots + 3, (float)own.p / scales[11]);
#pragma unroll
    for (int j = 0; j < kWidth; ++j) h[j] = tanhf(h[j]);
    float h2[kWidth];
    layer2(h, net.W2, net.b2, h2);
    float y[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) y[c] = net.b3[c];
#pragma unroll
    for (int m = 0; m < kWidth; ++m)
#pragma unroll
        for (int c = 0; c < 4; ++c) y[c] += h2[m] * bf(net.W3[m * 4 + c]);
    const unsigned char fl = flags[i];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        // y = f(x) - f(0); a safeguard clips the correction at 4 output scales
        float d = fminf(fmaxf(y[c] - y0[c], -kClip), kClip) * scales[4 + c];
        if ((c == 1 && (fl & 1)) || (c == 0 && (fl & 2))) d = 0.f;   // Dirichlet components stay fixed
        delta[i * 4 + c] = (T)d;
    }
}

// U += dt * delta on prognostic records; a non-finite delta is skipped
// (the node falls back to the uncorrected step) and counted.
template <class T>
__global__ void mlp_apply_kernel(T *U, const T *delta, int64_t n_prog, T dt, float4 alpha, unsigned long long *bad) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= n_prog * 4) return;
    const int f = (int)(e & 3);
    const T a = (T)(f == 0 ? alpha.x : f == 1 ? alpha.y : f == 2 ? alpha.z : alpha.w);
    const T d = delta[e];
    if (isfinite((double)d)) U[e] += a * dt * d;
    else atomicAdd(bad, 1ull);
}

__device__ __forceinline__ unsigned long long splitmix64(unsigned long long x) {
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}

struct TrainArgs {
    const float *S;       // states [n_runs][n_snap][n_all][4] (ghosts filled)
    const float *Tg;      // targets [n_runs][n_snap - 1][n_prog][4] (raw tendencies)
    int64_t n_states;     // targets: n_runs (n_snap - 1)
    int64_t n_snap;
    int64_t n_all, n_prog;
    const int32_t *idx;
    int n;
    const int64_t *samples;   // optional [B][2] (state, node); else drawn from seed
    unsigned long long seed;
    long long iter;
    int B;
    const __nv_bfloat16 *Pb;
    const float *P;
    const float *scales;
    float *Gp;            // [blocks][n_params]: this block's weight gradients
    int64_t n_params;
    float *Lp;            // [blocks]: this block's loss
};

// Shared memory of the training kernel, in floats: features, activations and
// their gradients are stored [unit][row] with kRS floats per unit, weights as
// FP32 values of their BF16 copies.
constexpr int kRS = kTrainRows + 4;   // row stride: 16-byte vectors of eight units hit distinct banks
struct TrainSmem {
    int X, W1, W2, W2t, W3, b, H1, H2, P, dH2, dH1, Y, end;
};
__host__ __device__ inline TrainSmem train_layout(int n_in) {
    TrainSmem L;
    L.X = 0;
    L.W1 = L.X + n_in * kRS;
    L.W2 = L.W1 + n_in * kWidth;
    L.W2t = L.W2 + kWidth * kWidth;       // [j][m], stride kWidth + 4
    L.W3 = L.W2t + kWidth * (kWidth + 4);
    L.b = L.W3 + kWidth * 4;              // b1, b2, b3
    L.H1 = L.b + 2 * kWidth + 4;
    L.H2 = L.H1 + kWidth * kRS;
    L.P = L.H2 + kWidth * kRS;            // two partial products
    L.dH2 = L.P + 2 * kWidth * kRS;
    L.dH1 = L.dH2 + kWidth * kRS;
    L.Y = L.dH1 + kWidth * kRS;           // [row][4]: outputs, then their gradients
    L.end = L.Y + kTrainRows * 4;
    return L;
}

__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }

// eight BF16 values as FP32
__device__ __forceinline__ void put8(float *dst, const uint4 &v) {
    const unsigned u[4] = {v.x, v.y, v.z, v.w};
    float f[8];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        f[2 * q] = __uint_as_float(u[q] << 16);
        f[2 * q + 1] = __uint_as_float(u[q] & 0xffff0000u);
    }
    *reinterpret_cast<float4 *>(dst) = make_float4(f[0], f[1], f[2], f[3]);
    *reinterpret_cast<float4 *>(dst + 4) = make_float4(f[4], f[5], f[6], f[7]);
}

// P[half][c][row] = sum over half of k of A[k][row] B[k][c] for 32 rows and 64
// columns: 128 threads per half of k, 4 rows x 4 columns each.
__device__ __forceinline__ void rows_times(const float *A, const float *B, int bs, int K, float *P) {
    if (threadIdx.x >= 256) return;
    const int half = threadIdx.x >> 7, t = threadIdx.x & 127, lane = t & 31, w = t >> 5;
    const int r0 = 4 * ((lane >> 3) + 4 * (w & 1)), c0 = 4 * ((lane & 7) + 8 * (w >> 1));
    const int k0 = half ? K / 2 : 0, k1 = half ? K : K / 2;
    float acc[4][4];   // [column][row]
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[c][r] = 0.f;
#pragma unroll 4
    for (int k = k0; k < k1; ++k) {
        const float4 x = ld4(A + k * kRS + r0), v = ld4(B + k * bs + c0);
        const float xr[4] = {x.x, x.y, x.z, x.w}, vc[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[c][r] += xr[r] * vc[c];
    }
    float *out = P + half * kWidth * kRS;
#pragma unroll
    for (int c = 0; c < 4; ++c)
        *reinterpret_cast<float4 *>(out + (c0 + c) * kRS + r0) = make_float4(acc[c][0], acc[c][1], acc[c][2], acc[c][3]);
}

// a block's partial: v of its first tile, then what the others add
__device__ __forceinline__ void put(float *p, float v, bool add) { *p = add ? *p + v : v; }

// G[a][b] = sum over the 32 rows of A[a][row] B[b][row] for a < na and 64
// columns b (a weight gradient), on top of what G holds with `add`: 4 x 4 outputs
// per thread, interleaved so that the vectors a warp reads lie in distinct banks.
__device__ __forceinline__ void outer_sum(const float *A, int na, const float *B, float *G, bool add) {
    const int ga = (na + 3) / 4;
    for (int e = threadIdx.x; e < ga * 16; e += blockDim.x) {
        const int tb = e & 15, ta = e >> 4;
        float acc[4][4];
        int ai[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            ai[i] = min(ta + i * ga, na - 1);
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
        }
#pragma unroll 2
        for (int r = 0; r < kTrainRows; r += 4) {
            float4 bv[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) bv[j] = ld4(B + (tb + 16 * j) * kRS + r);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 av = ld4(A + ai[i] * kRS + r);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    acc[i][j] += av.x * bv[j].x;
                    acc[i][j] += av.y * bv[j].y;
                    acc[i][j] += av.z * bv[j].z;
                    acc[i][j] += av.w * bv[j].w;
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (ta + i * ga < na)
#pragma unroll
                for (int j = 0; j < 4; ++j) put(G + (int64_t)(ta + i * ga) * kWidth + tb + 16 * j, acc[i][j], add);
    }
}

__device__ __forceinline__ float row_sum(const float *v) {
    float s = 0.f;
#pragma unroll
    for (int r = 0; r < kTrainRows; r += 4) {
        const float4 x = ld4(v + r);
        s += (x.x + x.y) + (x.z + x.w);
    }
    return s;
}

// Fused gather + forward + backward for tiles of 31 samples, one per block; from
// kTrainSets blocks on a block takes every gridDim-th tile, which bounds the
// partials (a set per tile would be 1.8 GB at a million samples).  The block's
// weight gradients (X^T dH1, H1^T dH2, H2^T dY and bias sums) and loss go to its
// own partials, which mlp_reduce_kernel sums over the blocks in block
// order (so training is deterministic).  Row 31 is the all-zero feature row:
// its output is f(0), which enters every y with the opposite sign, so its
// output gradient is minus the sum of the others'.
//
// What bounds it: FP32 FMA issue (1.0 M products per block, 8 k cycles at the
// full rate) behind the latency of the gather.  31 samples per block give one
// block per SM at the default batch of 4096 (133 blocks); every product runs
// from shared memory with 16 FMAs per two 16-byte loads.  One thread per
// sample with the activations in registers (32 blocks of 128 threads) took
// 207 us per launch and 217 us of device time per iteration with its two
// follow-up kernels at 4096 samples, n = 37; this form 21 us, reduction and Adam
// included.
__global__ void __launch_bounds__(kTrainThreads) mlp_train_kernel(TrainArgs a, Offs m_off) {
    extern __shared__ __align__(16) float sf[];
    __shared__ int64_t s_state[kTrainRows];   // first record of each row's state
    __shared__ int64_t s_target[kTrainRows];  // its target record
    __shared__ int s_node[kTrainRows];
    float *const gp = a.Gp + blockIdx.x * a.n_params;
    const int n_in = 4 * (a.n - 1) + 4, slots = a.n - 1;
    const TrainSmem L = train_layout(n_in);
    float *X = sf + L.X, *H1 = sf + L.H1, *H2 = sf + L.H2, *P = sf + L.P, *dH2 = sf + L.dH2, *dH1 = sf + L.dH1,
          *Y = sf + L.Y;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int64_t tiles = (a.B + (int64_t)kTrainSamples - 1) / kTrainSamples;
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const bool add = tile != blockIdx.x;
        if (add) __syncthreads();   // the rows of the tile before have been read
        // samples and features do not depend on the preceding kernel
        if (t < kTrainRows) {
            const int64_t s = tile * (int64_t)kTrainSamples + t;
            int64_t k = 0, i = -1;
            if (t < kTrainSamples && s < a.B) {
                if (a.samples) {
                    k = a.samples[2 * s];
                    i = a.samples[2 * s + 1];
                } else {
                    const unsigned long long h = splitmix64(a.seed ^ splitmix64((unsigned long long)a.iter * 0x100000001ull + s));
                    k = (int64_t)(h % (unsigned long long)a.n_states);
                    i = (int64_t)((h >> 32) % (unsigned long long)a.n_prog);
                }
            }
            s_state[t] = state_of(k, a.n_snap) * a.n_all;
            s_target[t] = k * a.n_prog + i;
            s_node[t] = (int)i;
        }
        __syncthreads();
        {
            // a warp takes one slot of the 32 rows at a time (the last one: the node's own values)
            const int i = s_node[lane];
            const float *Uk = a.S + s_state[lane] * 4;
            Rec<float> own = {0.f, 0.f, 0.f, 0.f};
            if (i >= 0) own = load_rec(Uk, i);
            const float is0 = 1.f / a.scales[0], is1 = 1.f / a.scales[1], is2 = 1.f / a.scales[2], is3 = 1.f / a.scales[3];
#pragma unroll 4
            for (int q = warp; q <= slots; q += kTrainThreads / 32) {
                float f0 = 0.f, f1 = 0.f, f2 = 0.f, f3 = 0.f;
                if (i >= 0) {
                    if (q < slots) {
                        const Rec<float> r = load_rec(Uk, __ldg(a.idx + (int64_t)i * a.n + q + 1));
                        f0 = (r.u - own.u) * is0;
                        f1 = (r.w - own.w) * is1;
                        f2 = (r.t - own.t) * is2;
                        f3 = (r.p - own.p) * is3;
                    } else {
                        f0 = own.u / a.scales[8];
                        f1 = own.w / a.scales[9];
                        f2 = own.t / a.scales[10];
                        f3 = own.p / a.scales[11];
                    }
                }
                const int c = q < slots ? q : 4 * slots, step = q < slots ? slots : 1;
                X[c * kRS + lane] = f0;
                X[(c + step) * kRS + lane] = f1;
                X[(c + 2 * step) * kRS + lane] = f2;
                X[(c + 3 * step) * kRS + lane] = f3;
            }
        }
        if (!add) {
            grid_dep_wait();     // the weights come from the preceding iteration's kernel
            grid_dep_launch();
            // BF16 weights, eight per load (every block of Pb starts at a multiple of 64 values)
            const uint4 *w1 = reinterpret_cast<const uint4 *>(a.Pb + m_off.oW1), *w2 = reinterpret_cast<const uint4 *>(a.Pb + m_off.oW2);
#pragma unroll 4
            for (int e = t; e < n_in * kWidth / 8; e += kTrainThreads) put8(sf + L.W1 + 8 * e, __ldcg(w1 + e));
#pragma unroll 2
            for (int e = t; e < kWidth * kWidth / 8; e += kTrainThreads) {
                float *v = sf + L.W2 + 8 * e;
                put8(v, __ldcg(w2 + e));
                const int m = e / (kWidth / 8), j = e % (kWidth / 8) * 8;
#pragma unroll
                for (int q = 0; q < 8; ++q) sf[L.W2t + (j + q) * (kWidth + 4) + m] = v[q];
            }
            for (int e = t; e < kWidth * 4; e += kTrainThreads) sf[L.W3 + e] = bf(a.Pb[m_off.oW3 + e]);
            if (t < kWidth) {
                sf[L.b + t] = a.P[m_off.ob1 + t];
                sf[L.b + kWidth + t] = a.P[m_off.ob2 + t];
            }
            if (t < 4) sf[L.b + 2 * kWidth + t] = a.P[m_off.ob3 + t];
        }
        __syncthreads();
        // forward
        rows_times(X, sf + L.W1, kWidth, n_in, P);
        __syncthreads();
        for (int e = t; e < kWidth * kTrainRows; e += kTrainThreads) {
            const int j = e / kTrainRows, at = j * kRS + e % kTrainRows;
            H1[at] = tanhf(sf[L.b + j] + (P[at] + P[kWidth * kRS + at]));
        }
        __syncthreads();
        rows_times(H1, sf + L.W2, kWidth, kWidth, P);
        __syncthreads();
        for (int e = t; e < kWidth * kTrainRows; e += kTrainThreads) {
            const int j = e / kTrainRows, at = j * kRS + e % kTrainRows;
            H2[at] = tanhf(sf[L.b + kWidth + j] + (P[at] + P[kWidth * kRS + at]));
        }
        __syncthreads();
        if (t < 4 * kTrainRows) {
            const int r = t % kTrainRows, c = t / kTrainRows;
            float y0 = 0.f, y1 = 0.f, y2 = 0.f, y3 = 0.f;
#pragma unroll 4
            for (int m = 0; m < kWidth; m += 4) {
                y0 += H2[m * kRS + r] * sf[L.W3 + m * 4 + c];
                y1 += H2[(m + 1) * kRS + r] * sf[L.W3 + m * 4 + 4 + c];
                y2 += H2[(m + 2) * kRS + r] * sf[L.W3 + m * 4 + 8 + c];
                y3 += H2[(m + 3) * kRS + r] * sf[L.W3 + m * 4 + 12 + c];
            }
            Y[r * 4 + c] = sf[L.b + 2 * kWidth + c] + ((y0 + y1) + (y2 + y3));
        }
        __syncthreads();
        if (warp == 0) {
            // loss and output gradients, one row per lane; row 31 holds f(0)
            const bool live = s_node[lane] >= 0;
            const float inv = 1.f / (4.f * (float)a.B);
            const float4 y = ld4(Y + lane * 4);
            const float yr[4] = {y.x, y.y, y.z, y.w};
            float loss = 0.f, d[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float f0 = __shfl_sync(0xffffffffu, yr[c], kTrainRows - 1);
                d[c] = 0.f;
                if (live) {
                    const float r = yr[c] - f0 - a.Tg[s_target[lane] * 4 + c] / a.scales[4 + c];
                    loss += r * r * inv;
                    d[c] = 2.f * r * inv;
                }
                float sum = d[c];
                for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                if (lane == kTrainRows - 1) d[c] = -sum;
                if (lane == c) put(gp + m_off.ob3 + c, sum - sum, add);   // the rows' gradients cancel: db3 = 0 (or NaN)
            }
            *reinterpret_cast<float4 *>(Y + lane * 4) = make_float4(d[0], d[1], d[2], d[3]);
            for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
            if (lane == 0) put(a.Lp + blockIdx.x, loss, add);
        }
        __syncthreads();
        // dW3 = H2^T dY; dH2 = (dY W3^T) o (1 - h2^2)
        for (int e = t; e < kWidth * 4; e += kTrainThreads) {
            const int m = e >> 2, c = e & 3;
            float s0 = 0.f, s1 = 0.f;
#pragma unroll 8
            for (int r = 0; r < kTrainRows; r += 2) {
                s0 += H2[m * kRS + r] * Y[r * 4 + c];
                s1 += H2[m * kRS + r + 1] * Y[r * 4 + 4 + c];
            }
            put(gp + m_off.oW3 + e, s0 + s1, add);
        }
        for (int e = t; e < kWidth * kTrainRows; e += kTrainThreads) {
            const int m = e / kTrainRows, r = e % kTrainRows;
            const float4 dy = ld4(Y + r * 4), w = ld4(sf + L.W3 + m * 4);
            const float h = H2[m * kRS + r];
            dH2[m * kRS + r] = (dy.x * w.x + dy.y * w.y + dy.z * w.z + dy.w * w.w) * (1.f - h * h);
        }
        __syncthreads();
        // dW2 = H1^T dH2, db2 = sum dH2; dH1 = (dH2 W2^T) o (1 - h1^2)
        outer_sum(H1, kWidth, dH2, gp + m_off.oW2, add);
        rows_times(dH2, sf + L.W2t, kWidth + 4, kWidth, P);
        const int tail = t - (kTrainThreads - kWidth);   // the last 64 threads sum the biases
        if (tail >= 0) put(gp + m_off.ob2 + tail, row_sum(dH2 + tail * kRS), add);
        __syncthreads();
        for (int e = t; e < kWidth * kTrainRows; e += kTrainThreads) {
            const int m = e / kTrainRows, at = m * kRS + e % kTrainRows;
            const float h = H1[at];
            dH1[at] = (P[at] + P[kWidth * kRS + at]) * (1.f - h * h);
        }
        __syncthreads();
        // dW1 = X^T dH1, db1 = sum dH1
        outer_sum(X, n_in, dH1, gp + m_off.oW1, add);
        if (tail >= 0) put(gp + m_off.ob1 + tail, row_sum(dH1 + tail * kRS), add);
    }
}

// G = sum over the blocks of their gradient partials and the iteration's loss
// = sum of the blocks' losses, in a fixed order: 8 threads per parameter take
// every eighth block, and their sums are added in thread order.  ADAM: the
// step of the FP32 master weights and the refresh of the BF16 copy in the same
// launch (G is then not kept).
template <bool ADAM>
__global__ void __launch_bounds__(256) mlp_reduce_kernel(const float *Gp, const float *Lp, int nb, int64_t n_params,
                                                         float *G, float *loss, float *P, __nv_bfloat16 *Pb, float *M,
                                                         float *V, float lr, float b1t, float b2t) {
    __shared__ float part[8][32];
    const int lane = threadIdx.x & 31, grp = threadIdx.x >> 5;
    const int64_t p = blockIdx.x * (int64_t)32 + lane;
    grid_dep_wait();
    grid_dep_launch();
    float g = 0.f;
    if (p < n_params) {
#pragma unroll 8
        for (int b = grp; b < nb; b += 8) g += __ldcg(Gp + b * n_params + p);
    }
    part[grp][lane] = g;
    __syncthreads();
    if (grp == 0 && p < n_params) {
        g = 0.f;
#pragma unroll
        for (int q = 0; q < 8; ++q) g += part[q][lane];
        if (ADAM) {
            const float m = 0.9f * M[p] + 0.1f * g;
            const float v = 0.999f * V[p] + 0.001f * g * g;
            M[p] = m;
            V[p] = v;
            const float w = P[p] - lr * (m / (1.f - b1t)) / (sqrtf(v / (1.f - b2t)) + 1e-8f);
            P[p] = w;
            Pb[p] = __float2bfloat16_rn(w);
        } else {
            G[p] = g;
        }
    }
    if (blockIdx.x == 0 && grp == 1) {
        float l = 0.f;
        for (int b = lane; b < nb; b += 32) l += Lp[b];
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (lane == 0) *loss = l;
    }
}

__global__ void to_bf16(const float *P, __nv_bfloat16 *Pb, int64_t n) {
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p < n) Pb[p] = __float2bfloat16_rn(P[p]);
}

// sums for the scales, one row of 12 per warp (the host adds the rows in warp
// order, so the scales do not depend on the warps' timing): [f] squared
// stencil differences of field f, [4+f] squared targets, [8+f] squared own values
__global__ void mlp_scale_sums(const float *S, const float *Tg, int64_t n_states, int64_t n_snap, int64_t n_all,
                               int64_t n_prog, const int32_t *idx, int n, double *acc) {
    double a[12] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    const int64_t total = n_states * n_prog;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = e / n_prog, i = e - k * n_prog;
        const float *Uk = S + state_of(k, n_snap) * n_all * 4;
        const Rec<float> own = load_rec(Uk, i);
        for (int q = 1; q < n; ++q) {
            const Rec<float> r = load_rec(Uk, idx[i * n + q]);
            const float d0 = r.u - own.u, d1 = r.w - own.w, d2 = r.t - own.t, d3 = r.p - own.p;
            a[0] += d0 * d0; a[1] += d1 * d1; a[2] += d2 * d2; a[3] += d3 * d3;
        }
        const float *tg = Tg + e * 4;
        for (int c = 0; c < 4; ++c) a[4 + c] += (double)tg[c] * tg[c];
        a[8] += (double)own.u * own.u; a[9] += (double)own.w * own.w;
        a[10] += (double)own.t * own.t; a[11] += (double)own.p * own.p;
    }
    for (int c = 0; c < 12; ++c) {
        double v = a[c];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0) acc[((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 12 + c] = v;
    }
}

template <class S_, class D_>
__global__ void restrict_kernel(const S_ *src, const int64_t *map, int64_t n_map, D_ *dst, int64_t block_records,
                                int64_t block_stride) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= n_map) return;
    const int64_t r = e / block_records, loc = e - r * block_records;
    const int64_t s = map[e], d = r * block_stride + loc;
#pragma unroll
    for (int c = 0; c < 4; ++c) dst[d * 4 + c] = (D_)src[s * 4 + c];
}

// dst record of entry e = sum_q w[e][q] src[idx[e][q]] (weighted restriction)
template <class S_>
__global__ void restrict_avg_kernel(const S_ *src, const int64_t *idx, const double *w, int m, int64_t n_map,
                                    float *dst, int64_t block_records, int64_t block_stride) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= n_map) return;
    double a[4] = {0, 0, 0, 0};
    for (int q = 0; q < m; ++q) {
        const double wq = w[e * m + q];
        const int64_t s = idx[e * m + q];
#pragma unroll
        for (int c = 0; c < 4; ++c) a[c] += wq * (double)src[s * 4 + c];
    }
    const int64_t r = e / block_records, loc = e - r * block_records;
    const int64_t d = r * block_stride + loc;
#pragma unroll
    for (int c = 0; c < 4; ++c) dst[d * 4 + c] = (float)a[c];
}

// targets = (next - step(this)) / dt on prognostic records
__global__ void target_kernel(const float *next, const float *stepped, float *tg, int64_t n_prog, float inv_dt) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e < n_prog * 4) tg[e] = (next[e] - stepped[e]) * inv_dt;
}

size_t train_smem(int n_in) { return (size_t)train_layout(n_in).end * sizeof(float); }

void mlp_launch_infer(Mlp &m, Problem &pb, const void *U, void *delta, cudaStream_t s) {
    const size_t smem = net_bytes(m.n_in);
    const dim3 grid(div_up(pb.n_prog, 128)), blk(128);
    if (pb.precision == 64)
        mlp_infer_kernel<double><<<grid, blk, smem, s>>>((const double *)U, pb.idx.p, m.n, pb.n_prog, m.Pb.p, m.P.p, offs_of(m),
                                                         m.scales.p, pb.flags.p, (double *)delta);
    else
        mlp_infer_kernel<float><<<grid, blk, smem, s>>>((const float *)U, pb.idx.p, m.n, pb.n_prog, m.Pb.p, m.P.p, offs_of(m),
                                                        m.scales.p, pb.flags.p, (float *)delta);
    RBF_CHECK_LAUNCH();
}

struct AdamStep {
    float lr = 0.f, b1t = 0.f, b2t = 0.f;   // step size, powers of the decay rates
};

void mlp_launch_train(Mlp &m, Problem &pb, const float *S, const float *Tg, int64_t n_runs, int64_t n_snap,
                      const int64_t *samples, int B, unsigned long long seed, long long iter, float *loss,
                      const AdamStep *adam) {
    TrainArgs a{};
    a.S = S;
    a.Tg = Tg;
    a.n_states = n_runs * (n_snap - 1);
    a.n_snap = n_snap;
    a.n_all = pb.n_all;
    a.n_prog = pb.n_prog;
    a.idx = pb.idx.p;
    a.n = m.n;
    a.samples = samples;
    a.seed = seed;
    a.iter = iter;
    a.B = B;
    a.Pb = m.Pb.p;
    a.P = m.P.p;
    a.scales = m.scales.p;
    const int nb = std::min(div_up(B, kTrainSamples), kTrainSets);
    if (m.Gp.n < (size_t)nb * m.n_params) m.Gp.alloc((size_t)nb * m.n_params);
    if (m.Lp.n < (size_t)nb) m.Lp.alloc(nb);
    a.Gp = m.Gp.p;
    a.n_params = m.n_params;
    a.Lp = m.Lp.p;
    // programmatic dependent launches: the next iteration's gather overlaps
    // this one's reduction
    launch_kernel_smem(mlp_train_kernel, dim3(nb), dim3(kTrainThreads), train_smem(m.n_in), m.st, true, a, offs_of(m));
    const AdamStep s = adam ? *adam : AdamStep{};
    launch_kernel(adam ? mlp_reduce_kernel<true> : mlp_reduce_kernel<false>, dim3(div_up(m.n_params, 32)), dim3(256), m.st,
                  true, (const float *)m.Gp.p, (const float *)m.Lp.p, nb, m.n_params, m.Gr.p, loss, m.P.p, m.Pb.p,
                  m.M.p, m.V.p, s.lr, s.b1t, s.b2t);
}

}  // namespace

void mlp_init(Mlp &m, Problem &pb, void *stream) {
    RBF_REQUIRE(pb.kind == kNS, "the learned correction needs a Navier-Stokes problem");
    RBF_REQUIRE(pb.idx.p != nullptr, "the coarse problem's stencils were released");
    m.st = as_stream(stream);
    m.n = pb.n;
    m.slots = pb.n - 1;
    m.n_in = 4 * m.slots + 4;
    RBF_REQUIRE(m.n_in <= kMaxInputs, "stencil of %d nodes too large for the training kernel", pb.n);
    m.oW1 = 0;
    m.ob1 = m.oW1 + (int64_t)m.n_in * kWidth;
    m.oW2 = m.ob1 + kWidth;
    m.ob2 = m.oW2 + kWidth * kWidth;
    m.oW3 = m.ob2 + kWidth;
    m.ob3 = m.oW3 + kWidth * 4;
    m.n_params = m.ob3 + 4;
    m.P.alloc(m.n_params);
    m.Gr.alloc(m.n_params);
    m.M.alloc(m.n_params);
    m.V.alloc(m.n_params);
    m.Pb.alloc(m.n_params);
    m.scales.alloc(12);
    m.acc.alloc(12 * kScaleWarps);
    m.bad.alloc(1);
    RBF_CUDA(cudaMemsetAsync(m.P.p, 0, m.P.bytes(), m.st));
    RBF_CUDA(cudaMemsetAsync(m.Gr.p, 0, m.Gr.bytes(), m.st));
    RBF_CUDA(cudaMemsetAsync(m.M.p, 0, m.M.bytes(), m.st));
    RBF_CUDA(cudaMemsetAsync(m.V.p, 0, m.V.bytes(), m.st));
    const float ones[12] = {1, 1, 1, 1, 1, 1, 1, 1, 1, 1, 1, 1};
    RBF_CUDA(cudaMemcpyAsync(m.scales.p, ones, sizeof(ones), cudaMemcpyHostToDevice, m.st));
    // the widest network's need: a later, narrower one must not lower the limit
    RBF_CUDA(cudaFuncSetAttribute(mlp_train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)train_smem(kMaxInputs)));
    RBF_CUDA(cudaStreamSynchronize(m.st));
}

}  // namespace rbf

struct rbf_mlp {
    rbf::Mlp impl;
    rbf_problem *coarse = nullptr;
};

using rbf::Mlp;

extern "C" {

int rbf_mlp_create(rbf_mlp **out, rbf_problem *coarse, void *stream) {
    return rbf::guarded([&] {
        RBF_REQUIRE(out && coarse, "null argument");
        *out = nullptr;
        auto *h = new rbf_mlp();
        try {
            h->coarse = coarse;
            rbf::mlp_init(h->impl, coarse->impl, stream);
            *out = h;
        } catch (...) {
            delete h;
            throw;
        }
    });
}

int rbf_mlp_n_params(const rbf_mlp *h, int64_t *out) {
    return rbf::guarded([&] {
        RBF_REQUIRE(h && out, "null argument");
        *out = h->impl.n_params;
    });
}

int rbf_mlp_set_params(rbf_mlp *h, const float *params) {
    return rbf::guarded([&] {
        RBF_REQUIRE(h && params, "null argument");
        Mlp &m = h->impl;
        RBF_CUDA(cudaMemcpyAsync(m.P.p, params, m.P.bytes(), cudaMemcpyHostToDevice, m.st));
        rbf::to_bf16<<<rbf::div_up(m.n_params, 256), 256, 0, m.st>>>(m.P.p, m.Pb.p, m.n_params);
        RBF_CHECK_LAUNCH();
        RBF_CUDA(cudaMemsetAsync(m.M.p, 0, m.M.bytes(), m.st));
        RBF_CUDA(cudaMemsetAsync(m.V.p, 0, m.V.bytes(), m.st));
        RBF_CUDA(cudaMemsetAsync(m.Gr.p, 0, m.Gr.bytes(), m.st));
        m.t = 0;
        RBF_CUDA(cudaStreamSynchronize(m.st));
    });
}

int rbf_mlp_get_params(const rbf_mlp *h, float *params) {
    return rbf::guarded([&] {
        RBF_REQUIRE(h && params, "null argument");
        const Mlp &m = h->impl;
        RBF_CUDA(cudaStreamSynchronize(m.st));
        RBF_CUDA(cudaMemcpy(params, m.P.p, m.P.bytes(), cudaMemcpyDeviceToHost));
    });
}

int rbf_mlp_set_scales(rbf_mlp *h, const float *scales) {
    return rbf::guarded([&] {
        RBF_REQUIRE(h && scales, "null argument");
        for (int c = 0; c < 12; ++c) RBF_REQUIRE(scales[c] > 0.f && std::isfinite(scales[c]), "scales must be > 0");
        RBF_CUDA(cudaMemcpyAsync(h->impl.scales.p, scales, 12 * sizeof(float), cudaMemcpyHostToDevice, h->impl.st));
        RBF_CUDA(cudaStreamSynchronize(h->impl.st));
    });
}

int rbf_mlp_get_scales(const rbf_mlp *h, float *scales) {
    return rbf::guarded([&] {
        RBF_REQUIRE(h && scales, "null argument");
        RBF_CUDA(cudaStreamSynchronize(h->impl.st));
        RBF_CUDA(cudaMemcpy(scales, h->impl.scales.p, 12 * sizeof(float), cudaMemcpyDeviceToHost));
    });
}

int rbf_mlp_fit_scales(rbf_mlp *h, const float *states, const float *targets, int64_t n_runs, int64_t n_snap) {
    return rbf::guarded([&] {
        RBF_REQUIRE(h && states && targets && n_runs > 0 && n_snap >= 2, "bad argument");
        const int64_t n_states = n_runs * (n_snap - 1);
        Mlp &m = h->impl;
        rbf::Problem &pb = h->coarse->impl;
        rbf::mlp_scale_sums<<<rbf::kScaleWarps / 8, 256, 0, m.st>>>(states, targets, n_states, n_snap, pb.n_all,
                                                                   pb.n_prog, pb.idx.p, m.n, m.acc.p);
        RBF_CHECK_LAUNCH();
        std::vector<double> rows(12 * rbf::kScaleWarps);
        RBF_CUDA(cudaMemcpyAsync(rows.data(), m.acc.p, rows.size() * sizeof(double), cudaMemcpyDeviceToHost, m.st));
        RBF_CUDA(cudaStreamSynchronize(m.st));
        double s[12] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
        for (int w = 0; w < rbf::kScaleWarps; ++w)
            for (int c = 0; c < 12; ++c) s[c] += rows[(size_t)w * 12 + c];
        float sc[12];
        const double cnt_in = (double)n_states * pb.n_prog * (m.n - 1), cnt_out = (double)n_states * pb.n_prog;
        for (int c = 0; c < 4; ++c) {
            sc[c] = (float)std::sqrt(std::max(s[c] / cnt_in, 1e-30));
            sc[4 + c] = (float)std::sqrt(std::max(s[4 + c] / cnt_out, 1e-30));
            sc[8 + c] = (float)std::sqrt(std::max(s[8 + c] / cnt_out, 1e-30));
        }
        RBF_CUDA(cudaMemcpyAsync(m.scales.p, sc, sizeof(sc), cudaMemcpyHostToDevice, m.st));
        RBF_CUDA(cudaStreamSynchronize(m.st));
    });
}

int rbf_mlp_grad(rbf_mlp *h, const float *states, const float *targets, int64_t n_runs, int64_t n_snap,
                 const int64_t *samples, int32_t batch, float *grad_host, float *loss_host) {
    return rbf::guarded([&] {
        RBF_REQUIRE(h && states && targets && samples && batch > 0 && n_runs > 0 && n_snap >= 2, "bad argument");
        Mlp &m = h->impl;
        rbf::DevBuf<float> loss(1);
        RBF_CUDA(cudaMemsetAsync(loss.p, 0, sizeof(float), m.st));
        RBF_CUDA(cudaMemsetAsync(m.Gr.p, 0, m.Gr.bytes(), m.st));
        rbf::mlp_launch_train(m, h->coarse->impl, states, targets, n_runs, n_snap, samples, batch, 0, 0, loss.p,
                              nullptr);
        if (grad_host) RBF_CUDA(cudaMemcpyAsync(grad_host, m.Gr.p, m.Gr.bytes(), cudaMemcpyDeviceToHost, m.st));
        if (loss_host) RBF_CUDA(cudaMemcpyAsync(loss_host, loss.p, sizeof(float), cudaMemcpyDeviceToHost, m.st));
        RBF_CUDA(cudaMemsetAsync(m.Gr.p, 0, m.Gr.bytes(), m.st));
        RBF_CUDA(cudaStreamSynchronize(m.st));
    });
}

int rbf_mlp_train(rbf_mlp *h, const float *states, const float *targets, int64_t n_runs, int64_t n_snap,
                  int64_t iters, int32_t batch, float lr, uint64_t seed, float *loss_host) {
    return rbf::guarded([&] {
        RBF_REQUIRE(h && states && targets && n_runs > 0 && n_snap >= 2 && iters >= 0 && batch > 0, "bad argument");
        RBF_REQUIRE(lr > 0.f && std::isfinite(lr), "lr must be > 0");
        Mlp &m = h->impl;
        m.loss.alloc(std::max<int64_t>(iters, 1));
        RBF_CUDA(cudaMemsetAsync(m.loss.p, 0, m.loss.bytes(), m.st));
        for (int64_t it = 0; it < iters; ++it) {
            m.t += 1;
            // cosine decay of the step size over the run
            rbf::AdamStep step;
            step.lr = lr * 0.5f * (1.f + std::cos(3.14159265358979f * (float)it / (float)iters));
            step.b1t = std::pow(0.9f, (float)m.t);
            step.b2t = std::pow(0.999f, (float)m.t);
            rbf::mlp_launch_train(m, h->coarse->impl, states, targets, n_runs, n_snap, nullptr, batch, seed, it,
                                  m.loss.p + it, &step);
        }
        if (loss_host) RBF_CUDA(cudaMemcpyAsync(loss_host, m.loss.p, iters * sizeof(float), cudaMemcpyDeviceToHost, m.st));
        RBF_CUDA(cudaStreamSynchronize(m.st));
    });
}

int rbf_mlp_forward(rbf_mlp *h, const void *U, void *delta) {
    return rbf::guarded([&] {
        RBF_REQUIRE(h && U && delta, "null argument");
        rbf::mlp_launch_infer(h->impl, h->coarse->impl, U, delta, h->impl.st);
    });
}

// The network as the persistent kernel reads it, with strengths alpha.
static rbf::MlpView mlp_view(Mlp &m, const double *alpha) {
    rbf::MlpView mv{};
    mv.Pb = m.Pb.p;
    mv.P = m.P.p;
    mv.oW1 = m.oW1; mv.ob1 = m.ob1; mv.oW2 = m.oW2; mv.ob2 = m.ob2; mv.oW3 = m.oW3; mv.ob3 = m.ob3;
    mv.scales = m.scales.p;
    for (int f = 0; f < 4; ++f) mv.alpha[f] = (float)alpha[f];
    mv.n_in = m.n_in;
    mv.bad = m.bad.p;
    return mv;
}

int rbf_mlp_tune_run(rbf_mlp *h) {
    return rbf::guarded([&] {
        RBF_REQUIRE(h, "null argument");
        Mlp &m = h->impl;
        rbf::Problem &pb = h->coarse->impl;
        RBF_CUDA(cudaStreamSynchronize(pb.st));
        RBF_CUDA(cudaStreamSynchronize(pb.cap));
        const double ones[4] = {1.0, 1.0, 1.0, 1.0};
        RBF_REQUIRE(rbf::persistent_tune_mlp(pb, mlp_view(m, ones)),
                    "no persistent kernel with the network fits this problem");
    });
}

int rbf_learned_run(rbf_mlp *h, double t0, double dt, int64_t n_steps, const double *alpha, void *U,
                    int64_t *n_fallback) {
    return rbf::guarded([&] {
        RBF_REQUIRE(h && U && alpha && n_steps >= 0, "bad argument");
        RBF_REQUIRE((reinterpret_cast<uintptr_t>(U) & 15) == 0, "state must be 16-byte aligned (node-major records)");
        for (int f = 0; f < 4; ++f) RBF_REQUIRE(alpha[f] >= 0.0 && std::isfinite(alpha[f]), "alpha must be >= 0");
        const float4 al = make_float4((float)alpha[0], (float)alpha[1], (float)alpha[2], (float)alpha[3]);
        Mlp &m = h->impl;
        rbf::Problem &pb = h->coarse->impl;
        RBF_CUDA(cudaMemsetAsync(m.bad.p, 0, sizeof(unsigned long long), pb.st));
        if (pb.run_mode == RBF_RUN_PERSISTENT && rbf::persistent_mlp_ready(pb)) {
            // the whole corrected run in one persistent launch (network evaluated
            // at stage 0 of every step from the records in shared memory)
            const rbf::MlpView mv = mlp_view(m, alpha);
            rbf::persistent_run_mlp(pb, dt, n_steps, U, pb.st, mv);
            unsigned long long bad = 0;
            RBF_CUDA(cudaMemcpyAsync(&bad, m.bad.p, sizeof(bad), cudaMemcpyDeviceToHost, pb.st));
            RBF_CUDA(cudaStreamSynchronize(pb.st));
            rbf::persistent_check(pb);
            if (n_fallback) *n_fallback = (int64_t)bad;
            return;
        }
        rbf::DevBuf<unsigned char> delta((size_t)pb.n_prog * 4 * pb.tsize());
        for (int64_t s = 0; s < n_steps; ++s) {
            // features need the ghosts of the current state; then step and add dt * delta
            rbf::enqueue_ghost_fill(pb, U, pb.st);
            rbf::mlp_launch_infer(m, pb, U, delta.p, pb.st);
            rbf::enqueue_rk4_step(pb, t0 + s * dt, dt, U, pb.st, false, 0);
            if (pb.precision == 64)
                rbf::mlp_apply_kernel<double><<<rbf::div_up(pb.n_prog * 4, 256), 256, 0, pb.st>>>(
                    (double *)U, (const double *)delta.p, pb.n_prog, dt, al, m.bad.p);
            else
                rbf::mlp_apply_kernel<float><<<rbf::div_up(pb.n_prog * 4, 256), 256, 0, pb.st>>>(
                    (float *)U, (const float *)delta.p, pb.n_prog, (float)dt, al, m.bad.p);
            RBF_CHECK_LAUNCH();
        }
        unsigned long long bad = 0;
        RBF_CUDA(cudaMemcpyAsync(&bad, m.bad.p, sizeof(bad), cudaMemcpyDeviceToHost, pb.st));
        RBF_CUDA(cudaStreamSynchronize(pb.st));
        if (n_fallback) *n_fallback = (int64_t)bad;
    });
}

int rbf_mlp_destroy(rbf_mlp *h) {
    return rbf::guarded([&] {
        if (!h) return;
        cudaStreamSynchronize(h->impl.st);
        delete h;
    });
}

int rbf_restrict(const void *src, int32_t src_precision, const int64_t *map, int64_t n_map, void *dst,
                 int32_t dst_precision, int64_t block_records, int64_t block_stride, void *stream) {
    return rbf::guarded([&] {
        RBF_REQUIRE(src && map && dst && n_map >= 0 && block_records > 0 && block_stride >= block_records,
                    "bad argument");
        RBF_REQUIRE((src_precision == 32 || src_precision == 64) && (dst_precision == 32 || dst_precision == 64),
                    "precision must be 32 or 64");
        if (n_map == 0) return;
        cudaStream_t s = rbf::as_stream(stream);
        const int grid = rbf::div_up(n_map, 256);
        if (src_precision == 64 && dst_precision == 32)
            rbf::restrict_kernel<double, float><<<grid, 256, 0, s>>>((const double *)src, map, n_map, (float *)dst,
                                                                     block_records, block_stride);
        else if (src_precision == 64)
            rbf::restrict_kernel<double, double><<<grid, 256, 0, s>>>((const double *)src, map, n_map, (double *)dst,
                                                                      block_records, block_stride);
        else if (dst_precision == 32)
            rbf::restrict_kernel<float, float><<<grid, 256, 0, s>>>((const float *)src, map, n_map, (float *)dst,
                                                                    block_records, block_stride);
        else
            rbf::restrict_kernel<float, double><<<grid, 256, 0, s>>>((const float *)src, map, n_map, (double *)dst,
                                                                     block_records, block_stride);
        RBF_CHECK_LAUNCH();
    });
}

int rbf_restrict_weighted(const void *src, int32_t src_precision, const int64_t *idx, const double *w, int32_t m,
                          int64_t n_map, float *dst, int64_t block_records, int64_t block_stride, void *stream) {
    return rbf::guarded([&] {
        RBF_REQUIRE(src && idx && w && dst && m >= 1 && n_map >= 0 && block_records > 0 &&
                        block_stride >= block_records, "bad argument");
        RBF_REQUIRE(src_precision == 32 || src_precision == 64, "precision must be 32 or 64");
        if (n_map == 0) return;
        cudaStream_t s = rbf::as_stream(stream);
        const int grid = rbf::div_up(n_map, 256);
        if (src_precision == 64)
            rbf::restrict_avg_kernel<double><<<grid, 256, 0, s>>>((const double *)src, idx, w, m, n_map, dst,
                                                                  block_records, block_stride);
        else
            rbf::restrict_avg_kernel<float><<<grid, 256, 0, s>>>((const float *)src, idx, w, m, n_map, dst,
                                                                 block_records, block_stride);
        RBF_CHECK_LAUNCH();
    });
}

int rbf_fill_ghosts(rbf_problem *h, void *U) {
    return rbf::guarded([&] {
        RBF_REQUIRE(h && U && h->impl.kind == rbf::kNS, "needs a Navier-Stokes problem and a state");
        RBF_REQUIRE((reinterpret_cast<uintptr_t>(U) & 15) == 0, "state must be 16-byte aligned (node-major records)");
        rbf::enqueue_ghost_fill(h->impl, U, h->impl.st);
    });
}

int rbf_mlp_targets(rbf_problem *h, const float *states, int64_t n_runs, int64_t n_snap, double dt, float *targets) {
    return rbf::guarded([&] {
        RBF_REQUIRE(h && states && targets && n_runs > 0 && n_snap >= 2, "bad argument");
        rbf::Problem &pb = h->impl;
        RBF_REQUIRE(pb.kind == rbf::kNS && pb.precision == 32, "targets need an FP32 Navier-Stokes problem");
        const int64_t rec = pb.n_all * 4;
        rbf::DevBuf<float> tmp(rec);
        for (int64_t r = 0; r < n_runs; ++r)
            for (int64_t k = 0; k + 1 < n_snap; ++k) {
                const float *cur = states + (r * n_snap + k) * rec;
                RBF_CUDA(cudaMemcpyAsync(tmp.p, cur, rec * 4, cudaMemcpyDeviceToDevice, pb.st));
                rbf::enqueue_rk4_step(pb, 0.0, dt, tmp.p, pb.st, false, 0);
                rbf::target_kernel<<<rbf::div_up(pb.n_prog * 4, 256), 256, 0, pb.st>>>(
                    cur + rec, tmp.p, targets + (r * (n_snap - 1) + k) * pb.n_prog * 4, pb.n_prog, (float)(1.0 / dt));
                RBF_CHECK_LAUNCH();
            }
        RBF_CUDA(cudaStreamSynchronize(pb.st));
    });
}

}  // extern "C"
