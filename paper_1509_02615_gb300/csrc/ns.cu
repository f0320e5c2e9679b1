// a3 + a5 + a6 + a7: packed operators and the fused right-hand side + RK4
// stage kernels of the Navier-Stokes (Sec. 6.2, Eqs. (uEq)-(piEq)) and the
// scalar advection (Sec. 6.1) problems.
//
// Packed layout (SELL with one slice per node group): neighbour slot t of
// node i goes to lane g = t % G, step s = t / G, and is stored at
// [s][i][g].  A warp covers 32/G nodes x G lanes, so every weight and index
// load of a step is one contiguous 128-byte (FP32) or 256-byte (FP64)
// segment.  The G lanes of a node reduce their partial sums with xor
// shuffles and then split the four fields' epilogues between them.
//
// FP32 mode uses the difference form sum_j w_ij (f_j - f_i) (every operator
// here annihilates constants: the p_0 = 1 constraint row of Eq. (weights)),
// which drops the centre slot and keeps cancellation errors relative to the
// local variation.  FP64 mode forms the plain product sum_j w_ij f_j, in fixed
// point on the integer units (fixdot.cuh).
//
// Each stage kernel evaluates all 12 stencil sums of a node (d/dx, d/dz of
// the four fields, the dissipation mu Lap + hyperviscosity on u, w, theta',
// hyperviscosity on pi'), the tendencies of Eqs. (uEq)-(piEq), and the
// classical RK4 update in its epilogue, so one RK4 stage is one pass.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "fixdot.cuh"
#include "stream32.cuh"
#include "problem.cuh"
#include "records.cuh"

namespace rbf {

namespace {

template <class T>
struct NSArgs {
    const T *Uin;     // [n_all][4] stage input (node-major records), ghosts filled
    const T *Un;      // [n_all][4] state at the start of the step
    T *Uout;          // [n_all][4] stage output (prognostic records)
    T *K;             // [n_prog][4] RK4 accumulator
    T *dUdt;          // [n_prog][4] tendency (stage < 0)
    const int32_t *pidx;
    const short4 *pnear;          // FP32: indices relative to the node (nodes without kFarFlag)
    const T *wx, *wz, *wd, *wh;   // FP64: fixed-point pairs (fixdot.cuh), not doubles
    const short4 *wexp;           // FP64: row exponents of each node, or of each class
    const int4 *nbr, *lnbr;       // FP64: neighbours and exponent bytes of two slots, in place of pidx, of loff
    const T *pibar;
    const unsigned char *flags;
    // split stage launches: each of the two launches takes its nodes from
    // nlist (n_list of them; null: every node, one launch per stage)
    const int32_t *nlist;
    int64_t n_list;
    // lattice storage (csrc/lattice.cu): class of each node (-1: per-node
    // operators), and per class the relative index and the packed operators
    // of every slot, [4][n_cls][SLQ][G][V] (null: per-node storage only)
    const int32_t *lcls, *loff;
    const T *lw;
    const short4 *lexp;
    int n_cls;
    int64_t n_prog, n_all;
    int SLQ;          // operand vectors per lane
    int stage;
    T a_next, b_stage;
    T cp, g_over_tb, theta_bar, dpibar, rd_cv;
};

// 16-byte operand vectors of 4 FP32 slots, with matching index vectors.
template <class T>
struct Vec;
template <>
struct Vec<float> {
    static constexpr int V = 4;
    using W = float4;
    using I = int4;
    __device__ static float at(const float4 &v, int k) { return k == 0 ? v.x : k == 1 ? v.y : k == 2 ? v.z : v.w; }
    __device__ static int at(const int4 &v, int k) { return k == 0 ? v.x : k == 1 ? v.y : k == 2 ? v.z : v.w; }
    __device__ static int4 shift(const int4 &v, int d) { return make_int4(v.x + d, v.y + d, v.z + d, v.w + d); }
};

constexpr int kPrefetchVec = 3;   // operand vectors per lane held in registers (prefetch variant)

// Tendencies of Eqs. (uEq)-(piEq) of node i from its record c and its sums,
// and the RK4 update (or the bare tendency when stage < 0); the node's G lanes
// split the four fields between them.
template <class T, int G>
__device__ __forceinline__ void finish_node(const NSArgs<T> &a, int64_t i, int g, const Rec<T> &c, T ux, T uz, T ud, T wx_,
                                            T wz_, T wd_, T tx, T tz, T td, T px, T pz, T ph) {
    const unsigned char fl = a.flags[i];
    const T cpth = a.cp * (a.theta_bar + c.t);
    T k[4];
    k[0] = -c.u * ux - c.w * uz - cpth * px + ud;
    k[1] = -c.u * wx_ - c.w * wz_ - cpth * pz + a.g_over_tb * c.t + wd_;
    k[2] = -c.u * tx - c.w * tz + td;
    k[3] = -c.u * px - c.w * (a.dpibar + pz) - a.rd_cv * (a.pibar[i] + c.p) * (ux + wz_) + ph;
    if (fl & 1) k[1] = 0;   // w = 0 held on bottom/top walls
    if (fl & 2) k[0] = 0;   // u = 0 held on left/right walls
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        if (f % G != g) continue;   // lanes split the four fields' epilogues
        const T kf = k[f];
        const int64_t e = i * 4 + f;
        if (a.stage < 0) {
            a.dUdt[e] = kf;
        } else {
            const T un = a.Un[e];
            if (a.stage == 0) {
                a.K[e] = a.b_stage * kf;
                a.Uout[e] = un + a.a_next * kf;
            } else if (a.stage < 3) {
                a.K[e] += a.b_stage * kf;
                a.Uout[e] = un + a.a_next * kf;
            } else {
                a.Uout[e] = un + (a.K[e] + a.b_stage * kf);
            }
        }
    }
}

// One FP32 RK4 stage (or the bare right-hand side when stage < 0) for G lanes
// per node.  Each lane reads its operands as 16-byte vectors (four slots each)
// and gathers one node record per neighbour.  PF > 0: the lane's operand vectors
// (constant data) are loaded into registers before grid_dep_wait(), so they
// stream in while the preceding ghost kernels finish; PF == 0 streams them
// through a ring in shared memory, with 16-bit indices where they suffice
// (stream32.cuh has the figures).  LAT: a node of a lattice class takes its
// operand vectors from the class table (neighbour = node + offset); the lanes of
// a warp whose nodes share a class read the same table entries, which stay in
// L1, and the nodes outside all classes are few and load plainly.
template <int PF, bool LAT>
constexpr int kStageThreads = PF == 0 && !LAT ? kThreads32 : 256;
template <class T, int G, bool DIFF, int PF, bool LAT>
__global__ void __launch_bounds__(kStageThreads<PF, LAT>, PF > 0 ? 1 : 1024 / kStageThreads<PF, LAT>) ns_stage_kernel(NSArgs<T> a) {
    using VT = Vec<T>;
    using W = typename VT::W;
    using I = typename VT::I;
    constexpr int V = VT::V;
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int g = (int)(tid % G);
    int64_t i = tid / G;
    bool live;
    if (a.nlist) {
        live = i < a.n_list;
        i = __ldg(a.nlist + (live ? i : a.n_list - 1));
    } else {
        live = i < a.n_prog;
        if (!live) i = a.n_prog - 1;   // keep the lanes of the warp in the shuffles
    }
    // lanes without a node leave unless a warp shuffle still needs them
    if (G == 1 ? !live : !__any_sync(0xffffffffu, live)) return;
    const int64_t stride = a.n_prog * G;   // in vectors, between consecutive q
    const int64_t off0 = i * G + g;
    const I *pidx = reinterpret_cast<const I *>(a.pidx);
    const W *wx = reinterpret_cast<const W *>(a.wx), *wz = reinterpret_cast<const W *>(a.wz);
    const W *wd = reinterpret_cast<const W *>(a.wd), *wh = reinterpret_cast<const W *>(a.wh);
    constexpr bool RING = PF == 0 && !LAT;
    // neighbour indices: 16 bits relative to the node where that suffices
    const bool near = RING && !(__ldg(a.flags + i) & kFarFlag);
    auto nbr = [&](int q) {
        const int64_t off = off0 + q * stride;
        return near ? near_at(__ldg(a.pnear + off), (int)i) : __ldg(pidx + off);
    };
    __shared__ Stage32<RING> ring;
    Stream32 st;
    if constexpr (RING) st.start(a.wx, off0, stride * a.SLQ, stride, a.SLQ, ring.at);
    constexpr int R = PF > 0 ? PF : 1;
    I jr[R];
    W rx[R], rz[R], rd[R], rh[R];
    if (PF > 0) {
#pragma unroll
        for (int q = 0; q < R; ++q) {
            if (q < a.SLQ) {
                const int64_t off = off0 + q * stride;
                jr[q] = __ldg(pidx + off);
                rx[q] = __ldg(wx + off);
                rz[q] = __ldg(wz + off);
                rd[q] = __ldg(wd + off);
                rh[q] = __ldg(wh + off);
            }
        }
    }
    grid_dep_wait();     // the stage input (and its ghosts) come from earlier kernels
    grid_dep_launch();
    const T *U = a.Uin;
    Rec<T> fi = {0, 0, 0, 0};
    if (DIFF) fi = load_rec(U, i);
    T ux = 0, uz = 0, ud = 0, wx_ = 0, wz_ = 0, wd_ = 0, tx = 0, tz = 0, td = 0, px = 0, pz = 0, ph = 0;
    auto vec = [&](const I &jv, const W &cx, const W &cz, const W &cd, const W &ch) {
#pragma unroll
        for (int v = 0; v < V; ++v) {
            Rec<T> r = load_rec(U, VT::at(jv, v));
            if (DIFF) { r.u -= fi.u; r.w -= fi.w; r.t -= fi.t; r.p -= fi.p; }
            const T x = VT::at(cx, v), z = VT::at(cz, v), d = VT::at(cd, v), h = VT::at(ch, v);
            ux += x * r.u; uz += z * r.u; ud += d * r.u;
            wx_ += x * r.w; wz_ += z * r.w; wd_ += d * r.w;
            tx += x * r.t; tz += z * r.t; td += d * r.t;
            px += x * r.p; pz += z * r.p; ph += h * r.p;
        }
    };
    if constexpr (RING) {
        stream_steps(st, ring.at, a.SLQ, nbr, vec);
    } else if (PF > 0) {
#pragma unroll
        for (int q = 0; q < R; ++q)
            if (q < a.SLQ) vec(jr[q], rx[q], rz[q], rd[q], rh[q]);
    } else if (LAT && __ldg(a.lcls + i) >= 0) {
        const int c = __ldg(a.lcls + i);
        const I *lo = reinterpret_cast<const I *>(a.loff);
        const W *lw = reinterpret_cast<const W *>(a.lw);
        const int64_t ls = (int64_t)a.n_cls * a.SLQ * G;   // in vectors, between operators
        int64_t off = (int64_t)c * a.SLQ * G + g;
#pragma unroll 2
        for (int q = 0; q < a.SLQ; ++q, off += G)
            vec(VT::shift(__ldg(lo + off), (int)i), __ldg(lw + off), __ldg(lw + ls + off), __ldg(lw + 2 * ls + off),
                __ldg(lw + 3 * ls + off));
    } else {
        int64_t off = off0;
#pragma unroll 2
        for (int q = 0; q < a.SLQ; ++q, off += stride)
            vec(__ldg(pidx + off), __ldg(wx + off), __ldg(wz + off), __ldg(wd + off), __ldg(wh + off));
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
        ux += __shfl_xor_sync(0xffffffffu, ux, o, G);
        uz += __shfl_xor_sync(0xffffffffu, uz, o, G);
        ud += __shfl_xor_sync(0xffffffffu, ud, o, G);
        wx_ += __shfl_xor_sync(0xffffffffu, wx_, o, G);
        wz_ += __shfl_xor_sync(0xffffffffu, wz_, o, G);
        wd_ += __shfl_xor_sync(0xffffffffu, wd_, o, G);
        tx += __shfl_xor_sync(0xffffffffu, tx, o, G);
        tz += __shfl_xor_sync(0xffffffffu, tz, o, G);
        td += __shfl_xor_sync(0xffffffffu, td, o, G);
        px += __shfl_xor_sync(0xffffffffu, px, o, G);
        pz += __shfl_xor_sync(0xffffffffu, pz, o, G);
        ph += __shfl_xor_sync(0xffffffffu, ph, o, G);
    }
    if (!live) return;
    const Rec<T> c = DIFF ? fi : load_rec(U, i);
    finish_node<T, G>(a, i, g, c, ux, uz, ud, wx_, wz_, wd_, tx, tz, td, px, pz, ph);
}

// The FP64 stage (or bare right-hand side): the sums in fixed point
// (fixdot.cuh), everything else in FP64.  On 308,097 scattered nodes with
// n = 56 a stage of a run (with its ghost kernels) took 380 us as 12 x 56 FP64
// FMAs per node (0.95 of the FP64 pipe) and takes 228 us; with one alignment
// per value in place of one per sum, 182 us.  What bounds it: the integer
// pipes, some 70 instructions per slot and thread beside 18 IMAD.WIDEs, and
// under them 109 us of operand traffic at the copy rate.  Five blocks of 128
// threads per SM (96 registers); before fix_low was there five took 224 us, six,
// with spills, 222 us, but the right-hand side of a 125 m box 19.4 us in place
// of 18.6, and seven 249 us.
template <int G, bool LAT>
__global__ void __launch_bounds__(kFixThreads, 5) ns_stage_fixed_kernel(NSArgs<double> a) {
    __shared__ FixRing ring;
    const int64_t pair = (blockIdx.x * (int64_t)kFixThreads + threadIdx.x) >> 1;
    const int h = threadIdx.x & 1, g = (int)(pair % G);
    int64_t i = pair / G;
    bool live;
    if (a.nlist) {
        live = i < a.n_list;
        i = __ldg(a.nlist + (live ? i : a.n_list - 1));
    } else {
        live = i < a.n_prog;
        if (!live) i = a.n_prog - 1;   // keep the lanes of the warp in the shuffles
    }
    if (!__any_sync(0xffffffffu, live)) return;
    FixStream s;
    s.SLQ = a.SLQ;
    s.step = a.n_prog * G;   // in vectors
    s.ops = s.step * a.SLQ;
    s.w = reinterpret_cast<const int4 *>(a.wx) + i * G + g;
    s.nbr = a.nbr + i * G + g;
    s.shift = 0;
    short4 ew;
    const int cl = LAT ? __ldg(a.lcls + i) : -1;
    if (LAT && cl >= 0) {
        s.step = G;
        s.ops = (int64_t)a.n_cls * a.SLQ * G;
        s.w = reinterpret_cast<const int4 *>(a.lw) + (int64_t)cl * a.SLQ * G + g;
        s.nbr = a.lnbr + (int64_t)cl * a.SLQ * G + g;
        s.shift = (int)i;
        ew = __ldg(a.lexp + cl);
    } else {
        ew = __ldg(a.wexp + i);
    }
    FixFetch<LAT> fetch;
    fetch.start(s, &ring[0][0][0], kFixThreads / 2);
    fetch.copy(0);
    fetch.copy(1);
    grid_dep_wait();     // the stage input (and its ghosts) come from earlier kernels
    grid_dep_launch();
    const HalfSums sums = fix_sums<G, LAT>(a.Uin, s, ring, fetch, ew);
    const Rec<double> c = load_rec(a.Uin, i);
    const double2 k = fix_tendency(sums, {a.cp, a.g_over_tb, a.theta_bar, a.dpibar, a.rd_cv}, h,
                                   make_double4(c.u, c.w, c.t, c.p), a.pibar[i], a.flags[i]);
    if (!live || g != 0) return;
    const int64_t e = 2 * i + h;   // the half record of both fields
    if (a.stage < 0) {
        reinterpret_cast<double2 *>(a.dUdt)[e] = k;
        return;
    }
    fix_rk4_update(a.stage, a.a_next, a.b_stage, k, reinterpret_cast<const double2 *>(a.Un) + e,
                   reinterpret_cast<double2 *>(a.K) + e, reinterpret_cast<double2 *>(a.Uout) + e);
}

// Velocity u(x, t) = sum_k c_k(t) (U_k, V_k)(x) with c_k(t) = fa_k + fb_k
// cos(fm_k pi t / T): one separable part for the deformational flow, two for
// the vortex flow of Sec. 6.1.  Packed block k holds part k's flux-form
// weights; the hyperviscosity block follows the parts.  Operand vectors hold
// two slots ([SLQ][n_prog][G][2]).
template <class T>
struct AdvArgs {
    const T *Uin, *Un;
    T *Uout, *K, *dUdt;
    const int32_t *pidx;
    const T *wa, *wa2, *wh;
    int64_t n_prog;
    int SLQ, stage;
    T a_next, b_stage;
    const double *ff;     // the stage's time factors (graph replays) or nullptr
    double t_host, t_frac_dt, period_T;
    double fa[2], fb[2], fm[2];
};

// Time factors of the four stages of the step at time *t (device), after
// setting it to t0 or moving it on by dt: ff[stage][part].  One warp; an FP64
// cosine costs a warp some 1,600 clocks of its SM's FP64 pipe, too much for
// every block of every stage.
struct AdvTimes {
    double t0, dt, frac[4], period_T, fa[2], fb[2], fm[2];
    int set, parts;
};
__global__ void adv_times_kernel(double *t, double *ff, AdvTimes a) {
    grid_dep_wait();
    const double now = a.set ? a.t0 : *t + a.dt;
    __syncwarp();
    if (threadIdx.x == 0) *t = now;
    const int st = threadIdx.x >> 1, k = threadIdx.x & 1;
    if (st < 4 && k < a.parts)
        ff[threadIdx.x] = velocity_time_factor(a.fa[k], a.fb[k], a.fm[k], now + a.frac[st], a.period_T);
}

template <class T>
struct Pair;
template <>
struct Pair<float> {
    using W = float2;
};
template <>
struct Pair<double> {
    using W = double2;
};

constexpr int kAdvAhead = 5;   // operand vectors loaded before the wait for the preceding kernel

// One stage of the advection problem.  Its operands (16 to 28 bytes per slot
// and velocity part) stay in L2 between stages for the problems of Sec. 6.1,
// so a launch is bound by L2 latency and by the gaps between launches: the
// first operand vectors, constant data, load before the wait, two slots each.
template <class T, int G, int NP>
__global__ void __launch_bounds__(256) adv_stage_kernel(AdvArgs<T> a) {
    using W = typename Pair<T>::W;
    __shared__ double s_ff[2];
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int g = (int)(tid % G);
    int64_t i = tid / G;
    const bool live = i < a.n_prog;
    if (!live) i = a.n_prog - 1;
    const int64_t stride = a.n_prog * G, off0 = i * G + g;   // in vectors
    const int2 *pidx = reinterpret_cast<const int2 *>(a.pidx) + off0;
    const W *wa = reinterpret_cast<const W *>(a.wa) + off0, *wh = reinterpret_cast<const W *>(a.wh) + off0;
    const W *wb = NP == 2 ? reinterpret_cast<const W *>(a.wa2) + off0 : nullptr;
    int2 j[kAdvAhead];
    W ra[kAdvAhead], rb[kAdvAhead], rh[kAdvAhead];
#pragma unroll
    for (int q = 0; q < kAdvAhead; ++q) {
        if (q < a.SLQ) {
            j[q] = __ldg(pidx + q * stride);
            ra[q] = __ldg(wa + q * stride);
            if (NP == 2) rb[q] = __ldg(wb + q * stride);
            rh[q] = __ldg(wh + q * stride);
        }
    }
    if (!a.ff && threadIdx.x < NP)   // velocity time factors at this stage's time
        s_ff[threadIdx.x] = velocity_time_factor(a.fa[threadIdx.x], a.fb[threadIdx.x], a.fm[threadIdx.x],
                                                 a.t_host + a.t_frac_dt, a.period_T);
    __syncthreads();
    grid_dep_wait();
    grid_dep_launch();
    T sa = 0, sb = 0, sh = 0;
    auto add = [&](const int2 &jv, const W &ca, const W &cb, const W &ch) {
        const T v0 = a.Uin[jv.x], v1 = a.Uin[jv.y];
        sa += ca.x * v0;
        if (NP == 2) sb += cb.x * v0;
        sh += ch.x * v0;
        sa += ca.y * v1;
        if (NP == 2) sb += cb.y * v1;
        sh += ch.y * v1;
    };
#pragma unroll
    for (int q = 0; q < kAdvAhead; ++q)
        if (q < a.SLQ) add(j[q], ra[q], NP == 2 ? rb[q] : W{}, rh[q]);
#pragma unroll 4
    for (int q = kAdvAhead; q < a.SLQ; ++q)
        add(__ldg(pidx + q * stride), __ldg(wa + q * stride), NP == 2 ? __ldg(wb + q * stride) : W{},
            __ldg(wh + q * stride));
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
        sa += __shfl_xor_sync(0xffffffffu, sa, o, G);
        if (NP == 2) sb += __shfl_xor_sync(0xffffffffu, sb, o, G);
        sh += __shfl_xor_sync(0xffffffffu, sh, o, G);
    }
    if (!live || g != 0) return;
    const double *ff = a.ff ? a.ff : s_ff;
    T kf = (T)ff[0] * sa + sh;
    if (NP == 2) kf += (T)ff[1] * sb;
    if (a.stage < 0) {
        a.dUdt[i] = kf;
    } else {
        const T un = a.Un[i];
        if (a.stage == 0) {
            a.K[i] = a.b_stage * kf;
            a.Uout[i] = un + a.a_next * kf;
        } else if (a.stage < 3) {
            a.K[i] += a.b_stage * kf;
            a.Uout[i] = un + a.a_next * kf;
        } else {
            a.Uout[i] = un + (a.K[i] + a.b_stage * kf);
        }
    }
}

// Packs FP64 weights [ops][n_prog][n] into [n_packed][SLQ][n_prog][G][V] of T
// (slot t = (q G + g) V + v of node i) and the indices alike.
// comb[q][o]: coefficient of weight block o in packed operator q.
template <class T>
__global__ void pack_kernel(const double *__restrict__ w64, const int32_t *__restrict__ idx, int64_t n_prog,
                            int n, int nops, int first, int n_slots, int SLQ, int G, int V, int n_packed,
                            const double *__restrict__ comb, T *__restrict__ pw, int32_t *__restrict__ pidx) {
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int per = SLQ * G * V;
    int64_t total = (int64_t)per * n_prog;
    if (t >= total) return;
    int64_t i = t / per;
    int slot = (int)(t - i * per);
    int v = slot % V, gq = slot / V;
    int g = gq % G, q = gq / G;
    int64_t dst = (((int64_t)q * n_prog + i) * G + g) * V + v;
    if (slot < n_slots) {
        int k = slot + first;
        pidx[dst] = idx[i * n + k];
        for (int p = 0; p < n_packed; ++p) {
            double val = 0.0;
            for (int o = 0; o < nops; ++o) {
                double c = comb[p * nops + o];
                if (c != 0.0) val += c * w64[((int64_t)o * n_prog + i) * n + k];
            }
            pw[(int64_t)p * total + dst] = (T)val;
        }
    } else {
        pidx[dst] = (int32_t)i;
        for (int p = 0; p < n_packed; ++p) pw[(int64_t)p * total + dst] = (T)0;
    }
}

// FP64 operators in fixed point (fixdot.cuh): one warp per node packs its rows
// as pack_kernel does, with (Wh, Wl) pairs in place of the values and their
// exponent bytes beside the indices, and writes the rows' exponents.
__global__ void __launch_bounds__(256) pack_fixed_kernel(const double *__restrict__ w64, const int32_t *__restrict__ idx,
                                                         int64_t n_prog, int n, int nops, int first, int n_slots,
                                                         int SLQ, int G, const double *__restrict__ comb,
                                                         int2 *__restrict__ pw, int4 *__restrict__ nbr,
                                                         short4 *__restrict__ wexp) {
    const int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (i >= n_prog) return;
    constexpr int V = 2;
    const int per = SLQ * G * V;
    const int64_t total = (int64_t)per * n_prog;
    short ex[4];
    for (int p = 0; p < 4; ++p) {
        auto weight = [&](int slot) {
            double val = 0.0;
            for (int o = 0; o < nops; ++o) {
                const double c = comb[p * nops + o];
                if (c != 0.0) val += c * w64[((int64_t)o * n_prog + i) * n + slot + first];
            }
            return val;
        };
        double top = 0.0;
        for (int t = lane; t < n_slots; t += 32) top = fix_larger(top, fabs(weight(t)));
        for (int o = 16; o > 0; o >>= 1) top = fix_larger(top, __shfl_xor_sync(0xffffffffu, top, o));
        const int e = fix_exponent(top);
        ex[p] = (short)e;
        for (int t = lane; t < per; t += 32) {
            const int v = t % V, gq = t / V, g = gq % G, q = gq / G;
            const int64_t dst = (((int64_t)q * n_prog + i) * G + g) * V + v;
            unsigned b = 0;
            pw[p * total + dst] = t < n_slots ? fix_weight(weight(t), e, &b) : make_int2(0, 0);
            int32_t *word = reinterpret_cast<int32_t *>(nbr + dst / V) + v;   // index; exponent bytes at [2]
            word[2] = (p ? word[2] : 0) | (int32_t)(b << (8 * p));
            if (p == 0) word[0] = t < n_slots ? idx[i * n + t + first] : (int32_t)i;
        }
    }
    if (lane == 0) wexp[i] = make_short4(ex[0], ex[1], ex[2], ex[3]);
}

// Neighbour indices relative to the node in 16 bits, in the layout of pidx
// (four slots each), and kFarFlag for the nodes one of whose neighbours is too
// far (ghosts, which follow all prognostic nodes, and the seams of the node
// order), or for all of them without `out`; counts them.  One thread per node.
__global__ void near_indices(const int32_t *__restrict__ pidx, int64_t n_prog, int SLQ, int G, short4 *__restrict__ out,
                             unsigned char *__restrict__ flags, unsigned long long *n_far) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n_prog) return;
    bool far = out == nullptr;
    for (int q = 0; q < SLQ; ++q)
        for (int g = 0; g < G; ++g) {
            const int64_t at = ((int64_t)q * n_prog + i) * G + g;
            const int4 j = reinterpret_cast<const int4 *>(pidx)[at];
            const int64_t d[4] = {j.x - i, j.y - i, j.z - i, j.w - i};
            for (int v = 0; v < 4; ++v) far = far || d[v] < -32768 || d[v] > 32767;
            if (out) out[at] = make_short4((short)d[0], (short)d[1], (short)d[2], (short)d[3]);
        }
    flags[i] = (unsigned char)((flags[i] & ~kFarFlag) | (far ? kFarFlag : 0));
    if (far) atomicAdd(n_far, 1ull);
}

// Advection: packed block k < NP = flux-form weights of velocity part k,
// -(Dx_ij U_k(x_j) + Dy_ij V_k(x_j)); block NP = (-1)^(k+1) gamma Delta^k
// weights; columns folded onto the source node of reflected nodes
// (Sec. 6.1).  Weight blocks in w64: Dx, Dy, Delta^k.  vel holds
// [NP][U, V][n_all].
template <class T>
__global__ void pack_adv_kernel(const double *__restrict__ w64, const int32_t *__restrict__ idx, int64_t n_prog,
                                int64_t n_all, int n, int has_hv, double hvc, const double *__restrict__ vel, int NP,
                                const int32_t *__restrict__ src, int SLQ, int G, T *__restrict__ pw,
                                int32_t *__restrict__ pidx) {
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    constexpr int V = 2;
    const int per = SLQ * G * V;
    int64_t total = (int64_t)per * n_prog;
    if (t >= total) return;
    int64_t i = t / per;
    int slot = (int)(t - i * per);
    int v = slot % V, gq = slot / V;
    int g = gq % G, q = gq / G;
    int64_t dst = (((int64_t)q * n_prog + i) * G + g) * V + v;
    if (slot < n) {
        int j = idx[i * n + slot];
        pidx[dst] = src[j];
        double dx = w64[((int64_t)0 * n_prog + i) * n + slot];
        double dy = w64[((int64_t)1 * n_prog + i) * n + slot];
        for (int k = 0; k < NP; ++k)
            pw[k * total + dst] = (T)(-(dx * vel[(2 * k) * n_all + j] + dy * vel[(2 * k + 1) * n_all + j]));
        pw[NP * total + dst] = has_hv ? (T)(hvc * w64[((int64_t)2 * n_prog + i) * n + slot]) : (T)0;
    } else {
        pidx[dst] = (int32_t)i;
        for (int k = 0; k <= NP; ++k) pw[k * total + dst] = (T)0;
    }
}

template <class T>
__global__ void minmax_kernel(const T *U, int64_t n_prog, int F, double *out, int *bad) {
    // node-major records U[i * F + f]; out[f*2+0] min, out[f*2+1] max via
    // ordered-int atomics on doubles
    for (int f = 0; f < F; ++f) {
        double lo = INFINITY, hi = -INFINITY;
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n_prog; i += (int64_t)gridDim.x * blockDim.x) {
            double v = (double)U[i * F + f];
            if (!isfinite(v)) atomicExch(bad, 1);
            lo = fmin(lo, v);
            hi = fmax(hi, v);
        }
        for (int o = 16; o > 0; o >>= 1) {
            lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
            hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        }
        if ((threadIdx.x & 31) == 0) {
            // monotone map of doubles to signed 64-bit integers
            long long l = __double_as_longlong(lo), h = __double_as_longlong(hi);
            l = l < 0 ? (long long)(0x8000000000000000ULL - (unsigned long long)l) : l;
            h = h < 0 ? (long long)(0x8000000000000000ULL - (unsigned long long)h) : h;
            atomicMin((long long *)&out[f * 2], l);
            atomicMax((long long *)&out[f * 2 + 1], h);
        }
    }
}

template <int G>
void launch_ns_fixed(const NSArgs<double> &a, cudaStream_t s, bool pdl, int prio) {
    const dim3 grid(div_up((a.nlist ? a.n_list : a.n_prog) * G * 2, kFixThreads)), blk(kFixThreads);   // two threads per lane
    if (a.lcls) launch_kernel_prio(ns_stage_fixed_kernel<G, true>, grid, blk, s, pdl, prio, a);
    else launch_kernel_prio(ns_stage_fixed_kernel<G, false>, grid, blk, s, pdl, prio, a);
}

void launch_ns(const NSArgs<double> &a, int G, int, cudaStream_t s, bool pdl, int prio = 0) {
    switch (G) {
        case 1: launch_ns_fixed<1>(a, s, pdl, prio); break;
        case 2: launch_ns_fixed<2>(a, s, pdl, prio); break;
        case 4: launch_ns_fixed<4>(a, s, pdl, prio); break;
        case 8: launch_ns_fixed<8>(a, s, pdl, prio); break;
        default: RBF_FAIL(RBF_E_ARG, "threads per node %d not in {1,2,4,8}", G);
    }
}

template <class T, int G, int PF>
void launch_ns_g(const NSArgs<T> &a, cudaStream_t s, bool pdl, int prio) {
    constexpr bool kDiff = true;   // difference form
    const int threads = a.lcls ? kStageThreads<0, true> : kStageThreads<PF, false>;
    const dim3 grid(div_up((a.nlist ? a.n_list : a.n_prog) * G, threads)), blk(threads);
    if (a.lcls) {
        if (PF == 0) launch_kernel_prio(ns_stage_kernel<T, G, kDiff, 0, true>, grid, blk, s, pdl, prio, a);
        else RBF_FAIL(RBF_E_ARG, "the lattice storage has no prefetch variant");
    } else {
        launch_kernel_prio(ns_stage_kernel<T, G, kDiff, PF, false>, grid, blk, s, pdl, prio, a);
    }
}

void launch_ns(const NSArgs<float> &a, int G, int pf, cudaStream_t s, bool pdl, int prio = 0) {
    if (pf > 0 && a.SLQ > kPrefetchVec)
        RBF_FAIL(RBF_E_ARG, "prefetch variant needs <= %d operand vectors per lane", kPrefetchVec);
    switch (G * 2 + (pf > 0)) {
        case 2: launch_ns_g<float, 1, 0>(a, s, pdl, prio); break;
        case 3: launch_ns_g<float, 1, kPrefetchVec>(a, s, pdl, prio); break;
        case 4: launch_ns_g<float, 2, 0>(a, s, pdl, prio); break;
        case 5: launch_ns_g<float, 2, kPrefetchVec>(a, s, pdl, prio); break;
        case 8: launch_ns_g<float, 4, 0>(a, s, pdl, prio); break;
        case 9: launch_ns_g<float, 4, kPrefetchVec>(a, s, pdl, prio); break;
        case 16: launch_ns_g<float, 8, 0>(a, s, pdl, prio); break;
        case 17: launch_ns_g<float, 8, kPrefetchVec>(a, s, pdl, prio); break;
        default: RBF_FAIL(RBF_E_ARG, "threads per node %d not in {1,2,4,8}", G);
    }
}

template <class T, int NP>
void launch_adv_np(const AdvArgs<T> &a, int G, cudaStream_t s, bool pdl) {
    const dim3 grid(div_up(a.n_prog * G, 256)), blk(256);
    switch (G) {
        case 1: launch_kernel(adv_stage_kernel<T, 1, NP>, grid, blk, s, pdl, a); break;
        case 2: launch_kernel(adv_stage_kernel<T, 2, NP>, grid, blk, s, pdl, a); break;
        case 4: launch_kernel(adv_stage_kernel<T, 4, NP>, grid, blk, s, pdl, a); break;
        case 8: launch_kernel(adv_stage_kernel<T, 8, NP>, grid, blk, s, pdl, a); break;
        default: RBF_FAIL(RBF_E_ARG, "threads per node %d not in {1,2,4,8}", G);
    }
}

template <class T>
void launch_adv(const AdvArgs<T> &a, int G, cudaStream_t s, bool pdl) {
    if (a.wa2) launch_adv_np<T, 2>(a, G, s, pdl);
    else launch_adv_np<T, 1>(a, G, s, pdl);
}

template <class T>
NSArgs<T> ns_args(Problem &pb) {
    NSArgs<T> a{};
    const int64_t total = (int64_t)pb.SLQ * pb.V * pb.G * pb.n_prog;
    const T *pw = (const T *)pb.pw.p;
    a.pidx = pb.pidx.p;
    a.pnear = pb.pnear.p;
    a.wx = pw;
    a.wz = pw + total;
    a.wd = pw + 2 * total;
    a.wh = pw + 3 * total;
    a.wexp = pb.wexp.p;
    a.nbr = pb.nbr.p;
    a.pibar = (const T *)pb.pibar.p;
    a.flags = pb.flags.p;
    if (pb.lat.enabled) {
        a.lexp = pb.lat.lexp.p;
        a.lnbr = pb.lat.lnbr.p;
        a.lcls = pb.lat.cls.p;
        a.loff = pb.lat.loff.p;
        a.lw = (const T *)pb.lat.lw.p;
        a.n_cls = pb.lat.n_cls;
    }
    a.n_prog = pb.n_prog;
    a.n_all = pb.n_all;
    a.SLQ = pb.SLQ;
    a.cp = (T)pb.cp;
    a.g_over_tb = (T)(pb.g / pb.theta_bar);
    a.theta_bar = (T)pb.theta_bar;
    a.dpibar = (T)(-pb.g / (pb.cp * pb.theta_bar));
    a.rd_cv = (T)(pb.rd / pb.cv);
    return a;
}

template <class T>
AdvArgs<T> adv_args(Problem &pb) {
    AdvArgs<T> a{};
    const int64_t total = (int64_t)pb.SL * pb.G * pb.n_prog;
    const T *pw = (const T *)pb.pw.p;
    a.pidx = pb.pidx.p;
    a.wa = pw;
    a.wa2 = pb.n_vparts == 2 ? pw + total : nullptr;
    a.wh = pw + pb.n_vparts * total;
    a.n_prog = pb.n_prog;
    a.SLQ = pb.SLQ;
    a.period_T = pb.period_T;
    for (int k = 0; k < 2; ++k) {
        a.fa[k] = pb.vpart[k][0];
        a.fb[k] = pb.vpart[k][1];
        a.fm[k] = pb.vpart[k][2];
    }
    return a;
}

// RK4 coefficients: stage s writes U_n + a[s] dt k_s and accumulates b[s] dt k_s
const double kA[4] = {0.5, 0.5, 1.0, 0.0};
const double kB[4] = {1.0 / 6.0, 1.0 / 3.0, 1.0 / 3.0, 1.0 / 6.0};

// One RK4 step on stream s.  With the split (pb.split, not while recording
// stage events), each stage runs as two launches: the nodes off the wall set
// on the side stream, the wall set (nodes whose records feed a ghost residual
// or whose stencils read a ghost) on s after the stage's ghost fill.  The
// ghost fill of stage st + 1 needs only the wall set of stage st, so it runs
// while the side stream finishes stage st.  Event pairs alternate by stage
// parity: ev_w[st & 1] marks stage st's wall set, ev_r[st & 1] the rest.
// `first` = false continues a step sequence whose side stream is still open
// (the previous call passed `last` = false); `last` joins the side stream
// back into s.
template <class T>
void rk4_ns(Problem &pb, double dt, T *U, cudaStream_t s, bool rec, int step, bool first, bool last) {
    NSArgs<T> a = ns_args<T>(pb);
    T *S0 = (T *)pb.S0.p, *S1 = (T *)pb.S1.p;
    T *in[4] = {U, S0, S1, S0};
    T *out[4] = {S0, S1, S0, U};
    a.Un = U;
    a.K = (T *)pb.K.p;
    const bool split = pb.split && !rec;
    if (split) {
        RBF_CUDA(cudaEventRecord(pb.ev_fork, s));
        RBF_CUDA(cudaStreamWaitEvent(pb.side, pb.ev_fork, 0));
    }
    for (int st = 0; st < 4; ++st) {
        a.Uin = in[st];
        a.Uout = out[st];
        a.stage = st;
        a.a_next = (T)(kA[st] * dt);
        a.b_stage = (T)(kB[st] * dt);
        if (split) {
            NSArgs<T> ar = a;   // every node off the wall set
            ar.nlist = pb.rlist.p;
            ar.n_list = pb.n_prog - pb.n_wall;
            if (st > 0) RBF_CUDA(cudaStreamWaitEvent(pb.side, pb.ev_w[(st - 1) & 1], 0));
            launch_ns(ar, pb.G, pb.pf, pb.side, pb.pdl);
            RBF_CUDA(cudaEventRecord(pb.ev_r[st & 1], pb.side));
            enqueue_ghost_fill(pb, in[st], s, pb.prio_hi);   // ahead of the other launch's blocks
            if (st > 0 || !first) RBF_CUDA(cudaStreamWaitEvent(s, pb.ev_r[(st + 3) & 1], 0));
            NSArgs<T> aw = a;   // the wall set, ahead of the other launch
            aw.nlist = pb.wlist.p;
            aw.n_list = pb.n_wall;
            launch_ns(aw, pb.G, pb.pf, s, pb.pdl, pb.prio_hi);
            RBF_CUDA(cudaEventRecord(pb.ev_w[st & 1], s));
            continue;
        }
        enqueue_ghost_fill(pb, in[st], s);
        if (rec) RBF_CUDA(cudaEventRecordWithFlags(pb.rhs_ev[(step * 4 + st) * 2], s, cudaEventRecordExternal));
        launch_ns(a, pb.G, pb.pf, s, pb.pdl && !rec);
        if (rec) RBF_CUDA(cudaEventRecordWithFlags(pb.rhs_ev[(step * 4 + st) * 2 + 1], s, cudaEventRecordExternal));
    }
    if (split && last) RBF_CUDA(cudaStreamWaitEvent(s, pb.ev_r[1], 0));
}

// device time factors of the current step, [stage][part], behind the time
double *adv_factors(Problem &pb) { return pb.tdev.p + 8; }

void launch_adv_times(Problem &pb, bool set, double t0, double dt, cudaStream_t s, bool pdl) {
    AdvTimes a{};
    a.t0 = t0;
    a.dt = dt;
    const double frac[4] = {0.0, 0.5, 0.5, 1.0};
    for (int k = 0; k < 4; ++k) a.frac[k] = frac[k] * dt;
    a.period_T = pb.period_T;
    a.parts = pb.n_vparts;
    a.set = set;
    for (int k = 0; k < 2; ++k) {
        a.fa[k] = pb.vpart[k][0];
        a.fb[k] = pb.vpart[k][1];
        a.fm[k] = pb.vpart[k][2];
    }
    launch_kernel(adv_times_kernel, dim3(1), dim3(32), s, pdl, pb.tdev.p, adv_factors(pb), a);
}

template <class T>
void rk4_adv(Problem &pb, double t, double dt, T *U, cudaStream_t s, bool use_tdev, bool rec, int step) {
    AdvArgs<T> a = adv_args<T>(pb);
    T *S0 = (T *)pb.S0.p, *S1 = (T *)pb.S1.p;
    T *in[4] = {U, S0, S1, S0};
    T *out[4] = {S0, S1, S0, U};
    const double frac[4] = {0.0, 0.5, 0.5, 1.0};
    a.Un = U;
    a.K = (T *)pb.K.p;
    a.t_host = t;
    for (int st = 0; st < 4; ++st) {
        a.Uin = in[st];
        a.Uout = out[st];
        a.stage = st;
        a.a_next = (T)(kA[st] * dt);
        a.b_stage = (T)(kB[st] * dt);
        a.t_frac_dt = frac[st] * dt;
        a.ff = use_tdev ? adv_factors(pb) + 2 * st : nullptr;
        if (rec) RBF_CUDA(cudaEventRecordWithFlags(pb.rhs_ev[(step * 4 + st) * 2], s, cudaEventRecordExternal));
        launch_adv<T>(a, pb.G, s, pb.pdl && !rec);
        if (rec) RBF_CUDA(cudaEventRecordWithFlags(pb.rhs_ev[(step * 4 + st) * 2 + 1], s, cudaEventRecordExternal));
    }
    if (use_tdev) launch_adv_times(pb, false, 0.0, dt, s, pb.pdl && !rec);
}

}  // namespace

void pack_operators(Problem &pb, bool near) {
    const int nops = (int)pb.ops.size();
    pb.n_slots = pb.diff ? pb.n - 1 : pb.n;
    // NS: 16-byte operand vectors; advection: two slots per load (37 slots on 4
    // lanes then pad to 40, as with one)
    pb.V = pb.kind == kNS ? (int)(16 / pb.tsize()) : 2;
    pb.SLQ = div_up(pb.n_slots, pb.G * pb.V);
    pb.SL = pb.SLQ * pb.V;
    const int64_t total = (int64_t)pb.SL * pb.G * pb.n_prog;
    const bool fixed = pb.kind == kNS && pb.precision == 64;   // its indices are in pb.nbr
    if (!fixed) pb.pidx.alloc(total);
    if (pb.kind == kAdvection) {
        pb.n_packed = pb.n_vparts + 1;
        pb.pw.alloc((size_t)pb.n_packed * total * pb.tsize());
        const int has_hv = nops > 2;
        if (pb.precision == 64)
            pack_adv_kernel<double><<<div_up(total, 256), 256, 0, pb.st>>>(
                pb.w64.p, pb.idx.p, pb.n_prog, pb.n_all, pb.n, has_hv, pb.hvc, pb.vel.p, pb.n_vparts, pb.src.p,
                pb.SLQ, pb.G, (double *)pb.pw.p, pb.pidx.p);
        else
            pack_adv_kernel<float><<<div_up(total, 256), 256, 0, pb.st>>>(
                pb.w64.p, pb.idx.p, pb.n_prog, pb.n_all, pb.n, has_hv, pb.hvc, pb.vel.p, pb.n_vparts, pb.src.p,
                pb.SLQ, pb.G, (float *)pb.pw.p, pb.pidx.p);
        RBF_CHECK_LAUNCH();
        RBF_CUDA(cudaStreamSynchronize(pb.st));
        return;
    }
    // Navier-Stokes: packed operators as combinations of the FP64 weight blocks
    auto slot = [&](int op) {
        for (int i = 0; i < nops; ++i)
            if (pb.ops[i] == op) return i;
        RBF_FAIL(RBF_E_ARG, "operator %d was not built", op);
    };
    std::vector<double> comb(4 * nops, 0.0);
    pb.n_packed = 4;
    comb[0 * nops + slot(RBF_OP_DX)] = 1.0;
    comb[1 * nops + slot(RBF_OP_DZ)] = 1.0;
    comb[2 * nops + slot(RBF_OP_LAP)] = pb.mu;
    if (pb.hv_k > 0) {
        comb[2 * nops + slot(RBF_OP_HV)] += pb.hvc;
        comb[3 * nops + slot(RBF_OP_HV)] = pb.hvc;
    }
    DevBuf<double> dcomb(comb.size());
    RBF_CUDA(cudaMemcpyAsync(dcomb.p, comb.data(), dcomb.bytes(), cudaMemcpyHostToDevice, pb.st));
    pb.pw.alloc((size_t)pb.n_packed * total * pb.tsize());
    if (pb.precision == 64) {
        // the exponents do not depend on the lanes: one buffer for good, which captured
        // graphs keep reading when a persistent plan packs its own operands
        if (pb.wexp.n != (size_t)pb.n_prog) pb.wexp.alloc(pb.n_prog);
        pb.nbr.alloc(total / pb.V);
        pack_fixed_kernel<<<div_up(pb.n_prog, 8), 256, 0, pb.st>>>(pb.w64.p, pb.idx.p, pb.n_prog, pb.n, nops, pb.diff,
                                                                   pb.n_slots, pb.SLQ, pb.G, dcomb.p, (int2 *)pb.pw.p,
                                                                   pb.nbr.p, pb.wexp.p);
    } else
        pack_kernel<float><<<div_up(total, 256), 256, 0, pb.st>>>(pb.w64.p, pb.idx.p, pb.n_prog, pb.n, nops, pb.diff,
                                                                  pb.n_slots, pb.SLQ, pb.G, pb.V, pb.n_packed,
                                                                  dcomb.p, (float *)pb.pw.p, pb.pidx.p);
    RBF_CHECK_LAUNCH();
    if (near && pb.precision == 32) {
        // a tenth more operand storage, where it leaves room for the states;
        // without it every node is marked far
        size_t free_b = 0, total_b = 0;
        RBF_CUDA(cudaMemGetInfo(&free_b, &total_b));
        pb.pnear.release();
        if (!pb.lat.enabled && free_b >= 8 * (size_t)total) pb.pnear.alloc((size_t)total / 4);
        unsigned long long far = 0;
        DevBuf<unsigned long long> dfar(1);
        RBF_CUDA(cudaMemsetAsync(dfar.p, 0, sizeof(far), pb.st));
        near_indices<<<div_up(pb.n_prog, 256), 256, 0, pb.st>>>(pb.pidx.p, pb.n_prog, pb.SLQ, pb.G, pb.pnear.p,
                                                                pb.flags.p, dfar.p);
        RBF_CHECK_LAUNCH();
        RBF_CUDA(cudaMemcpyAsync(&far, dfar.p, sizeof(far), cudaMemcpyDeviceToHost, pb.st));
        RBF_CUDA(cudaStreamSynchronize(pb.st));
        pb.n_far = (int64_t)far;
    }
    RBF_CUDA(cudaStreamSynchronize(pb.st));
    if (pb.lat.enabled) pack_lattice(pb, comb, nops);
}

void enqueue_set_time(Problem &pb, double t0, double dt, cudaStream_t s) {
    if (pb.kind == kAdvection) launch_adv_times(pb, true, t0, dt, s, false);
}

void enqueue_rk4_step(Problem &pb, double t, double dt, void *U, cudaStream_t s, bool rec, int step, bool first,
                      bool last) {
    const bool tdev = (s == pb.cap);
    if (pb.kind == kNS) {
        if (pb.precision == 64) rk4_ns<double>(pb, dt, (double *)U, s, rec, step, first, last);
        else rk4_ns<float>(pb, dt, (float *)U, s, rec, step, first, last);
    } else {
        if (pb.precision == 64) rk4_adv<double>(pb, t, dt, (double *)U, s, tdev, rec, step);
        else rk4_adv<float>(pb, t, dt, (float *)U, s, tdev, rec, step);
    }
}

void enqueue_rhs(Problem &pb, double t, void *U, void *dUdt, cudaStream_t s) {
    if (pb.kind == kNS) {
        enqueue_ghost_fill(pb, U, s);
        // after the ghost kernels the stage launches early, as in a run, and
        // brings its first operands in while they finish: 26.6 -> 24.6 us per
        // call in FP64 (the 10 km x 10 km box at 125 m)
        const bool pdl = pb.pdl && pb.gh.n_ghost > 0;
        if (pb.precision == 64) {
            NSArgs<double> a = ns_args<double>(pb);
            a.Uin = (const double *)U;
            a.dUdt = (double *)dUdt;
            a.stage = -1;
            launch_ns(a, pb.G, pb.pf, s, pdl);
        } else {
            NSArgs<float> a = ns_args<float>(pb);
            a.Uin = (const float *)U;
            a.dUdt = (float *)dUdt;
            a.stage = -1;
            launch_ns(a, pb.G, pb.pf, s, pdl);
        }
    } else {
        if (pb.precision == 64) {
            AdvArgs<double> a = adv_args<double>(pb);
            a.Uin = (const double *)U;
            a.dUdt = (double *)dUdt;
            a.stage = -1;
            a.t_host = t;
            launch_adv<double>(a, pb.G, s, false);
        } else {
            AdvArgs<float> a = adv_args<float>(pb);
            a.Uin = (const float *)U;
            a.dUdt = (float *)dUdt;
            a.stage = -1;
            a.t_host = t;
            launch_adv<float>(a, pb.G, s, false);
        }
    }
}

// Autotuner: for every (threads per node, register prefetch) choice it
// repacks the operators and times whole RK4 steps through the real launch
// path (ghost kernels, programmatic launches) on a zero state, then keeps the
// fastest; a problem with a wall set then times its steps with split stage
// launches on and off.  The advection problem times its right-hand side per
// lane count.
void autotune_threads_per_node(Problem &pb) {
    const int cands[4] = {1, 2, 4, 8};
    float best = 1e30f;
    int bestG = 4, bestPf = 0;
    cudaEvent_t e0, e1;
    RBF_CUDA(cudaEventCreate(&e0));
    RBF_CUDA(cudaEventCreate(&e1));
    const size_t ts = pb.tsize();
    const int64_t rows = pb.kind == kNS ? pb.n_all : pb.n_prog;
    DevBuf<unsigned char> U((size_t)pb.F * rows * ts);
    DevBuf<unsigned char> D((size_t)pb.F * pb.n_prog * ts);
    RBF_CUDA(cudaMemsetAsync(U.p, 0, U.bytes(), pb.st));
    for (int G : cands) {
        pb.G = G;
        pack_operators(pb);
        for (int pf : {0, kPrefetchVec}) {
            if (pf > 0 && (pb.kind != kNS || pb.precision == 64 || pb.SLQ > kPrefetchVec || pb.lat.enabled)) continue;
            pb.pf = pf;
            float ms = 1e30f;
            for (int rep = 0; rep < 3; ++rep) {
                RBF_CUDA(cudaEventRecord(e0, pb.st));
                for (int it = 0; it < 4; ++it) {
                    if (pb.kind == kNS) enqueue_rk4_step(pb, 0.0, 1e-3, U.p, pb.st, false, 0);
                    else enqueue_rhs(pb, 0.0, U.p, D.p, pb.st);
                }
                RBF_CUDA(cudaEventRecord(e1, pb.st));
                RBF_CUDA(cudaEventSynchronize(e1));
                float t = 0.f;
                RBF_CUDA(cudaEventElapsedTime(&t, e0, e1));
                ms = std::min(ms, t);
            }
            if (ms < best) { best = ms; bestG = G; bestPf = pf; }
        }
    }
    pb.G = bestG;
    pb.pf = bestPf;
    pack_operators(pb);
    if (pb.kind == kNS && pb.wlist.p) {
        // split stage launches, on or off, timed the same way
        float t[2] = {1e30f, 1e30f};
        for (int on = 0; on < 2; ++on) {
            pb.split = on != 0;
            for (int rep = 0; rep < 3; ++rep) {
                RBF_CUDA(cudaEventRecord(e0, pb.st));
                for (int it = 0; it < 4; ++it) enqueue_rk4_step(pb, 0.0, 1e-3, U.p, pb.st, false, 0);
                RBF_CUDA(cudaEventRecord(e1, pb.st));
                RBF_CUDA(cudaEventSynchronize(e1));
                float ms = 0.f;
                RBF_CUDA(cudaEventElapsedTime(&ms, e0, e1));
                t[on] = std::min(t[on], ms);
            }
        }
        pb.split = t[1] < t[0];
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
}

void minmax(Problem &pb, const void *U, double *out) {
    DevBuf<double> d(2 * pb.F);
    DevBuf<int> bad(1);
    std::vector<long long> init(2 * pb.F);
    for (int f = 0; f < pb.F; ++f) {
        init[2 * f] = 0x7fffffffffffffffLL;
        init[2 * f + 1] = (long long)0x8000000000000000ULL;
    }
    RBF_CUDA(cudaMemcpyAsync(d.p, init.data(), d.bytes(), cudaMemcpyHostToDevice, pb.st));
    RBF_CUDA(cudaMemsetAsync(bad.p, 0, sizeof(int), pb.st));
    // an ensemble's records interleave members' ghosts: scan every record
    const int64_t rows = pb.kind == kEnsemble ? pb.n_all : pb.n_prog;
    if (pb.precision == 64) minmax_kernel<double><<<128, 256, 0, pb.st>>>((const double *)U, rows, pb.F, d.p, bad.p);
    else minmax_kernel<float><<<128, 256, 0, pb.st>>>((const float *)U, rows, pb.F, d.p, bad.p);
    RBF_CHECK_LAUNCH();
    std::vector<long long> h(2 * pb.F);
    int hb = 0;
    RBF_CUDA(cudaMemcpyAsync(h.data(), d.p, d.bytes(), cudaMemcpyDeviceToHost, pb.st));
    RBF_CUDA(cudaMemcpyAsync(&hb, bad.p, sizeof(int), cudaMemcpyDeviceToHost, pb.st));
    RBF_CUDA(cudaStreamSynchronize(pb.st));
    for (int q = 0; q < 2 * pb.F; ++q) {
        long long v = h[q];
        if (v < 0) v = (long long)(0x8000000000000000ULL - (unsigned long long)v);
        double dv;
        memcpy(&dv, &v, 8);
        out[q] = dv;
    }
    if (hb) RBF_FAIL(RBF_E_NONFINITE, "non-finite value in the state");
}

}  // namespace rbf
