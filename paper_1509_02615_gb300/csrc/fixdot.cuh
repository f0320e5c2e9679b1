// FP64 stencil sums on the integer units.
//
// GB300's FP64 pipe takes 2 FMAs per SM and clock, its integer units 32
// multiply-adds of 32 x 32 bits into 64 (IMAD.WIDE; both measured).  The twelve
// sums of a node over an n-point stencil are 12 n FMAs, so the FP64 stage
// kernels were bound by that pipe at a quarter of the memory rate.  Here every
// product of a sum is a product of integers, aligned to the largest product of
// that sum:
//
//   weights   w = W 2^(e - 53), 2^52 <= |W| < 2^53 (every bit of the double), in
//             halves W = Wh 2^28 + Wl with Wl in [-2^27, 2^27), packed as
//             (Wh, Wl), 8 bytes like the double; beside it a byte per operator and
//             slot, q = 255 - (er - e) for the row's largest exponent er (0: no
//             weight; weights below 2^-254 of the row's largest are cut there)
//   values    f = M 2^(c - 1075), c the biased exponent and M the 53-bit mantissa;
//             F = M 2^6 shifted right by E - (c + q), E the largest c + q of the
//             sum, in halves F = Fh 2^28 + Fl with Fl in [0, 2^28); formed from the
//             double's bits as it is gathered, per operator
//   sums      hh = sum Wh Fh, cr = sum Wh Fl + Wl Fh (64-bit integers; at most 128
//             products below 2^56 each keep hh in range, cr is folded into hh
//             every sixteen slots), value (hh 2^56 + cr 2^28) 2^(E + er - 1389)
//
// A product keeps its 106 bits down to 2^-58 of the sum's largest product and
// the dropped Wl Fl is below 2^-55 of it, where an FP64 sum rounds every partial
// sum at 2^-53 of itself: the error is bounded by that of the FP64 sum whatever the
// weights and values, and measured two to eight times smaller, except where one
// product outweighs all others together, where both round at that product's last
// place (tests/test_gpu_fixed_point*.py, against 113-bit sums).  An alignment to
// max |w| max |f| instead (one shift per value, exponents from the values alone)
// is a fifth faster, but takes from every product the lead of a value that its
// own weight does not share: a spike a thousand times its neighbours, at its own
// node in a centred derivative, cost them 63 times an FP64 sum's error.
//
// The largest exponents come from a first pass over the stencil's records
// (they stay in L1 or shared memory for the second) and its weights' bytes, and
// the integer sums of a node's lanes are added before anything is rounded, so
// results do not depend on the number of lanes.  Warps with a stencil whose
// values all lie below 2^-950 or so (the tails ahead of every front in a run from
// rest) go to fix_low, the same sums with a look at each value's implicit bit;
// sums of non-finite values, or that would overflow, go to fix_plain: FP64 FMAs
// from the same operands.  (With the tails in fix_plain too, a step of the 25 m
// bubble took 1.29 ms in its first 25 steps from rest, with fix_low 0.94, in a
// developed flow 0.91.)
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

namespace rbf {

constexpr int kFixZero = -4000;   // row exponent of a row of zeros
constexpr int kFixBad = 4000;     // of a row with a weight that is not finite: its sums are NaN

// ---- weights (host and device) ---------------------------------------------
// The exponent er of a row with the given largest magnitude: |w| < 2^er (NaN
// must not be lost on the way: see fix_larger).
__host__ __device__ inline int fix_exponent(double largest) {
    if (largest == 0.0) return kFixZero;
    if (!(largest <= 1.7976931348623157e308)) return kFixBad;
    int e;
    frexp(largest, &e);
    return e;
}
// larger of two magnitudes, or NaN if either is
__host__ __device__ inline double fix_larger(double a, double b) { return a >= b || a != a ? a : b; }
// w as (Wh, Wl) and its exponent byte q for the row exponent er
__host__ __device__ inline int2 fix_weight(double w, int er, unsigned *q) {
    *q = 0;
    if (w == 0.0 || er == kFixBad) return make_int2(0, 0);
    int e;
    const double m = frexp(w, &e);
    const int r = er - e < 254 ? er - e : 254;
    *q = 255u - (unsigned)r;
    const long long W = llrint(ldexp(m, 53 - (er - e - r)));
    const long long h = (W + (1LL << 27)) >> 28;
    return make_int2((int)h, (int)(W - h * (1LL << 28)));
}

// ---- sums (device) ------------------------------------------------------------
// arithmetic shift; amounts above 63 leave the sign
__device__ __forceinline__ long long sar64(long long v, int d) {
    long long r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(d));
    return r;
}
__device__ __forceinline__ void mad_wide(long long &acc, int a, int b) { acc += (long long)a * b; }

// exponent byte o of a slot
template <int O>
__device__ __forceinline__ int fix_byte(unsigned q) {
    return (int)__byte_perm(q, 0, 0x4440 + O);
}

// What the first pass finds of one field's values over the stencil, two 16-bit
// numbers in a word.
struct FixScan {
    unsigned xz = 0, dc = 0;   // largest c + q of d/dx and d/dz; of the third operator, and largest c
    unsigned bits = 0;         // any bit of any value but its sign
    __device__ __forceinline__ void take(unsigned lo, int hi, unsigned qxz, unsigned qd) {
        const unsigned a = (unsigned)hi & 0x7fffffffu, e = (a >> 20) * 0x10001u;
        bits |= lo | a;
        xz = __viaddmax_u16x2(e, qxz, xz);
        dc = __viaddmax_u16x2(e, qd, dc);
    }
    // over the node's G slot lanes (every other lane of the warp)
    template <int G>
    __device__ __forceinline__ void over_lanes() {
#pragma unroll
        for (int k = G; k > 1; k >>= 1) {
            bits |= __shfl_xor_sync(0xffffffffu, bits, k);
            xz = __vmaxu2(xz, __shfl_xor_sync(0xffffffffu, xz, k));
            dc = __vmaxu2(dc, __shfl_xor_sync(0xffffffffu, dc, k));
        }
    }
    __device__ __forceinline__ int E(int o) const { return (int)(o == 0 ? xz & 0xffffu : o == 1 ? xz >> 16 : dc & 0xffffu); }
    // whether the integer sums of operators with row exponents x, z, d hold: the
    // values finite and every result below the largest number
    __device__ __forceinline__ bool holds(int x, int z, int d) const {
        auto one = [&](int e, int er) { return er == kFixZero || e + er <= 2356; };
        return bits == 0 || (dc >> 16 < 2047u && one(E(0), x) && one(E(1), z) && one(E(2), d));
    }
    // whether they take fix_low: results below the normal range and 28 bits above it,
    // or zeros (exponent 0, whose implicit bit is not there) not shifted out
    __device__ __forceinline__ bool low(int x, int z, int d) const {
        auto one = [&](int e, int er) { return er != kFixZero && (e < 324 || e + er < 340); };
        return bits != 0 && (one(E(0), x) || one(E(1), z) || one(E(2), d));
    }
};

// One field's sums with three operators.  LOW: for values at the low end of the
// range too (subnormal ones have exponent 1 and no implicit bit).
template <bool LOW>
struct FixSums {
    long long hh[3], cr[3];
    int E[3];
    __device__ __forceinline__ void start(const FixScan &s) {
#pragma unroll
        for (int o = 0; o < 3; ++o) {
            hh[o] = cr[o] = 0;
            // zeros: everything is shifted out; LOW: no exponent is below 1 + q
            E[o] = s.bits ? (LOW ? max(s.E(o), 256) : s.E(o)) : 0x10000;
        }
    }
    // A value (lo, hi) as F 2^4 without its shift, complemented if negative (so that
    // after the shift the upper word is Fh and the lower one Fl 2^4), and its exponent.
    struct Value {
        long long Y;
        int c;
        __device__ __forceinline__ Value(unsigned lo, int hi) {
            const int s = hi >> 31;
            c = (hi & 0x7fffffff) >> 20;
            const unsigned one = LOW && c == 0 ? 0u : 0x100000u;
            const unsigned T = __funnelshift_r(lo, ((unsigned)hi & 0xfffffu) | one, 22) ^ (unsigned)s;
            Y = (long long)((unsigned long long)T << 32 | ((lo << 10) ^ (unsigned)s));
            if (LOW) c = max(c, 1);
        }
    };
    __device__ __forceinline__ void add(int o, const Value &v, int q, int wh, int wl) {
        const long long F = sar64(v.Y, E[o] - v.c - q);
        int Fh = (int)(F >> 32), Fl = (int)((unsigned)F >> 4);
        // keep the ranges from the compiler: with Fl known to be non-negative it
        // widens the products to 64 x 64 bits
        asm("" : "+r"(Fh), "+r"(Fl));
        mad_wide(hh[o], wh, Fh);
        mad_wide(cr[o], wh, Fl);
        mad_wide(cr[o], wl, Fh);
    }
    __device__ __forceinline__ void fold() {
#pragma unroll
        for (int o = 0; o < 3; ++o) {
            hh[o] += cr[o] >> 28;
            cr[o] &= 0xfffffff;
        }
    }
    // the sum of the G lanes of a node for the row exponent er, after a fold
    template <int G>
    __device__ __forceinline__ double value(int o, int er) const {
        long long h = hh[o], c = cr[o];
#pragma unroll
        for (int k = G; k > 1; k >>= 1) {   // every other lane
            h += __shfl_xor_sync(0xffffffffu, h, k);
            c += __shfl_xor_sync(0xffffffffu, c, k);
        }
        h += c >> 28;
        c &= 0xfffffff;
        const int z = min(__clzll(h ^ (h >> 63)) - 1, 28);   // bits of c that fit below h
        const long long V = (h << z) + (c >> (28 - z));
        if (LOW) return er == kFixZero || E[o] == 0x10000 ? 0.0
                        : er == kFixBad                   ? __hiloint2double(0x7ff80000, 0)
                                                          : ldexp((double)V, E[o] + er - 1333 - z);
        const int e = E[o] + er - 310 - z;   // exponent field of the power of two
        const int hi = er == kFixBad ? 0x7ff80000 : (unsigned)(e - 1) < 2046u ? e << 20 : 0;   // zeros: 0
        return (double)V * __hiloint2double(hi, 0);
    }
};

// selector of the second field's third operator: dissipation (w) or hyperviscosity (pi')
__device__ __forceinline__ unsigned fix_third(int h) { return 0x4442u + (unsigned)h; }

// The first pass over a half's two fields.
struct FixHalfScan {
    FixScan a, b;
    __device__ __forceinline__ void take(const int4 &r, unsigned q, unsigned sel) {
        const unsigned qxz = __byte_perm(q, 0, 0x4140);
        a.take((unsigned)r.x, r.y, qxz, __byte_perm(q, 0, 0x4442));
        b.take((unsigned)r.z, r.w, qxz, __byte_perm(q, 0, sel));
    }
    template <int G>
    __device__ __forceinline__ void over_lanes() {
        a.template over_lanes<G>();
        b.template over_lanes<G>();
    }
    __device__ __forceinline__ bool holds(short4 ew, int h) const {
        return a.holds(ew.x, ew.y, ew.z) && b.holds(ew.x, ew.y, h ? ew.w : ew.z);
    }
    __device__ __forceinline__ bool low(short4 ew, int h) const {
        return a.low(ew.x, ew.y, ew.z) || b.low(ew.x, ew.y, h ? ew.w : ew.z);
    }
};

// One half of a node's sums: two threads share a node (and, with more lanes, a
// slot lane), h = 0 for the fields u, w and h = 1 for theta', pi'.  Each
// gathers its 16-byte half of the neighbours' records and holds the d/dx, d/dz
// and dissipation (pi': hyperviscosity) sums of its two fields: half the
// registers of the whole node, so that twice the warps hide the gathers.
template <bool LOW>
struct FixHalf {
    using Value = typename FixSums<LOW>::Value;
    FixSums<LOW> a, b;
    __device__ __forceinline__ void start(const FixHalfScan &s) {
        a.start(s.a);
        b.start(s.b);
    }
    // sel: which byte of q is the second field's third operator (fix_third)
    __device__ __forceinline__ void slot(const int4 &r, unsigned q, unsigned sel, int xh, int xl, int zh, int zl, int dh,
                                         int dl, int bh, int bl) {
        const int qx = fix_byte<0>(q), qz = fix_byte<1>(q);
        const Value va((unsigned)r.x, r.y);
        a.add(0, va, qx, xh, xl);
        a.add(1, va, qz, zh, zl);
        a.add(2, va, fix_byte<2>(q), dh, dl);
        const Value vb((unsigned)r.z, r.w);
        b.add(0, vb, qx, xh, xl);
        b.add(1, vb, qz, zh, zl);
        b.add(2, vb, (int)__byte_perm(q, 0, sel), bh, bl);
    }
    // two slots from one operand vector of each operator (d: third operator of
    // the first field, e: of the second)
    __device__ __forceinline__ void slots(const int4 &r0, const int4 &r1, uint2 q, unsigned sel, const int4 &x,
                                          const int4 &z, const int4 &d, const int4 &e) {
        slot(r0, q.x, sel, x.x, x.y, z.x, z.y, d.x, d.y, e.x, e.y);
        slot(r1, q.y, sel, x.z, x.w, z.z, z.w, d.z, d.w, e.z, e.w);
    }
    __device__ __forceinline__ void fold() {
        a.fold();
        b.fold();
    }
};
// A half's six sums as doubles (a: first field, b: second; x, z, d).
struct HalfSums {
    double ax, az, ad, bx, bz, bd;
};
template <int G, bool LOW>
__device__ __forceinline__ HalfSums fix_finish(const FixHalf<LOW> &f, short4 ew, int h) {
    const int e = h ? ew.w : ew.z;
    return {f.a.template value<G>(0, ew.x), f.a.template value<G>(1, ew.y), f.a.template value<G>(2, ew.z),
            f.b.template value<G>(0, ew.x), f.b.template value<G>(1, ew.y), f.b.template value<G>(2, e)};
}

// Tendencies of Eqs. (uEq)-(piEq) of the half's two fields from its sums and
// the node's record; the other half's u_x, w_z or pi'_x, pi'_z come by shuffle
// (every lane of the warp takes part).
struct FixPhysics {
    double cp, g_over_tb, theta_bar, dpibar, rd_cv;
};
__device__ __forceinline__ double2 fix_tendency(const HalfSums &s, const FixPhysics &p, int h, double4 c, double pibar,
                                                unsigned char flags) {
    // h = 0 gives u_x, w_z and takes pi'_x, pi'_z; h = 1 the other way round
    const double o0 = __shfl_xor_sync(0xffffffffu, h ? s.bx : s.ax, 1);
    const double o1 = __shfl_xor_sync(0xffffffffu, s.bz, 1);
    double2 k;
    if (h == 0) {
        const double cpth = p.cp * (p.theta_bar + c.z);
        k.x = -c.x * s.ax - c.y * s.az - cpth * o0 + s.ad;
        k.y = -c.x * s.bx - c.y * s.bz - cpth * o1 + p.g_over_tb * c.z + s.bd;
        if (flags & 2) k.x = 0;   // u = 0 held on left/right walls
        if (flags & 1) k.y = 0;   // w = 0 held on bottom/top walls
    } else {
        k.x = -c.x * s.ax - c.y * s.az + s.ad;
        k.y = -c.x * s.bx - c.y * (p.dpibar + s.bz) - p.rd_cv * (pibar + c.w) * (o0 + o1) + s.bd;
    }
    return k;
}

// RK4 update of a half record: stage s < 3 writes U_n + a k and accumulates b k.
__device__ __forceinline__ void fix_rk4_update(int stage, double a, double b, double2 k, const double2 *Un, double2 *K,
                                               double2 *out) {
    const double2 un = *Un;
    if (stage == 3) {
        const double2 k0 = *K;
        *out = make_double2(un.x + (k0.x + b * k.x), un.y + (k0.y + b * k.y));
        return;
    }
    double2 kk = make_double2(b * k.x, b * k.y);
    if (stage > 0) {
        const double2 k0 = *K;
        kk = make_double2(k0.x + b * k.x, k0.y + b * k.y);
    }
    *K = kk;
    *out = make_double2(un.x + a * k.x, un.y + a * k.y);
}

// ---- the launch-per-stage kernels' operand stream -------------------------------
// The operand vectors of a pair of threads (four 16-byte ones per step, two
// fetched by each) pass through a ring in shared memory, two steps ahead of
// their use.
constexpr int kFixThreads = 128, kFixRing = 4;
using FixRing = int4[kFixRing][4][kFixThreads / 2];

struct FixStream {
    const int4 *w;     // the pair's first vector of operator 0
    int64_t ops;       // vectors between operators
    const int4 *nbr;   // its first two neighbours' indices (x, y) and weights' exponent bytes (z, w)
    int64_t step;      // vectors between steps
    int shift;         // added to the indices
    int SLQ;           // steps
};

// Fetches a pair's vectors step by step: `next` is where the thread's two
// vectors of the following step lie.
template <bool CACHED>
struct FixFetch {
    const int4 *next;
    int64_t ops, step;
    int left;       // steps not fetched yet
    unsigned dst;   // shared-memory address of the thread's first vector of ring slot 0
    unsigned kOp;   // bytes between a slot's operators: 16 per pair of the block
    // ring: [kFixRing][4][pairs] vectors
    __device__ __forceinline__ void start(const FixStream &s, int4 *ring, int pairs) {
        const int h = threadIdx.x & 1, pair = threadIdx.x >> 1;
        next = s.w + 2 * h * s.ops;
        ops = s.ops;
        step = s.step;
        left = s.SLQ;
        kOp = sizeof(int4) * pairs;
        dst = (unsigned)__cvta_generic_to_shared(ring + 2 * h * pairs + pair);
    }
    __device__ __forceinline__ void copy(int slot) {   // slot: a constant once the callers are unrolled
        if (left > 0) {
            const unsigned at = dst + slot * 4 * kOp;
            // class tables are shared by neighbouring nodes: through L1
            if (CACHED) {
                asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(at), "l"(next) : "memory");
                asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(at + kOp), "l"(next + ops) : "memory");
            } else {
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(at), "l"(next) : "memory");
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(at + kOp), "l"(next + ops) : "memory");
            }
            next += step;
            --left;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
};

// The thread's part of a half's sums in FP64, for what the integer sums do not
// hold (FixScan::holds): half is the thread's half of record 0, nbr(k) the
// neighbours of step k as in FixStream::nbr.
template <class Nbr>
__device__ __noinline__ HalfSums fix_plain(const int4 *half, Nbr nbr, const int4 *w, int64_t ops, int64_t step, int SLQ,
                                           short4 ew, int h) {
    double s[6] = {0, 0, 0, 0, 0, 0};
    const int er[4] = {ew.x, ew.y, ew.z, h ? ew.w : ew.z};
    for (int k = 0; k < SLQ; ++k, w += step) {
        const int4 j = nbr(k);
        for (int v = 0; v < 2; ++v) {
            const int4 r = half[2 * (int64_t)(v ? j.y : j.x)];
            const unsigned qv = (unsigned)(v ? j.w : j.z);
            double wd[4];
            for (int o = 0; o < 4; ++o) {
                const int4 W = __ldg(w + (o < 3 ? o : 2 + h) * ops);
                const long long i = (long long)(v ? W.z : W.x) * (1LL << 28) + (v ? W.w : W.y);
                const int b = (int)(qv >> (8 * (o < 3 ? o : 2 + h)) & 255u);
                wd[o] = er[o] == kFixBad ? __hiloint2double(0x7ff80000, 0)
                        : b == 0         ? 0.0
                                         : ldexp((double)i, er[o] + b - 308);
            }
            const double fa = __hiloint2double(r.y, r.x), fb = __hiloint2double(r.w, r.z);
            s[0] = fma(wd[0], fa, s[0]);
            s[1] = fma(wd[1], fa, s[1]);
            s[2] = fma(wd[2], fa, s[2]);
            s[3] = fma(wd[0], fb, s[3]);
            s[4] = fma(wd[1], fb, s[4]);
            s[5] = fma(wd[3], fb, s[5]);
        }
    }
    return {s[0], s[1], s[2], s[3], s[4], s[5]};
}

// A half's integer sums at the low end of the range, with the operands straight
// from memory: every lane of the warp takes part if any needs it.
template <int G, class Nbr>
__device__ __noinline__ HalfSums fix_low(const FixHalfScan top, const int4 *half, Nbr nbr, const int4 *w, int64_t ops,
                                         int64_t step, int SLQ, short4 ew, int h) {
    asm volatile("cp.async.wait_all;" ::: "memory");   // what the ring has begun to fetch
    FixHalf<true> f;
    f.start(top);
    const unsigned sel = fix_third(h);
#pragma unroll 2
    for (int k = 0; k < SLQ; ++k, w += step) {
        const int4 j = nbr(k);
        f.slots(half[2 * (int64_t)j.x], half[2 * (int64_t)j.y], make_uint2(j.z, j.w), sel, __ldg(w), __ldg(w + ops),
                __ldg(w + 2 * ops), __ldg(w + (2 + h) * ops));
        if ((k & 7) == 7) f.fold();
    }
    f.fold();
    return fix_finish<G>(f, ew, h);
}

// s, or over the G lanes of plain sums if any of the warp's do not hold (every
// lane of the warp takes part).
template <int G, class Nbr>
__device__ __forceinline__ HalfSums fix_choose(const HalfSums &s, bool holds, const int4 *half, Nbr nbr, const int4 *w,
                                               int64_t ops, int64_t step, int SLQ, short4 ew, int h) {
    if (__all_sync(0xffffffffu, holds)) return s;
    HalfSums p = fix_plain(half, nbr, w, ops, step, SLQ, ew, h);
#pragma unroll
    for (int k = G; k > 1; k >>= 1) {
        p.ax += __shfl_xor_sync(0xffffffffu, p.ax, k);
        p.az += __shfl_xor_sync(0xffffffffu, p.az, k);
        p.ad += __shfl_xor_sync(0xffffffffu, p.ad, k);
        p.bx += __shfl_xor_sync(0xffffffffu, p.bx, k);
        p.bz += __shfl_xor_sync(0xffffffffu, p.bz, k);
        p.bd += __shfl_xor_sync(0xffffffffu, p.bd, k);
    }
    return holds ? s : p;
}

// A half's sums over the records U (two 16-byte halves each); every lane of the
// warp takes part, with the same number of steps.  `fetch` has been started
// and its first two steps copied (constant data, before the wait for the
// preceding kernel).
template <int G, bool CACHED>
__device__ __forceinline__ HalfSums fix_sums(const double *U, const FixStream &s, FixRing &ring, FixFetch<CACHED> &fetch,
                                             short4 ew) {
    const int h = threadIdx.x & 1, pair = threadIdx.x >> 1;
    const int4 *half = reinterpret_cast<const int4 *>(U) + h + 2 * (int64_t)s.shift;
    const unsigned sel = fix_third(h);
    FixHalfScan top;
    const int4 *pn = s.nbr;
#pragma unroll 4
    for (int q = 0; q < s.SLQ; ++q, pn += s.step) {
        const int4 j = __ldg(pn);
        top.take(__ldg(half + 2 * (int64_t)j.x), (unsigned)j.z, sel);
        top.take(__ldg(half + 2 * (int64_t)j.y), (unsigned)j.w, sel);
    }
    top.over_lanes<G>();
    const bool holds = top.holds(ew, h);
    const int4 *first = s.nbr;
    const int64_t step = s.step;
    auto nbr = [first, step](int k) { return __ldg(first + k * step); };
    if (__any_sync(0xffffffffu, top.low(ew, h)))
        return fix_choose<G>(fix_low<G>(top, half, nbr, s.w, s.ops, step, s.SLQ, ew, h), holds, half, nbr, s.w, s.ops, step,
                             s.SLQ, ew, h);
    FixHalf<false> f;
    f.start(top);
    pn = first;
    int4 j = __ldg(pn);
    int4 n0 = __ldg(half + 2 * (int64_t)j.x), n1 = __ldg(half + 2 * (int64_t)j.y);
    uint2 e1 = make_uint2(j.z, j.w);
    pn += s.step;
    if (s.SLQ > 1) j = __ldg(pn);
    const int4 *v = &ring[0][0][pair];
#pragma unroll 1
    for (int q0 = 0; q0 < s.SLQ; q0 += kFixRing) {
#pragma unroll
        for (int u = 0; u < kFixRing; ++u) {
            const int q = q0 + u;
            if (q >= s.SLQ) break;
            const int4 r0 = n0, r1 = n1;
            const uint2 e = e1;
            if (q + 1 < s.SLQ) {   // the next step's records, and the indices of the one after
                n0 = __ldg(half + 2 * (int64_t)j.x);
                n1 = __ldg(half + 2 * (int64_t)j.y);
                e1 = make_uint2(j.z, j.w);
                if (q + 2 < s.SLQ) {
                    pn += s.step;
                    j = __ldg(pn);
                }
            }
            // step q + 2 overwrites slots that were read in step q - 2: step q - 1's
            // barrier lies between
            fetch.copy((u + 2) % kFixRing);
            asm volatile("cp.async.wait_group 2;" ::: "memory");
            __syncwarp();   // the other thread's vectors of this step
            constexpr int kOp = kFixThreads / 2;
            const int4 *w = v + 4 * u * kOp;
            f.slots(r0, r1, e, sel, w[0], w[kOp], w[2 * kOp], w[(2 + h) * kOp]);
        }
        if (q0 & kFixRing) f.fold();
    }
    f.fold();
    return fix_choose<G>(fix_finish<G>(f, ew, h), holds, half, nbr, s.w, s.ops, step, s.SLQ, ew, h);
}

}  // namespace rbf
