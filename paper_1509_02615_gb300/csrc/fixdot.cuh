// FP64 stencil sums on the integer units.
//
// GB300's FP64 pipe takes 2 FMAs per SM and clock, its integer units 32
// multiply-adds of 32 x 32 bits into 64 (IMAD.WIDE; both measured).  The twelve
// sums of a node over an n-point stencil are 12 n FMAs, so the FP64 stage
// kernels were bound by that pipe at a quarter of the memory rate.  Here each
// factor of a sum is a fixed-point number and each product three
// IMAD.WIDEs; sums are exact apart from the product of the two low halves:
//
//   weights   w = W 2^-k, k the largest scale of the node's row of that operator
//             with |W| <= 2^58 and sum |W| <= 2^61; W = Wh 2^28 + Wl with Wl in
//             [-2^27, 2^27); packed as (Wh, Wl), 8 bytes like the double
//   values    f = F 2^(ef - 1078), ef the largest biased exponent of the field
//             in the stencil, F = Fh 2^28 + Fl with Fl in [0, 2^28), |F| < 2^56;
//             formed from the double's bits as it is gathered
//   sums      hh = sum Wh Fh, cr = sum Wh Fl + Wl Fh (64-bit integers: sum |Wh|
//             <= 2^33 + 64 and at most 128 slots keep |hh| <= 2^62 and
//             |cr| < 2^63), value (hh 2^56 + cr 2^28) 2^(ef - k - 1078)
//
// The stencil's largest exponents come from a first pass over its records
// (they stay in L1 or shared memory for the second), so all lanes of a node
// work at the same exponent and their integer sums do not depend on the number
// of lanes.  Against a double, the largest weights keep five bits more and the
// largest values three; smaller ones are cut at that absolute place, and the
// dropped Wl Fl is about 2^-58 of the largest product.  A plain FP64 sum rounds
// every partial sum at 2^-53 of itself, so the fixed-point sum's error is the
// smaller one (two to six times; tests/test_gpu_fixed_point.py measures both
// against 113-bit sums) unless one value of a stencil exceeds the others by
// more than 2^3 where its own weight vanishes: then the others lose what
// exceeds that.
// Exponents below kMinExp (values under 1e-277) count as zero; a non-finite
// value in the stencil makes the field's sums NaN.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

namespace rbf {

constexpr int kFixZero = -4000;   // row exponent of a row of zeros
constexpr int kMinExp = 100;

// ---- weights (host and device) ---------------------------------------------
// The row exponent ew = 58 - k of a row with the given largest magnitude and
// sum of magnitudes: |w| <= 2^ew and sum |w| <= 2^(ew + 3).
__host__ __device__ inline int fix_exponent(double largest, double sum) {
    if (largest == 0.0) return kFixZero;
    int e, s;
    frexp(largest, &e);   // largest < 2^e
    frexp(sum, &s);
    return e > s - 3 ? e : s - 3;
}
// w as (Wh, Wl) for the row exponent ew
__host__ __device__ inline int2 fix_weight(double w, int ew) {
    if (w == 0.0) return make_int2(0, 0);
    const long long W = llrint(ldexp(w, 58 - ew));
    const long long h = (W + (1LL << 27)) >> 28;
    return make_int2((int)h, (int)(W - h * (1LL << 28)));
}

// ---- sums (device) ------------------------------------------------------------
// logical shift; amounts above 31 give 0
__device__ __forceinline__ unsigned shr32(unsigned v, int d) {
    unsigned r;
    asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(d));
    return r;
}
__device__ __forceinline__ void mad_wide(long long &acc, int a, int b) { acc += (long long)a * b; }

// One field's sums with NO operators; e20 = ef << 20.
template <int NO>
struct FixSums {
    long long hh[NO], cr[NO];
    int e20;
    // largest: the stencil's largest high word without its sign
    __device__ __forceinline__ void start(int largest) {
#pragma unroll
        for (int o = 0; o < NO; ++o) hh[o] = cr[o] = 0;
        e20 = max(largest & 0x7ff00000, kMinExp << 20);
    }
    // the value (lo, hi) as F, at the field's exponent: the high 28 bits of its
    // mantissa and the other 25 (left-aligned), shifted down by the exponents'
    // difference in 32-bit shifts (64-bit ones cost twice the instructions)
    __device__ __forceinline__ void split(unsigned lo, int hi, int &Fh, int &Fl) const {
        const unsigned d = (unsigned)(e20 - (hi & 0x7ff00000)) >> 20, s = (unsigned)(hi >> 31);
        const unsigned m = ((unsigned)hi & 0xfffffu) | 0x100000u;
        const unsigned top = __funnelshift_r(lo, m, 25);
        const unsigned low = shr32(__funnelshift_rc(lo << 7, top, d), 4 + max((int)d - 32, 0));
        Fl = (int)((low ^ s) & 0xfffffffu);
        Fh = (int)(shr32(top, d) ^ s);
        // keep the ranges from the compiler: with Fl known to be non-negative it
        // widens the products to 64 x 64 bits
        asm("" : "+r"(Fh), "+r"(Fl));
    }
    __device__ __forceinline__ void add(int o, int wh, int wl, int Fh, int Fl) {
        mad_wide(hh[o], wh, Fh);
        mad_wide(cr[o], wh, Fl);
        mad_wide(cr[o], wl, Fh);
    }
    // the sum of the G lanes of a node for the row exponent ew
    template <int G>
    __device__ __forceinline__ double value(int o, int ew) const {
        long long V = hh[o] * 2 + (cr[o] >> 27);
#pragma unroll
        for (int k = G; k > 1; k >>= 1) V += __shfl_xor_sync(0xffffffffu, V, k);   // every other lane
        const int e = (e20 >> 20) + ew - 58;   // exponent field of 2^(ef + ew - 1081)
        const int hi = e20 == 0x7ff00000 ? 0x7ff80000 : min(max(e, 0), 2046) << 20;
        return (double)V * __hiloint2double(hi, 0);
    }
};

// One half of a node's sums: two threads share a node (and, with more lanes, a
// slot lane), h = 0 for the fields u, w and h = 1 for theta', pi'.  Each
// gathers its 16-byte half of the neighbours' records and holds the d/dx, d/dz
// and dissipation (pi': hyperviscosity) sums of its two fields: half the
// registers of the whole node, so that twice the warps hide the gathers.
struct FixHalf {
    FixSums<3> a, b;
    __device__ __forceinline__ void slot(const int4 &r, int xh, int xl, int zh, int zl, int dh, int dl, int bh, int bl) {
        int Fh, Fl;
        a.split((unsigned)r.x, r.y, Fh, Fl);
        a.add(0, xh, xl, Fh, Fl);
        a.add(1, zh, zl, Fh, Fl);
        a.add(2, dh, dl, Fh, Fl);
        b.split((unsigned)r.z, r.w, Fh, Fl);
        b.add(0, xh, xl, Fh, Fl);
        b.add(1, zh, zl, Fh, Fl);
        b.add(2, bh, bl, Fh, Fl);
    }
    // two slots from one operand vector of each operator (d: third operator of
    // the first field, e: of the second)
    __device__ __forceinline__ void slots(const int4 &r0, const int4 &r1, const int4 &x, const int4 &z, const int4 &d,
                                          const int4 &e) {
        slot(r0, x.x, x.y, z.x, z.y, d.x, d.y, e.x, e.y);
        slot(r1, x.z, x.w, z.z, z.w, d.z, d.w, e.z, e.w);
    }
};

// Largest high words (signs dropped) of a half record's two fields over a stencil.
struct FixLargest {
    int a = 0, b = 0;
    __device__ __forceinline__ void take(const int4 &r) {
        a = max(a, r.y & 0x7fffffff);
        b = max(b, r.w & 0x7fffffff);
    }
    // over the node's G slot lanes (every other lane of the warp)
    template <int G>
    __device__ __forceinline__ void over_lanes() {
#pragma unroll
        for (int k = G; k > 1; k >>= 1) {
            a = max(a, __shfl_xor_sync(0xffffffffu, a, k));
            b = max(b, __shfl_xor_sync(0xffffffffu, b, k));
        }
    }
};

// A half's six sums as doubles (a: first field, b: second; x, z, d).
struct HalfSums {
    double ax, az, ad, bx, bz, bd;
};
template <int G>
__device__ __forceinline__ HalfSums fix_finish(const FixHalf &f, short4 ew, int h) {
    const int e = h ? ew.w : ew.z;
    return {f.a.value<G>(0, ew.x), f.a.value<G>(1, ew.y), f.a.value<G>(2, ew.z),
            f.b.value<G>(0, ew.x), f.b.value<G>(1, ew.y), f.b.value<G>(2, e)};
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
    const int2 *idx;   // its first two neighbour indices
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

// The thread's part of a node's sums over the records U (two 16-byte halves
// each); every lane of the warp takes part, with the same number of steps.
// `fetch` has been started and its first two steps copied (constant data,
// before the wait for the preceding kernel).
template <int G, bool CACHED>
__device__ __forceinline__ void fix_sums(const double *U, const FixStream &s, FixRing &ring, FixFetch<CACHED> &fetch,
                                         FixHalf &f) {
    const int h = threadIdx.x & 1, pair = threadIdx.x >> 1;
    const int4 *half = reinterpret_cast<const int4 *>(U) + h + 2 * (int64_t)s.shift;
    FixLargest top;
    const int2 *pi = s.idx;
#pragma unroll 4
    for (int q = 0; q < s.SLQ; ++q, pi += s.step) {
        const int2 j = __ldg(pi);
        top.take(__ldg(half + 2 * (int64_t)j.x));
        top.take(__ldg(half + 2 * (int64_t)j.y));
    }
    top.over_lanes<G>();
    f.a.start(top.a);
    f.b.start(top.b);
    pi = s.idx;
    int2 j = __ldg(pi);
    int4 n0 = __ldg(half + 2 * (int64_t)j.x), n1 = __ldg(half + 2 * (int64_t)j.y);
    pi += s.step;
    if (s.SLQ > 1) j = __ldg(pi);
    const int4 *v = &ring[0][0][pair];
#pragma unroll 1
    for (int q0 = 0; q0 < s.SLQ; q0 += kFixRing) {
#pragma unroll
        for (int u = 0; u < kFixRing; ++u) {
            const int q = q0 + u;
            if (q >= s.SLQ) break;
            const int4 r0 = n0, r1 = n1;
            if (q + 1 < s.SLQ) {   // the next step's records, and the indices of the one after
                n0 = __ldg(half + 2 * (int64_t)j.x);
                n1 = __ldg(half + 2 * (int64_t)j.y);
                if (q + 2 < s.SLQ) {
                    pi += s.step;
                    j = __ldg(pi);
                }
            }
            // step q + 2 overwrites slots that were read in step q - 2: step q - 1's
            // barrier lies between
            fetch.copy((u + 2) % kFixRing);
            asm volatile("cp.async.wait_group 2;" ::: "memory");
            __syncwarp();   // the other thread's vectors of this step
            constexpr int kOp = kFixThreads / 2;
            const int4 *w = v + 4 * u * kOp;
            f.slots(r0, r1, w[0], w[kOp], w[2 * kOp], w[(2 + h) * kOp]);
        }
    }
}

}  // namespace rbf
