// Operand stream of the FP32 stage kernels: each thread copies its operand
// vectors (four slots of the four packed operators, 64 bytes per step) into its
// own places of a ring in shared memory, two steps ahead of their use, so that
// the stream from memory runs on while the thread waits for its gathers.
//
// The stage is bound by HBM: on 608,256 nodes with n = 37 it moves 437 MB in
// 74 us (0.87 of the copy rate).  With 32-bit indices and plain loads, two steps
// unrolled, a stage of a run (with its ghost kernels) took 84.9 us there, 28.1
// us on 152,576 nodes, whose operands stay in L2, and the 12-member ensemble
// 2.92 ms; with 16-bit indices 84.3 us, 25.7 us and 2.69 ms; with the ring as
// well 82.7 us, 24.4 us and 2.63 ms.  A ring of two steps (83.9 and 27.4 us) leaves more
// of L1 to the gathers but too little in flight; blocks of 128 threads take 84.7
// and 25.3 us.  At 64 registers and 48 KB four blocks share an SM.
#pragma once
#include "common.cuh"
#include "problem.cuh"

namespace rbf {

constexpr int kThreads32 = 256, kRing32 = 3;
using Ring32 = float4[kRing32][4][kThreads32];
// shared memory of a kernel, or next to none in a variant without the ring
template <bool USED>
struct Stage32 {
    Ring32 at;
};
template <>
struct Stage32<false> {
    float4 at[1][4][1];
};

struct Stream32 {
    const float4 *next;      // the following step's vector of operator 0
    int64_t ops, step;       // vectors between operators, between steps
    int left;                // steps not copied yet
    unsigned dst;            // the thread's place in the ring

    __device__ __forceinline__ void start(const void *w, int64_t off0, int64_t n_ops, int64_t n_step, int SLQ,
                                          Ring32 &ring) {
        next = reinterpret_cast<const float4 *>(w) + off0;
        ops = n_ops;
        step = n_step;
        left = SLQ;
        dst = (unsigned)__cvta_generic_to_shared(&ring[0][0][threadIdx.x]);
#pragma unroll
        for (int q = 0; q + 1 < kRing32; ++q) copy(q);
    }
    __device__ __forceinline__ void copy(int slot) {   // slot: a constant once the callers are unrolled
        if (left > 0) {
#pragma unroll
            for (int o = 0; o < 4; ++o)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                 dst + (unsigned)((slot * 4 + o) * kThreads32 * sizeof(float4))),
                             "l"(next + o * ops)
                             : "memory");
            next += step;
            --left;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
};

// Runs vec(indices, x, z, d, h) over the steps.  idx(q): the step's neighbour
// indices.  All threads of a warp that are still running call it together.
template <class Idx, class Vec>
__device__ __forceinline__ void stream_steps(Stream32 &s, Ring32 &ring, int SLQ, Idx idx, Vec vec) {
    int4 j = idx(0);
    for (int q0 = 0; q0 < SLQ; q0 += kRing32) {
#pragma unroll
        for (int u = 0; u < kRing32; ++u) {
            const int q = q0 + u;
            if (q >= SLQ) break;
            __syncwarp();   // the reads of step q - 1 are done: step q + 2 takes their places
            s.copy((u + kRing32 - 1) % kRing32);
            const int4 at = j;
            if (q + 1 < SLQ) j = idx(q + 1);
            asm volatile("cp.async.wait_group %0;" ::"n"(kRing32 - 1) : "memory");
            const float4(*w)[kThreads32] = ring[u];
            const int t = threadIdx.x;
            vec(at, w[0][t], w[1][t], w[2][t], w[3][t]);
        }
    }
}

}  // namespace rbf
