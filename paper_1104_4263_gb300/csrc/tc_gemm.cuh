// BF16 tensor-core GEMM on the 5th-generation tensor cores (tcgen05, sm_103a) for the
// learned preconditioner: C(m, n) = alpha * sum_k A(m, k) B(n, k) + beta * C(m, n)
// (+ bias), with FP32 operands in global memory at arbitrary strides, rounded to BF16
// when they are staged into shared memory, and FP32 accumulation in tensor memory.
//
// A CTA of 256 threads computes 128 x BN tiles (BN = 32, 64 or 128) one after another:
//   * the operand tiles of a 64-wide K step are copied by all threads into shared
//     memory in the canonical K-major, no-swizzle layout of the tensor cores (8-row x
//     16-byte core matrices; core matrices adjacent in K are BM * 16 bytes apart, the
//     leading-dimension offset; 8-row groups are 128 bytes apart, the stride offset).
//     A thread moves the 8 consecutive k of a row (one 16-byte shared store) from two
//     16-byte loads where k has unit stride, or 4 rows x 8 k from eight 16-byte loads where
//     the row index has; other strides and unaligned operands take scalar loads;
//   * two tile buffers: the loads of the next one to four steps (of this tile or the next)
//     are in flight in registers while a step is stored, fenced and multiplied and while a
//     finished tile is written, and a buffer is overwritten only when the mbarrier of its
//     last tcgen05.commit has completed (bounded waits);
//   * one elected thread issues the tcgen05.mma (K = 16 each) into a TMEM accumulator of BN
//     columns, in the order of k;
//   * the epilogue reads the accumulator with tcgen05.ld (warp w owns TMEM lanes
//     32 (w mod 4) .. + 31, and half of the columns) and writes C.
// Strides make every transpose of the network's forward and backward passes a plain
// call.  What bounds it at the sizes of a Fourier neural operator: the operands' loads and the
// latency of a tile's chain (loads, barrier, commit, epilogue); the tensor pipe is idle most
// of the time.  Per launch at 16 x 32 x 128^2, one tile per CTA with scalar loads -> this:
// pointwise maps 98 -> 33 us, transforms along x 52 -> 19 us, weight gradients (K = 16384, 16
// tiles) 2145 -> 147 us.
#pragma once

#include "common.cuh"

namespace die {

struct GemmArgs {
    int M = 0, N = 0, K = 0, batch = 1;
    const float* A = nullptr;   // A(m, k) of batch b at A[b * sab + m * sam + k * sak]
    long sam = 0, sak = 0, sab = 0;
    const float* B = nullptr;   // B(n, k) at B[b * sbb + n * sbn + k * sbk]
    long sbn = 0, sbk = 0, sbb = 0;
    float* C = nullptr;         // C(m, n) at C[b * scb + m * scm + n * scn]
    long scm = 0, scn = 0, scb = 0;
    // Two-level output indices (0: one level): an index i with inner extent e steps by
    // (i mod e) s + (i / e) s2.
    int mi = 0, ni = 0, bi = 0;
    long scm2 = 0, scn2 = 0, scb2 = 0;
    float alpha = 1.f, beta = 0.f;   // beta == 0: C is not read
    const float* bias = nullptr;     // optional: + bias[n]
    const float* Cin = nullptr;      // optional: beta * Cin instead of beta * C (C's indices)
    const float* dgelu = nullptr;    // optional: times GELU'(dgelu[..]) (C's indices)
    float* gelu = nullptr;           // optional: receives GELU of C (C's indices)
    int* err = nullptr;              // optional device flag: set to 1 when a wait gave up
    int spare = 0;                   // resident CTAs left to a kernel on another stream
    bool vec16 = false;              // set by tc_gemm: outputs and what is read with them 16-byte aligned
};

// GELU(v) = v Phi(v) and its derivative.
__device__ __forceinline__ float gelu_f(float v) { return v * normcdff(v); }
__device__ __forceinline__ float gelu_d(float v) {
    return normcdff(v) + v * 0.3989422804014327f * __expf(-0.5f * v * v);
}

// Launch on `st`.  DIE_EINVAL on bad sizes or a NULL operand, DIE_ECUDA on a launch error.
die_status tc_gemm(const GemmArgs& g, cudaStream_t st);

}  // namespace die
