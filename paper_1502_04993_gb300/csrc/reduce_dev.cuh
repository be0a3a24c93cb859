// Row sums of an evaluation, shared by the reductions (reduce.cu) and the fit's line search (fit.cu).
#pragma once

#include "glm_internal.h"

namespace glm {

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

struct ReduceArgs {
    int32_t n;
    int64_t ntile;
    double dt;
    const float* W;
    const float* b;
    const double* C;       // spike term (dL/dW)
    const double* part_s;  // [n][ntile] sums of U - b at the spike bins
    const double* qd;
    const double* part_e;  // [n][ntile]
    int32_t planes;        // planes of part_s and part_e, [planes][n][ntile] (continuous time: CT_PARTS)
    int32_t r0, r1;        // rows outside [r0, r1) (a row range) get L_i = 0 and dL/db_i = 0
    bool spk_from_c;       // spike part q_i b_i + sum_j W_ij C_ij (FP32 form) instead of the part_s sums
    const double* part_self;  // self-delay: [n][ntile] per-tile parts of the diagonal's gradient, or null
    double* gself;            //   their row sums
    double* L_rows;
    double* gb;
    EvalOut* out;          // with the total: where sum_i L_i and the flags go, else null
    int* flags;            // error flags (cleared once reported) and the row blocks' ticket
    unsigned row_blocks;   // the launch's first blocks reduce rows, the others the gradient
};

// sum of p[lane], p[lane + 32], ... in that order, the loads of 8 terms in flight
__device__ __forceinline__ void strided_sums(const double* __restrict__ p, const double* __restrict__ q, int64_t n,
                                             int lane, double& sp, double& sq) {
    for (int64_t t0 = lane; t0 < n; t0 += 32 * 8) {
        double a[8], b[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const bool in = t0 + 32 * u < n;
            a[u] = in ? p[t0 + 32 * u] : 0.0;
            b[u] = (in && q) ? q[t0 + 32 * u] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            sp += a[u];
            sq += b[u];
        }
    }
}

// Whether this block is the last of `blocks` to come here: every other one's writes are then visible to it.
__device__ __forceinline__ bool last_block(int* ticket, unsigned blocks) {
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        last = atomicAdd(ticket, 1) == (int)blocks - 1;
        if (last) *ticket = 0;
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// Sum of v[0 .. n) by one block, in the order of 1024 strided threads whatever the block's size: thread t adds
// v[t], v[t + 1024], ..., warps of 32 by shuffles, then their sums.  Valid in thread 0.
__device__ __forceinline__ double total_1024(const double* v, int32_t n) {
    __shared__ double sh[32];
    const int lane = threadIdx.x & 31;
    for (int w = threadIdx.x >> 5; w < 32; w += blockDim.x >> 5) {
        double s = 0.0;
        for (int32_t i = 32 * w + lane; i < n; i += 1024) s += __ldcg(v + i);
        s = warp_sum(s);
        if (lane == 0) sh[w] = s;
    }
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x < 32) t = warp_sum(sh[lane]);
    return t;
}

// One warp per row.  The lanes' FP64 sums are chains of dependent loads and adds, so eight terms of both sums are
// loaded ahead (N = 1000, 1.8 M bins: rows, gradient and total
// in one launch 73 us, in three with one load in flight 115 us).
__device__ __forceinline__ void reduce_row(const ReduceArgs& A, int32_t i, int lane) {
    double spk = 0.0, integ = 0.0, none = 0.0;
    if (A.spk_from_c) {
        const float* Wi = A.W + (int64_t)i * A.n;
        const double* Ci = A.C + (int64_t)i * A.n;
#pragma unroll 4
        for (int32_t j = lane; j < A.n; j += 32) spk += (double)Wi[j] * Ci[j];
    }
    for (int32_t pl = 0; pl < A.planes; ++pl) {
        const int64_t o = ((int64_t)pl * A.n + i) * A.ntile;
        if (A.spk_from_c) strided_sums(A.part_e + o, nullptr, A.ntile, lane, integ, none);
        else strided_sums(A.part_e + o, A.part_s + o, A.ntile, lane, integ, spk);
    }
    if (A.part_self) {
        double gs = 0.0;
        strided_sums(A.part_self + (int64_t)i * A.ntile, nullptr, A.ntile, lane, gs, none);
        gs = warp_sum(gs);
        if (lane == 0) A.gself[i] = gs;
    }
    spk = warp_sum(spk);
    integ = warp_sum(integ);
    if (lane == 0) {
        const double q = A.qd[i];
        const bool in = i >= A.r0 && i < A.r1;
        A.L_rows[i] = in ? q * (double)A.b[i] + spk - A.dt * integ : 0.0;
        if (A.gb) A.gb[i] = in ? q - A.dt * integ : 0.0;
    }
}

// reduce.cu: the row sums' arguments for context c at (W, b); L_rows and gb (or null) are outputs
ReduceArgs reduce_args(glm_ctx* c, const float* W, const float* b, double* L_rows, double* gb, int64_t ntile);

}  // namespace glm
