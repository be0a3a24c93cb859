// Step a7: reductions in a fixed order (bitwise reproducible): the per-tile sums in FP64, the FP32 partials of
// the split products as FP32 TwoSum pairs (~48 bits) converted once to FP64.
//   L_i   = sum_{t in sp(i)} U_i[t] - dt sum_t exp(U_i[t])        (Eq. 7), the spike part as
//           q_i b_i + sum over tiles of (sum of U - b at the row's spike bins) from the U-product epilogue in
//           the 16-bit forms (the bias of the tensor cores' FP32 accumulation of U then cancels between the
//           two parts), and in the plain FP32 form as q_i b_i + sum_j W_ij C_ij in FP64 from the exact spike
//           term C (the same sum, since U - b = W X; free of the FP32 rounding of U summed over the spikes)
//   dL/db_i = q_i - dt sum_t exp(U_i[t])                         (Eq. 12, j = 0)
//   dL/dW_ij = C_ij - sum_s P_s[i][j],  P_s = sum_{t in split s} dt exp(U_i[t]) X_j[t]   (Eq. 12)
//   L = sum_i L_i                                                (Eq. 1)
#include <cmath>

#include "glm_internal.h"
#include "reduce_dev.cuh"

namespace glm {

// a row block of a launch: its rows, then in the last of them L = sum_i L_i and the error flags for the host
__device__ __forceinline__ void reduce_rows_block(const ReduceArgs& A) {
    const int32_t i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (i < A.n) reduce_row(A, i, threadIdx.x & 31);
    if (!A.out || !last_block(A.flags + 2, A.row_blocks)) return;
    const double t = total_1024(A.L_rows, A.n);
    if (threadIdx.x == 0) {
        A.out->total = t;
        A.out->flags[0] = __ldcg(A.flags);
        A.out->flags[1] = __ldcg(A.flags + 1);
        A.flags[0] = A.flags[1] = 0;
    }
}
__global__ void __launch_bounds__(256) reduce_rows_kernel(const __grid_constant__ ReduceArgs A) {
    reduce_rows_block(A);
}

// Sums over the splits p = 0 .. nsplit-1 of the partials of E X^T (part_g, blocked: part_coord), added in split
// order.  The FP32 partials are accumulated as an unevaluated FP32 pair hi + lo with TwoSum (Knuth:
// hi + err = hi_old + v exactly), which keeps ~48 significant bits, and the pair becomes one FP64 value at the
// end: FP64 arithmetic is a scarce pipe on this GPU, and summing the partials in FP64 made these kernels
// pipe-bound at a tenth of the memory bandwidth.
//
// One thread per element of the plane.  A small n has few elements and hundreds of splits (n = 50: 2600 and
// 313), so a thread that walks the splits alone waits for memory all the time; there the block has SUM_GROUPS
// times as many threads, each group loads other splits of the same elements into shared memory while the first
// group adds up the previous round in order.
template <int GROUPS>
constexpr int SUM_E = GROUPS == 1 ? 128 : 64;  // elements per block
constexpr int SUM_GROUPS = 8;
template <int GROUPS>
constexpr int SUM_U = GROUPS == 1 ? 16 : 8;    // loads in flight per thread
// One group and more splits than two such sets (DEEP): the next set loads while the current one is added, or nothing is
// in flight meanwhile: n = 203, 469 splits 27 -> 20 us, n = 500, 152 splits 30 -> 27.  With few splits the registers
// only cost resident warps (n = 2000, 10 splits 67 -> 127 us)
constexpr int SUM_DEEP = 24;

__device__ __forceinline__ void two_sum_f(float& hi, float& lo, float v) {
    const float s = hi + v;
    const float bp = s - hi;
    lo += (hi - (s - bp)) + (v - bp);
    hi = s;
}

// the sum of element e over the splits, valid in the block's first SUM_E<GROUPS> threads
template <int GROUPS, bool DEEP>
__device__ __forceinline__ double sum_parts(const float* __restrict__ part_g, int64_t plane, int64_t e, int nsplit) {
    float hi = 0.f, lo = 0.f;
    const bool in = e < plane;
    const float* src = part_g + (in ? e : 0);
    if constexpr (GROUPS == 1 && DEEP) {
        constexpr int U = SUM_DEEP;
        float v[2][U];
        auto load = [&](int p, float (&d)[U]) {
#pragma unroll
            for (int u = 0; u < U; ++u) d[u] = p + u < nsplit ? __ldcs(src + (p + u) * plane) : 0.f;  // + 0: no change
        };
        load(0, v[0]);
        for (int p = 0; p < nsplit; p += 2 * U) {
            load(p + U, v[1]);
#pragma unroll
            for (int u = 0; u < U; ++u) two_sum_f(hi, lo, v[0][u]);
            load(p + 2 * U, v[0]);
#pragma unroll
            for (int u = 0; u < U; ++u) two_sum_f(hi, lo, v[1][u]);
        }
    } else if constexpr (GROUPS == 1) {
        constexpr int U = SUM_U<1>;
        for (int p = 0; p < nsplit; p += U) {
            float v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) v[u] = p + u < nsplit ? __ldcs(src + (p + u) * plane) : 0.f;  // + 0: no change
#pragma unroll
            for (int u = 0; u < U; ++u) two_sum_f(hi, lo, v[u]);
        }
    } else {
        constexpr int U = SUM_U<GROUPS>, ROUND = GROUPS * U, E = SUM_E<GROUPS>;
        __shared__ float sh[2][ROUND][E];
        const int g = threadIdx.x / E, t = threadIdx.x % E;
        float v[U];
        auto load = [&](int p0) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int p = p0 + u * GROUPS + g;
                v[u] = p < nsplit ? __ldcs(src + p * plane) : 0.f;
            }
        };
        load(0);
        int buf = 0;
        for (int p0 = 0; p0 < nsplit; p0 += ROUND, buf ^= 1) {
#pragma unroll
            for (int u = 0; u < U; ++u) sh[buf][u * GROUPS + g][t] = v[u];
            __syncthreads();  // the other buffer's readers passed the previous round's barrier after their adds
            if (p0 + ROUND < nsplit) load(p0 + ROUND);
            if (g == 0) {
                const int m = min(ROUND, nsplit - p0);
#pragma unroll 8
                for (int k = 0; k < m; ++k) two_sum_f(hi, lo, sh[buf][k][t]);
            }
        }
    }
    return (double)hi + (double)lo;
}

// The rows' sums (the first A.row_blocks blocks) and the gradient (the others) of an evaluation in one launch.
// G rows outside [r0, r1) (a row range) are set to zero.  Self-delay: the diagonal element (i, i) also subtracts
// gself[i] = sum_t dt e^U_i[t] (X_i with the self-delay - X_i)[t], which E X^T does not cover; those sums come from
// reduce_rows_kernel in a launch before (row_blocks = 0 here).
template <int GROUPS, bool DEEP>
__global__ void __launch_bounds__(SUM_E<GROUPS> * GROUPS)
    reduce_eval_kernel(const __grid_constant__ ReduceArgs A, int nsplit, const float* __restrict__ part_g,
                       const double* __restrict__ Gacc, double* __restrict__ G) {
    if (blockIdx.x < A.row_blocks) {
        reduce_rows_block(A);
        return;
    }
    const int32_t n = A.n;
    const int64_t plane = part_plane(n);
    const int64_t eb = (int64_t)(blockIdx.x - A.row_blocks) * SUM_E<GROUPS>;  // the block's first element
    const int64_t e = eb + threadIdx.x % SUM_E<GROUPS>;
    // a block of rows outside the range: there are no partial sums to read (40 rows of N = 2000: 31 us instead of 59)
    bool outside = false;
    if (A.r1 - A.r0 < n) {
        const int64_t brow = 32 * (plane / n);  // elements of 32 rows
        const int64_t last = min(eb + SUM_E<GROUPS>, plane) - 1;
        outside = 32 * (last / brow + 1) <= A.r0 || 32 * (eb / brow) >= A.r1;
    }
    // Gacc: the sums are there already, row-major
    const double s = (Gacc || outside) ? 0.0 : sum_parts<GROUPS, DEEP>(part_g, plane, e, nsplit);
    if (threadIdx.x >= SUM_E<GROUPS> || e >= plane) return;
    int32_t i, j;
    part_coord(n, e, &i, &j);
    if (j >= n) return;
    const int64_t o = (int64_t)i * n + j;
    double g = 0.0;
    if (i >= A.r0 && i < A.r1) {
        g = A.C[o] - (Gacc ? Gacc[o] : s);
        if (A.part_self && i == j) g -= A.gself[i];
    }
    G[o] = g;
}

// C[e] (+)= sum over splits of part_g, in split order.
template <int GROUPS, bool DEEP>
__global__ void __launch_bounds__(SUM_E<GROUPS> * GROUPS)
    sum_splits_kernel(int32_t n, int nsplit, const float* __restrict__ part_g, double* __restrict__ C, bool accumulate) {
    const int64_t plane = part_plane(n);
    const int64_t e = (int64_t)blockIdx.x * SUM_E<GROUPS> + threadIdx.x % SUM_E<GROUPS>;
    const double s = sum_parts<GROUPS, DEEP>(part_g, plane, e, nsplit);
    if (threadIdx.x >= SUM_E<GROUPS> || e >= plane) return;
    int32_t i, j;
    part_coord(n, e, &i, &j);
    if (j >= n) return;
    const int64_t o = (int64_t)i * n + j;
    C[o] = accumulate ? C[o] + s : s;
}

// groups per block: one when the plane's elements, 16 loads each, keep the memory busy by themselves, or the splits are
// few (the whole reduction: n = 203, 469 splits 20 us against 35, n = 317, 391 splits 14 against 33, n = 500, 152
// splits 27 against 72)
static bool many_groups(const glm_ctx* c, int nsplit) {
    return part_plane(c->pb.n) < 200 * (int64_t)c->sm_count && nsplit > 16;
}
static bool deep_loads(int nsplit) { return nsplit > 2 * SUM_DEEP; }
template <int GROUPS>
static unsigned sum_blocks(int32_t n) {
    return (unsigned)((part_plane(n) + SUM_E<GROUPS> - 1) / SUM_E<GROUPS>);
}

cudaError_t launch_sum_splits(glm_ctx* c, int nsplit, double* C, bool accumulate) {
    const int32_t n = c->pb.n;
    constexpr int M = SUM_GROUPS;
    if (many_groups(c, nsplit))
        sum_splits_kernel<M, false><<<sum_blocks<M>(n), SUM_E<M> * M, 0, c->stream>>>(n, nsplit, c->buf.part_g, C, accumulate);
    else if (deep_loads(nsplit))
        sum_splits_kernel<1, true><<<sum_blocks<1>(n), SUM_E<1>, 0, c->stream>>>(n, nsplit, c->buf.part_g, C, accumulate);
    else
        sum_splits_kernel<1, false><<<sum_blocks<1>(n), SUM_E<1>, 0, c->stream>>>(n, nsplit, c->buf.part_g, C, accumulate);
    return cudaGetLastError();
}

// Row i's share of dL/dtau, up to the factor da/dtau = a dt / tau^2 (applied on the host):
//   r_i = sum_t R_i[t] Z_i[t] = sum_{t in sp(i)} Z_i[t] - dt e^{b_i} sum_t e^{v_i[t]} Z_i[t],
// with Z_i = W_i Y, Y = dX/da on the grid, i.e. Z_i[t] = a Z_i[t-1] + v_i[t-1] (v = U - b).  The epilogue
// left per tile k: P1 = sum e^v a^(t-t0), P2 = sum e^v Z_loc, Zend = Z_loc at the next tile, P3 = sum over
// the spike bins of a^(t-t0), P4 = sum over the spike bins of Z_loc; with Z_start(0) = 0 and
// Z_start(k+1) = A Z_start(k) + Zend(k) (A = a^256) a weight family contributes sum_k Z_start(k) P(k) + P'(k).
// Warp per row: lanes own contiguous tile ranges, a shuffle scan supplies each range's Z_start.
__device__ __forceinline__ void tau_row(int32_t n, int32_t i, int64_t ntile, double dt, double A256,
                                        const double* __restrict__ eb, const double* __restrict__ part_tau,
                                        double* __restrict__ rows) {
    const int lane = threadIdx.x & 31;
    if (i >= n) return;
    const int64_t plane = (int64_t)n * ntile;
    const double* p1 = part_tau + (int64_t)i * ntile;
    const double* p2 = p1 + plane;
    const double* ze = p1 + 2 * plane;
    const double* p3 = p1 + 3 * plane;
    const double* p4 = p1 + 4 * plane;
    const int64_t len = (ntile + 31) / 32;
    const int64_t k0 = min((int64_t)lane * len, ntile), k1 = min(k0 + len, ntile);
    // with z = Z_start relative to the range start (0) and w = A^(k - k0):
    double z = 0.0, w = 1.0, Qe = 0.0, Se = 0.0, Qs = 0.0, Ss = 0.0;
    constexpr int U = 4;  // tiles loaded ahead of the recursion
    for (int64_t kb = k0; kb < k1; kb += U) {
        double c[U][5];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t k = min(kb + u, k1 - 1);
            c[u][0] = p1[k], c[u][1] = p2[k], c[u][2] = ze[k], c[u][3] = p3[k], c[u][4] = p4[k];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (kb + u >= k1) break;
            Qe = fma(w, c[u][0], Qe);
            Se += fma(z, c[u][0], c[u][1]);
            Qs = fma(w, c[u][3], Qs);
            Ss += fma(z, c[u][3], c[u][4]);
            z = fma(A256, z, c[u][2]);
            w *= A256;
        }
    }
    double v = z, m = w;
    for (int d = 1; d < 32; d <<= 1) {
        const double o = __shfl_up_sync(0xffffffffu, v, d), om = __shfl_up_sync(0xffffffffu, m, d);
        if (lane >= d) {
            v = fma(m, o, v);
            m *= om;
        }
    }
    double zin = __shfl_up_sync(0xffffffffu, v, 1);
    if (lane == 0) zin = 0.0;
    double integ = fma(zin, Qe, Se);
    double spk = fma(zin, Qs, Ss);
    integ = warp_sum(integ);
    spk = warp_sum(spk);
    if (lane == 0) rows[i] = spk - dt * eb[i] * integ;
}

// Continuous time: row i's dL/dtau itself, r_i = sum_{spikes} z / tau^2 - e^{c_i} (sum_m e^sh (G_m / tau) z_m /
// tau + sum_m e^sh dF_m/dtau), with z = W y at the column starts (y = tau^2 dv/dtau).  The epilogue left,
// per tile and part of a tile's columns (in column order: tile-major, part-minor), the sums P1, P2, Zend,
// P3, P4, Pex and the part's decay product Aend; with z_start of the first segment 0 (no input before
// t_begin) and z_start(next) = Aend z_start + Zend, a weight family contributes sum z_start P + P'.  The
// chain of segments is cut into contiguous lane ranges as in tau_rows_kernel, each range's own decay
// product composing the shuffle scan.
__device__ __forceinline__ void ct_tau_row(int32_t n, int32_t i, int64_t ntile, double tau,
                                           const double* __restrict__ eb, const double* __restrict__ part_tau,
                                           double* __restrict__ rows) {
    const int lane = threadIdx.x & 31;
    if (i >= n) return;
    const int64_t pl = (int64_t)CT_PARTS * n * ntile;  // one value over all parts, rows and tiles
    const int64_t nseg = ntile * CT_PARTS;
    const int64_t len = (nseg + 31) / 32;
    const int64_t s0 = min((int64_t)lane * len, nseg), s1 = min(s0 + len, nseg);
    double z = 0.0, w = 1.0, Qe = 0.0, Se = 0.0, Qs = 0.0, Ss = 0.0, Ex = 0.0;
    constexpr int U = 4;  // segments loaded ahead of the recursion
    for (int64_t sb = s0; sb < s1; sb += U) {
        double c[U][7];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t sg = min(sb + u, s1 - 1), tile = sg / CT_PARTS, part = sg % CT_PARTS;
            const int64_t o = (part * n + i) * ntile + tile;
#pragma unroll
            for (int x = 0; x < 7; ++x) c[u][x] = part_tau[x * pl + o];  // P1, P2, Zend, P3, P4, Pex, Aend
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (sb + u >= s1) break;
            Qe = fma(w, c[u][0], Qe);
            Se += fma(z, c[u][0], c[u][1]);
            Qs = fma(w, c[u][3], Qs);
            Ss += fma(z, c[u][3], c[u][4]);
            Ex += c[u][5];
            z = fma(c[u][6], z, c[u][2]);
            w *= c[u][6];
        }
    }
    double v = z, m = w;
    for (int d = 1; d < 32; d <<= 1) {
        const double o = __shfl_up_sync(0xffffffffu, v, d), om = __shfl_up_sync(0xffffffffu, m, d);
        if (lane >= d) {
            v = fma(m, o, v);
            m *= om;
        }
    }
    double zin = __shfl_up_sync(0xffffffffu, v, 1);
    if (lane == 0) zin = 0.0;
    double integ = fma(zin, Qe, Se);
    double spk = fma(zin, Qs, Ss);
    integ = warp_sum(integ);
    spk = warp_sum(spk);
    Ex = warp_sum(Ex);
    if (lane == 0) rows[i] = spk / (tau * tau) - eb[i] * (integ / tau + Ex);
}

// a warp per row; with out, the last block adds the rows up
__global__ void tau_rows_kernel(int32_t n, int64_t ntile, double dt, double tau, double A256, bool ct,
                                const double* __restrict__ eb, const double* __restrict__ part_tau, double* rows,
                                EvalOut* out, int* ticket) {
    const int32_t i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (ct) ct_tau_row(n, i, ntile, tau, eb, part_tau, rows);
    else tau_row(n, i, ntile, dt, A256, eb, part_tau, rows);
    if (!out || !last_block(ticket, gridDim.x)) return;
    const double t = total_1024(rows, n);
    if (threadIdx.x == 0) out->gtau = t;
}

cudaError_t launch_tau_rows(glm_ctx* c, double* rows, bool total) {
    const Problem& P = c->pb;
    const double A256 = P.ct ? 0.0 : std::exp(-(double)SEG * P.dt / P.tau);
    tau_rows_kernel<<<(P.n + 7) / 8, 256, 0, c->stream>>>(P.n, P.Tpad / tc_tile_t(), P.dt, P.tau, A256, P.ct, c->buf.eb,
                                                          c->buf.part_tau, rows, total ? c->out_dev : nullptr,
                                                          c->buf.flags + 3);
    return cudaGetLastError();
}

ReduceArgs reduce_args(glm_ctx* c, const float* W, const float* b, double* L_rows, double* gb, int64_t ntile) {
    const Problem& P = c->pb;
    ReduceArgs A;
    A.n = P.n;
    A.ntile = ntile;
    A.dt = P.dt_int;
    A.W = W;
    A.b = b;
    A.C = c->buf.C;
    A.part_s = c->buf.part_s;
    A.qd = c->buf.qd;
    A.part_e = c->buf.part_e;
    A.planes = P.ct ? CT_PARTS : 1;
    A.r0 = c->row_r0;
    A.r1 = c->row_r1 < 0 ? P.n : c->row_r1;
    A.spk_from_c = P.prec == GLM_PREC_F32 && !P.ct;
    A.part_self = P.self_shift > 0 ? c->buf.part_self : nullptr;
    A.gself = c->buf.gself;
    A.L_rows = L_rows;
    A.gb = gb;
    A.out = nullptr;
    A.flags = c->buf.flags;
    A.row_blocks = 0;
    return A;
}

cudaError_t launch_reduce(glm_ctx* c, const float* W, const float* b, double* L_rows, double* G, double* gb,
                          bool want_grad, int64_t ntile, int nsplit, const double* Gacc, bool want_total) {
    const Problem& P = c->pb;
    ReduceArgs A = reduce_args(c, W, b, L_rows, gb, ntile);
    A.out = want_total ? c->out_dev : nullptr;
    // Not under programmatic dependence: scheduled while the product before still holds every SM, the many small blocks
    // end up unevenly spread (n = 203: 43 us against 31)
    const bool grad = want_grad && G;
    cudaError_t e = cudaSuccess;
    if (!grad || A.part_self) {
        A.row_blocks = (unsigned)(P.n + 7) / 8;
        e = launch_pdl(c, false, reduce_rows_kernel, A.row_blocks, 256, 0, A);
        if (e != cudaSuccess || !grad) return e;
        A.row_blocks = 0;
    }
    constexpr int M = SUM_GROUPS;
    const bool many = !Gacc && many_groups(c, nsplit);
    const int threads = many ? SUM_E<M> * M : SUM_E<1>;
    if (!A.part_self) A.row_blocks = (unsigned)((P.n + threads / 32 - 1) / (threads / 32));
    auto launch = [&](auto* kernel, unsigned blocks) {
        return launch_pdl(c, false, kernel, A.row_blocks + blocks, threads, 0, A, nsplit, c->buf.part_g, Gacc, G);
    };
    if (many) return launch(reduce_eval_kernel<M, false>, sum_blocks<M>(P.n));
    if (!Gacc && deep_loads(nsplit)) return launch(reduce_eval_kernel<1, true>, sum_blocks<1>(P.n));
    return launch(reduce_eval_kernel<1, false>, sum_blocks<1>(P.n));
}

}  // namespace glm
