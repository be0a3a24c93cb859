// The plain FP32 form of the two contractions (CUDA cores, no tensor cores):
//   step a3/a4:  U = b 1^T + W X (Eq. 3) with the link applied in the epilogue (Eq. 5):
//                E[i][t] = dt exp(U_i[t]) stored FP32, per (bin tile, row) FP64 sums of exp(U).  The
//                spike-time term of Eq. 7 is not taken from this U: the FP32 form forms it in the row
//                reduction as q_i b_i + sum_j W_ij C_ij from the FP64 spike term C, because the rounding of
//                U's FP32 accumulation, summed over the spike bins, alone comes to ~1e-9 of L
//   step a5:     P_s = E X^T over a split s of the bins (FP32, two-level accumulation)
// 128 x 128 output tiles, 256 threads, 8 x 8 outputs per thread, operands staged in shared memory.
#include <cmath>

#include "expm1_acc.cuh"
#include "glm_internal.h"

namespace glm {

constexpr int SB = 128;   // tile edge
constexpr int SK = 16;    // k step
constexpr int ST = 256;   // threads
constexpr int G_INNER = 1024;  // bins accumulated in the inner FP32 sum of the gradient product
// row stride (floats) of the operand tiles in shared memory: 16-byte aligned rows, and the transposing
// stores of four k-rows by one warp fall into two banks per address group instead of four
constexpr int SBP = SB + 4;

int simt_tile_t() { return SB; }

struct SimtUArgs {
    int32_t n;
    int64_t T, Tpad;
    double dt;
    const float* Wt;  // [n][ldw]  the evaluated rows of W, packed and transposed (simt_prep_kernel)
    int64_t ldw;      // their count (its upper bound) rounded up to 4
    const float* b;   // [n]
    const double* eb; // [n]  exp(b_i) in FP64
    const float* X;   // [n][Tpad]
    float* E;         // [n][Tpad]
    double* part_e;   // [n][ntile]
    int64_t ntile;    // bin tiles, Tpad / 128
    int* flags;
    const int32_t* rows;  // evaluated rows (null: all n); tile row l is row rows[l] for l < m
    int32_t m;
    const int32_t* m_dev; // their count on the device (m: its upper bound), or null
};

__device__ __forceinline__ int32_t row_of(const SimtUArgs& A, int32_t m, int32_t l) {
    return l < m ? (A.rows ? A.rows[l] : l) : A.n;
}

// 16-byte asynchronous copy global -> shared (cp.async, both addresses 16-byte aligned), through L2 only; pred false
// fills zeros and reads nothing
__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool pred) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(sa), "l"(src), "r"(pred ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }

template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// One tile of U: RT of the evaluated rows (i0..) x 128 bins (t0..).  A = W (row-major, K contiguous), B = X (K x N, N
// contiguous).  Thread (ty, tx) owns R = RT / 16 rows and the columns tx*4.. and 64+tx*4..; a warp spans 4 ty x 8 tx, so
// each of its 16-byte operand loads per k covers 64 or 128 contiguous bytes: one wavefront.
//
// Two-level accumulation: a single running FP32 sum over ~1000 sources drops the many small terms (sources whose
// filtered train has decayed) below half an ulp of the total, and since most inputs are excitatory those losses have
// one sign: at N = 1000 the mean of U came out ~2e-8 low, ~1.4e-8 of L.  The products of U_FLUSH k-steps (32
// sources) go into a register tile sum, which is added to the thread's column of totals in shared memory.  With both
// levels in registers the kernel needed over 200 registers and ran one block (eight warps) per SM; with the totals in
// shared memory two blocks fit, and their sixteen warps hide the shared-memory latency of the inner loop.  The
// epilogue runs as a rolled loop over rows staged in shared memory: fully unrolled, the k-tile body and the 64 inlined
// exponentials of the epilogue outgrew the instruction cache.
//
// A row tile of at most 64 or 32 rows (a small n, the last tile, a line search with few open rows) is cut to that
// height, with two more k-steps in flight: n = 50, 20 000 bins 14 us a launch in a fit's line searches, against 45 us.
constexpr int EPI_LD = SB + 4;  // row stride of the epilogue staging (floats): 16-byte rows, fewer bank conflicts
constexpr int U_FLUSH = 2;      // k-steps per register tile sum
template <int RT>
struct UTile {
    static constexpr int R = RT / 16;
    static constexpr int LDA = RT + 4;
    static constexpr int NST = RT == 128 ? 2 : 4;             // k-steps of operands in shared memory
    static constexpr int OPER = NST * SK * (LDA + SBP);       // floats
    static constexpr int STAGED = RT < 64 ? RT : 64;          // rows of U staged at a time by the epilogue
    static constexpr int FLOATS = (OPER > STAGED * EPI_LD ? OPER : STAGED * EPI_LD) + R * 8 * ST;
};
constexpr size_t U_SMEM = (size_t)(UTile<128>::FLOATS > UTile<64>::FLOATS ? UTile<128>::FLOATS : UTile<64>::FLOATS) * sizeof(float);
static_assert(UTile<32>::FLOATS <= UTile<64>::FLOATS, "U_SMEM covers every tile height");

template <int RT>
__device__ __forceinline__ void simt_u_tile(const SimtUArgs& A, float* sm, int32_t m, int32_t i0, int64_t bt) {
    using T = UTile<RT>;
    constexpr int R = T::R, NST = T::NST;
    // operands: As[NST][SK][LDA] then Bs[NST][SK][SBP] (after the k loop the same memory stages rows of U); then the
    // totals, float4 [R * 2][ST]: columns tx*4.. and 64+tx*4.. of the thread's row r at [2 r][tid] and [2 r + 1][tid]
    float* As = sm;
    float* Bs = sm + NST * SK * T::LDA;
    float4* tot = reinterpret_cast<float4*>(sm + T::FLOATS - R * 8 * ST);
    const int tid = threadIdx.x;
    const int tx = ((tid >> 5) & 1) * 8 + (tid & 7), ty = (tid >> 6) * 4 + ((tid >> 3) & 3);
    const int64_t t0 = bt * SB;
    const int32_t n = A.n;
    // first row of the thread's group of four (RT = 32: two) rows
    auto row_at = [&](int r) { return RT == 128 ? (r < 4 ? ty * 4 + r : 64 + ty * 4 + (r - 4)) : ty * R + r; };
    // operand tiles by 16-byte asynchronous copies issued NST - 1 k-steps ahead (no staging registers); zeros past n
    // and past the evaluated rows.  W comes transposed: copied from its rows 4 bytes at a time, it took more of the L1
    // data path than X: n = 300, 60k bins 445 -> 406 us, n = 1000, 200k 10.4 -> 9.5 ms (9.3 with vector totals)
    constexpr int AQ = RT / 4;                           // 16-byte words of W per k
    const int b_row = tid >> 5, b_col = (tid & 31) * 4;  // k rows b_row and b_row + 8, bins b_col..+3
    auto load = [&](int kt) {
        const int k0 = kt * SK;
        float* as = As + (kt % NST) * SK * T::LDA;
        float* bs = Bs + (kt % NST) * SK * SBP;
#pragma unroll
        for (int x = tid; x < SK * AQ; x += ST) {
            const int32_t k = k0 + x / AQ, l = i0 + 4 * (x % AQ);
            const bool ok = k < n && l < m;
            cp_async16(as + (x / AQ) * T::LDA + 4 * (x % AQ), A.Wt + (ok ? k * A.ldw + l : 0), ok);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int32_t kb = k0 + b_row + 8 * h;
            cp_async16(bs + (b_row + 8 * h) * SBP + b_col, A.X + (kb < n ? (int64_t)kb * A.Tpad + t0 + b_col : 0), kb < n);
        }
    };
    const int nk = (n + SK - 1) / SK;
#pragma unroll
    for (int s = 0; s < NST - 1; ++s) {
        if (s < nk) load(s);
        cp_async_commit();
    }
    // what the epilogue needs of its rows, while the operands come: lane l holds the warp's row l (warp + 8 l of the
    // tile).  Read row by row in the epilogue, each waited for two loads in a chain
    const int warp = tid >> 5, lane = tid & 31;
    static_assert(ST / 32 == 8 && RT / 8 <= 32, "rows of a warp");
    int32_t my_row = 0;
    double my_eb = 0.0;
    float my_sh = 0.f;
    if (lane < RT / 8 && i0 + warp + 8 * lane < m) {
        my_row = row_of(A, m, i0 + warp + 8 * lane);
        my_eb = A.eb[my_row];
        my_sh = fminf(A.b[my_row] - EXP_SPLIT_FLOOR, 0.f);  // U - c = v + sh
    }
    const float my_dteb = (float)(A.dt * my_eb);
#pragma unroll
    for (int e = 0; e < R * 2; ++e) tot[e * ST + tid] = make_float4(0.f, 0.f, 0.f, 0.f);
    float tl[R][8];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < 8; ++c) tl[r][c] = 0.f;
    for (int kt = 0; kt < nk; ++kt) {
        cp_async_wait<NST - 2>();  // this k-step's tiles have landed
        __syncthreads();           // ... for every thread, and every thread is done with the buffer loaded next
        if (kt + NST - 1 < nk) load(kt + NST - 1);
        cp_async_commit();
        const float* as = As + (kt % NST) * SK * T::LDA;
        const float* bs = Bs + (kt % NST) * SK * SBP;
#pragma unroll 4
        for (int k = 0; k < SK; ++k) {
            float av[R];
            if constexpr (RT == 128) {
                const float4 a0 = *reinterpret_cast<const float4*>(as + k * T::LDA + ty * 4);
                const float4 a1 = *reinterpret_cast<const float4*>(as + k * T::LDA + 64 + ty * 4);
                av[0] = a0.x, av[1] = a0.y, av[2] = a0.z, av[3] = a0.w;
                av[4] = a1.x, av[5] = a1.y, av[6] = a1.z, av[7] = a1.w;
            } else if constexpr (RT == 64) {
                const float4 a0 = *reinterpret_cast<const float4*>(as + k * T::LDA + ty * 4);
                av[0] = a0.x, av[1] = a0.y, av[2] = a0.z, av[3] = a0.w;
            } else {
                const float2 a0 = *reinterpret_cast<const float2*>(as + k * T::LDA + ty * 2);
                av[0] = a0.x, av[1] = a0.y;
            }
            const float4 b0 = *reinterpret_cast<const float4*>(bs + k * SBP + tx * 4);
            const float4 b1 = *reinterpret_cast<const float4*>(bs + k * SBP + 64 + tx * 4);
            const float bv[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int c = 0; c < 8; ++c) tl[r][c] = fmaf(av[r], bv[c], tl[r][c]);
        }
        if ((kt + 1) % U_FLUSH == 0 || kt + 1 == nk) {
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float4 v = tot[(2 * r + h) * ST + tid];
                    v.x += tl[r][4 * h];
                    v.y += tl[r][4 * h + 1];
                    v.z += tl[r][4 * h + 2];
                    v.w += tl[r][4 * h + 3];
                    tot[(2 * r + h) * ST + tid] = v;
                    tl[r][4 * h] = tl[r][4 * h + 1] = tl[r][4 * h + 2] = tl[r][4 * h + 3] = 0.f;
                }
        }
    }
    __syncthreads();  // the operands are read: their memory is free
    // epilogue.  With v = (W X)_i[t]:  e^{U} = e^{b_i} (1 + expm1(v)).  e^{b_i} comes in FP64 and the
    // integer count of bins is kept apart from the FP32 sum of expm1(v), so the part of the integral that
    // repeats over quiet bins (U ~ b_i) carries no FP32 rounding of exp or of b + v; expm1 is correctly
    // rounded (expm1_acc.cuh), so its rounding carries no bias into the sum either.
    // E = dt e (0 beyond T) in FP32; FP64 row sums of e per tile.  STAGED rows at a time: the threads stage their v,
    // then the warps take rows in turn, a lane 4 consecutive bins of a row; rows past the evaluated ones are skipped.
    bool bad = false;
#pragma unroll
    for (int half = 0; half < RT / T::STAGED; ++half) {
        constexpr int RH = R / (RT / T::STAGED);  // the thread's rows in this half
        // the barrier before (or the previous half's) has passed: the staging memory is free
#pragma unroll
        for (int rr = 0; rr < RH; ++rr) {
            float* dst = sm + (row_at(half * RH + rr) - half * T::STAGED) * EPI_LD;
            *reinterpret_cast<float4*>(dst + tx * 4) = tot[2 * (half * RH + rr) * ST + tid];
            *reinterpret_cast<float4*>(dst + 64 + tx * 4) = tot[(2 * (half * RH + rr) + 1) * ST + tid];
        }
        __syncthreads();
        // The warp takes rows warp, warp + 8, ...: up to NR.  The FP64 sums over the lanes go through one butterfly for all
        // of them, each exchange halving the rows a lane carries: 9 FP64 adds for 8 rows instead of 40 (they are
        // scarce: about 64 clocks per warp), every row's tree of additions as before.
        constexpr int NR = T::STAGED / (ST / 32);
        double rs[NR];
#pragma unroll
        for (int q = 0; q < NR; ++q) rs[q] = 0.0;
        const int32_t rows_here = min(T::STAGED, m - i0 - half * T::STAGED);  // the evaluated rows come first
#pragma unroll 1
        for (int q = 0; q < NR && warp + q * (ST / 32) < rows_here; ++q) {
            const int lr = warp + q * (ST / 32);
            const int from = half * NR + q;  // the lane with the row's constants
            const int32_t i = __shfl_sync(0xffffffffu, my_row, from);
            const double ebi = __shfl_sync(0xffffffffu, my_eb, from);
            const float sh = __shfl_sync(0xffffffffu, my_sh, from), dteb = __shfl_sync(0xffffffffu, my_dteb, from);
            const float4 v = *reinterpret_cast<const float4*>(sm + lr * EPI_LD + lane * 4);
            const float vv[4] = {v.x, v.y, v.z, v.w};
            float ev[4];
            float msum = 0.f;
            int cnt = 0;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int64_t t = t0 + lane * 4 + c;
                const float mm = expm1_acc(vv[c] + sh);
                const bool valid = t < A.T;
                bad |= valid && !(mm <= 3.0e38f);
                if (valid) {
                    msum += mm;
                    ++cnt;
                }
                ev[c] = valid ? fmaf(dteb, mm, dteb) : 0.f;
            }
            *reinterpret_cast<float4*>(A.E + (int64_t)i * A.Tpad + t0 + lane * 4) = make_float4(ev[0], ev[1], ev[2], ev[3]);
            const double rv = ebi * ((cnt == 4 ? 4.0 : (double)cnt) + (double)msum);
#pragma unroll
            for (int x = 0; x < NR; ++x) rs[x] = x == q ? rv : rs[x];
        }
        // after the exchange at distance `off`, lanes with that bit hold the upper half of the rows
        int row_q = 0;
#pragma unroll
        for (int off = 16, live = NR; off >= 1; off >>= 1) {
            if (live > 1) {
                live >>= 1;
                const bool up = lane & off;
                row_q = 2 * row_q + (up ? 1 : 0);
#pragma unroll
                for (int x = 0; x < NR / 2; ++x) {
                    if (x >= live) break;
                    const double keep = up ? rs[x + live] : rs[x], give = up ? rs[x] : rs[x + live];
                    rs[x] = keep + __shfl_xor_sync(0xffffffffu, give, off);
                }
            } else {
                rs[0] += __shfl_xor_sync(0xffffffffu, rs[0], off);
            }
        }
        constexpr int OWN = 32 / NR;  // lanes that end with the same row
        const int lr = warp + row_q * (ST / 32);
        const int32_t i = __shfl_sync(0xffffffffu, my_row, half * NR + row_q);
        if (lane % OWN == 0 && lr < rows_here) A.part_e[(int64_t)i * A.ntile + bt] = rs[0];
        __syncthreads();
    }
    if (bad) atomicOr(A.flags, 1);
}

// H: rows per block, 128 (cut to 64 or 32 where there are no more) or 32.
// Blocks run row tile fastest (block id = bin tile * mt + row tile): the row tiles of one bin tile read the same X
// tile while it is in L2.  H = 32: three blocks fit an SM's shared memory; the bound of four was measured with, and
// keeps the kernel at 64 registers.
template <int H>
__global__ void __launch_bounds__(ST, H == 128 ? 2 : 4) simt_u_kernel(const __grid_constant__ SimtUArgs A) {
    pdl_wait();
    extern __shared__ __align__(16) float sm[];
    const int32_t m = A.m_dev ? __ldcg(A.m_dev) : A.m;
    const int32_t mt = (m + H - 1) / H;
    if ((int64_t)blockIdx.x >= mt * A.ntile) return;
    const int32_t i0 = (int32_t)(blockIdx.x % mt) * H, left = m - i0;
    const int64_t bt = (int64_t)(blockIdx.x / mt);
    pdl_trigger();
    if constexpr (H == 32) {
        simt_u_tile<32>(A, sm, m, i0, bt);
    } else {
        if (left > 64) simt_u_tile<128>(A, sm, m, i0, bt);
        else if (left > 32) simt_u_tile<64>(A, sm, m, i0, bt);
        else simt_u_tile<32>(A, sm, m, i0, bt);
    }
}

struct SimtGArgs {
    int32_t n;
    int64_t Tpad;
    int64_t k_per_split;
    const float* E;   // [n][Tpad]
    const float* X;   // [n][Tpad]
    float* part_g;    // [nsplit][part_plane(n)]
};

// part_g[s][i][j] = sum over bins of split s of E[i][t] X[j][t].  Both operands are K contiguous and stay so in shared
// memory, [row][SK + 4]: 16-byte asynchronous copies in, 16-byte loads of four k's of a row out (a thread's rows are 16
// apart, so the rows that a warp reads together are neighbours and fall into different banks).  Copied in 4 bytes at a
// time and transposed, the operands took a third of the L1 data path beside the loads that bound this kernel: n = 300,
// 60 000 bins 470 -> 431 us, n = 1000, 200 000 bins 10.8 -> 9.9 ms.  The outer level of the two-level sum (every
// G_INNER bins) lives in shared memory, one column per thread: with it in registers the kernel ran one block per SM,
// whose eight warps could not hide the shared-memory latency of the inner loop; without, two blocks fit.
constexpr int G_LD = SK + 4;
constexpr size_t G_SMEM = (size_t)(2 * 2 * SB * G_LD + 64 * ST) * sizeof(float);
__global__ void __launch_bounds__(ST, 2) simt_grad_kernel(const __grid_constant__ SimtGArgs A) {
    pdl_wait();
    extern __shared__ __align__(16) float gsm[];
    float* As = gsm;                    // [2][SB][G_LD]
    float* Bs = gsm + 2 * SB * G_LD;    // [2][SB][G_LD]
    float* tot = gsm + 4 * SB * G_LD;   // [64][ST]: element r * 8 + c of thread tid at [(r * 8 + c) * ST + tid]
    const int tid = threadIdx.x;
    // thread (ty, tx) owns rows ty + 16 r and columns tx + 16 c; a warp spans 4 ty x 8 tx
    const int tx = ((tid >> 5) & 1) * 8 + (tid & 7), ty = (tid >> 6) * 4 + ((tid >> 3) & 3);
    const int32_t i0 = blockIdx.y * SB, j0 = blockIdx.x * SB;
    const int64_t kb = (int64_t)blockIdx.z * A.k_per_split;
    const int64_t ke = min(kb + A.k_per_split, A.Tpad);
    const int32_t n = A.n;
    float acc[8][8];
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            acc[r][c] = 0.f;
            tot[(r * 8 + c) * ST + tid] = 0.f;
        }
    const int l_row = tid >> 2, l_col = (tid & 3) * 4;  // rows l_row, l_row + 64; k l_col..+3
    const float* src[2][2];
    bool in[2][2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int32_t i = i0 + l_row + 64 * h, j = j0 + l_row + 64 * h;
        in[0][h] = i < n;
        in[1][h] = j < n;
        src[0][h] = A.E + (int64_t)(i < n ? i : 0) * A.Tpad + l_col;
        src[1][h] = A.X + (int64_t)(j < n ? j : 0) * A.Tpad + l_col;
    }
    auto load = [&](int64_t k0, int buf) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            cp_async16(As + (buf * SB + l_row + 64 * h) * G_LD + l_col, src[0][h] + k0, in[0][h]);
            cp_async16(Bs + (buf * SB + l_row + 64 * h) * G_LD + l_col, src[1][h] + k0, in[1][h]);
        }
        cp_async_commit();
    };
    if (kb < ke) load(kb, 0);
    int64_t since = 0;
    for (int64_t k0 = kb; k0 < ke; k0 += SK) {
        const int cur = (int)(((k0 - kb) / SK) & 1);
        cp_async_wait<0>();
        __syncthreads();  // this k-step's tiles are here, and every thread is done with the buffer loaded next
        if (k0 + SK < ke) load(k0 + SK, cur ^ 1);
        const float* as = As + (cur * SB + ty) * G_LD;
        const float* bs = Bs + (cur * SB + tx) * G_LD;
#pragma unroll 1
        for (int k = 0; k < SK; k += 4) {
            float4 bv[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) bv[c] = *reinterpret_cast<const float4*>(bs + 16 * c * G_LD + k);
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const float4 a = *reinterpret_cast<const float4*>(as + 16 * r * G_LD + k);
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    acc[r][c] = fmaf(a.w, bv[c].w, fmaf(a.z, bv[c].z, fmaf(a.y, bv[c].y, fmaf(a.x, bv[c].x, acc[r][c]))));
            }
        }
        since += SK;
        if (since == G_INNER) {
#pragma unroll
            for (int r = 0; r < 8; ++r)
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    tot[(r * 8 + c) * ST + tid] += acc[r][c];
                    acc[r][c] = 0.f;
                }
            since = 0;
        }
    }
    float* plane = A.part_g + (int64_t)blockIdx.z * part_plane(n);
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const int32_t i = i0 + ty + 16 * r;
        if (i >= n) continue;
        const int32_t rh = min(n - (i & ~31), 32);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const int32_t j = j0 + tx + 16 * c;
            if (j < n) plane[part_group(n, i / 32, j / 4, rh) + (i % 32) * 4 + j % 4] = tot[(r * 8 + c) * ST + tid] + acc[r][c];
        }
    }
}

// The same sums over 32 x 32 tiles, R x C outputs to a thread, for a small n, where 128 x 128 tiles leave most of the chip
// idle (n = 50, 20 000 bins: 20 blocks, one k-step of loads in flight each).  Every output adds up its bins in the same
// order, 1024 of them in one chain, so what counts is how many chains an SM works on.  Up to two blocks per SM,
// 2 x 2 outputs (eight warps a block): the whole evaluation at n = 50, 20 000 bins 105 -> 78 us, n = 96 127 -> 111, n = 60,
// 60 000 bins 129 -> 112.  Beyond, their operand loads (twice as many per FMA) are the limit and 4 x 4 outputs are faster:
// n = 128, 20 000 bins 139 us against 162, n = 60, 200 000 bins 205 against 240.  4 x 2 and 2 x 4 were slower than both.
constexpr int GS_K = 32, GS_ST = 4, GS_LD = GS_K + 4;
template <int R, int C>
constexpr int GS_T = 32 / R * (32 / C);
template <int R, int C>
__global__ void __launch_bounds__(GS_T<R, C>) simt_grad_small_kernel(const __grid_constant__ SimtGArgs A) {
    pdl_wait();
    __shared__ __align__(16) float As[GS_ST][32][GS_LD], Bs[GS_ST][32][GS_LD];
    constexpr int TX = 32 / C, TY = 32 / R;
    const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;  // rows ty + TY r, columns tx + TX c
    const int32_t i0 = blockIdx.y * 32, j0 = blockIdx.x * 32, n = A.n;
    const int64_t kb = (int64_t)blockIdx.z * A.k_per_split;
    const int64_t ke = min(kb + A.k_per_split, A.Tpad);
    const int nk = (int)((ke - kb) / GS_K);  // Tpad and k_per_split are multiples of 256
    auto load = [&](int kt) {
        const int s = kt % GS_ST;
#pragma unroll
        for (int x = tid; x < 256; x += GS_T<R, C>) {  // eight 16-byte words a row
            const int row = x >> 3, col = 4 * (x & 7);
            const bool vi = i0 + row < n, vj = j0 + row < n;
            const int64_t k = kb + (int64_t)kt * GS_K + col;
            cp_async16(&As[s][row][col], A.E + (int64_t)(vi ? i0 + row : 0) * A.Tpad + k, vi);
            cp_async16(&Bs[s][row][col], A.X + (int64_t)(vj ? j0 + row : 0) * A.Tpad + k, vj);
        }
    };
    float acc[R][C], tot[R][C];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < C; ++c) acc[r][c] = tot[r][c] = 0.f;
#pragma unroll
    for (int s = 0; s < GS_ST - 1; ++s) {
        if (s < nk) load(s);
        cp_async_commit();
    }
    auto flush = [&]() {
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int c = 0; c < C; ++c) {
                tot[r][c] += acc[r][c];
                acc[r][c] = 0.f;
            }
    };
    for (int kt = 0; kt < nk; ++kt) {
        cp_async_wait<GS_ST - 2>();
        __syncthreads();
        if (kt + GS_ST - 1 < nk) load(kt + GS_ST - 1);
        cp_async_commit();
        const int s = kt % GS_ST;
#pragma unroll
        for (int k = 0; k < GS_K; k += 4) {
            float4 av[R], bv[C];
#pragma unroll
            for (int r = 0; r < R; ++r) av[r] = *reinterpret_cast<const float4*>(&As[s][ty + TY * r][k]);
#pragma unroll
            for (int c = 0; c < C; ++c) bv[c] = *reinterpret_cast<const float4*>(&Bs[s][tx + TX * c][k]);
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int c = 0; c < C; ++c)
                    acc[r][c] = fmaf(av[r].w, bv[c].w, fmaf(av[r].z, bv[c].z, fmaf(av[r].y, bv[c].y, fmaf(av[r].x, bv[c].x, acc[r][c]))));
        }
        if ((kt + 1) % (G_INNER / GS_K) == 0) flush();
    }
    flush();
    float* plane = A.part_g + (int64_t)blockIdx.z * part_plane(n);
    const int32_t rh = min(n - i0, 32);
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int32_t ir = ty + TY * r, j = j0 + tx + TX * c;
            if (i0 + ir < n && j < n) plane[part_group(n, i0 / 32, j / 4, rh) + ir * 4 + j % 4] = tot[r][c];
        }
}

// bins per split: a multiple of G_INNER, from the splits that give about four 128 x 128 tiles per SM
static int64_t grad_split_bins(const glm_ctx* c) {
    const int64_t tiles = (int64_t)((c->pb.n + SB - 1) / SB) * ((c->pb.n + SB - 1) / SB);
    int64_t s = (4 * (int64_t)c->sm_count + tiles - 1) / tiles;
    const int64_t kmax = c->pb.Tpad / SK;
    if (s > kmax) s = kmax;
    if (s < 1) s = 1;
    if (s > 256) s = 256;
    auto bins = [&](int64_t splits) {
        const int64_t kps = (c->pb.Tpad + splits - 1) / splits;
        return (kps + G_INNER - 1) / G_INNER * G_INNER;
    };
    const int64_t kps = bins(s), planes = c->buf.part_planes;
    return planes > 0 && (c->pb.Tpad + kps - 1) / kps > planes ? bins(planes) : kps;
}
int grad_nsplit(const glm_ctx* c) {
    const int64_t kps = grad_split_bins(c);
    return (int)((c->pb.Tpad + kps - 1) / kps);
}

// What the U product needs of (W, b): the evaluated rows of W, packed and transposed, Wt[k][l] = W[rows[l]][k] (zeros
// up to ldw), by 32 x 32 tiles, and in the blocks after those e^c, c = max(b_i, floor), in FP64 (b_i of every row).
__global__ void __launch_bounds__(256) simt_prep_kernel(int32_t n, int32_t m, int64_t ldw, const float* __restrict__ W,
                                                        const float* __restrict__ b, const int32_t* __restrict__ rows,
                                                        float* __restrict__ Wt, double* __restrict__ eb, int* flags) {
    __shared__ float tile[32][33];
    pdl_trigger();
    const int32_t kt = (n + 31) / 32, lt = (m + 31) / 32, x = threadIdx.x & 31, y = threadIdx.x >> 5;
    if ((int32_t)blockIdx.x < kt * lt) {
        const int32_t k0 = blockIdx.x % kt * 32, l0 = blockIdx.x / kt * 32;
        for (int q = y; q < 32; q += 8) {
            const int32_t l = l0 + q;
            tile[q][x] = (l < m && k0 + x < n) ? W[(int64_t)(rows ? rows[l] : l) * n + k0 + x] : 0.f;
        }
        __syncthreads();
        for (int q = y; q < 32; q += 8)
            if (k0 + q < n && l0 + x < ldw) Wt[(k0 + q) * ldw + l0 + x] = tile[x][q];
        return;
    }
    const int32_t i = ((int32_t)blockIdx.x - kt * lt) * 256 + threadIdx.x;
    if (i >= n) return;
    const double v = exp((double)fmaxf(b[i], EXP_SPLIT_FLOOR));
    if (!isfinite(b[i]) || !(v <= 1e300)) atomicOr(flags, 1);
    eb[i] = v;
}

// The transposed rows lie in part_g: free while a U product runs, and never smaller (a plane of partials holds n rows of
// n rounded up to 4).
float* simt_wt(const glm_ctx* c) { return c->buf.part_g; }
int64_t simt_ldw(int32_t m) { return (m + 3) & ~(int64_t)3; }

cudaError_t launch_simt_u_epilogue(glm_ctx* c, const float* W, const float* b, const int32_t* rows, int32_t m,
                                   const int32_t* m_dev) {
    const Problem& P = c->pb;
    const int32_t mr = rows ? m : P.n;
    if (!m_dev) {
        const unsigned blocks = (unsigned)((P.n + 31) / 32 * ((mr + 31) / 32) + (P.n + 255) / 256);
        simt_prep_kernel<<<blocks, 256, 0, c->stream>>>(P.n, mr, simt_ldw(mr), W, b, rows, simt_wt(c), c->buf.eb, c->buf.flags);
    }
    SimtUArgs A;
    A.n = P.n;
    A.T = P.T;
    A.Tpad = P.Tpad;
    A.dt = P.dt;
    A.Wt = simt_wt(c);
    A.ldw = simt_ldw(mr);
    A.b = b;
    A.eb = c->buf.eb;
    A.X = reinterpret_cast<const float*>(c->buf.X);
    A.E = reinterpret_cast<float*>(c->buf.E);
    A.part_e = c->buf.part_e;
    A.ntile = P.Tpad / SB;
    A.flags = c->buf.flags;
    A.rows = rows;
    A.m = mr;
    A.m_dev = m_dev;
    // one block per (row tile, bin tile), row tiles fastest
    const int64_t blocks = (int64_t)((A.m + SB - 1) / SB) * A.ntile;
    // one wave of blocks or less: tiles of 32 rows, up to four times the blocks at three per SM (58 KB of shared memory
    // each; the whole evaluation at n = 96, 20 000 bins 111 -> 101 us, though its 474 blocks are 18 more than one wave,
    // n = 128 140 -> 132; the same at n = 50, where the tile is 64 rows high); with more, the higher tiles' fewer operand
    // loads per FMA win
    if (blocks <= 2 * (int64_t)c->sm_count) {
        constexpr size_t smem = (size_t)UTile<32>::FLOATS * sizeof(float);
        const cudaError_t e = cudaFuncSetAttribute(simt_u_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        return launch_pdl(c, true, simt_u_kernel<32>, (unsigned)((A.m + 31) / 32 * A.ntile), ST, smem, A);
    }
    const cudaError_t e = cudaFuncSetAttribute(simt_u_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)U_SMEM);
    if (e != cudaSuccess) return e;
    return launch_pdl(c, true, simt_u_kernel<128>, (unsigned)blocks, ST, U_SMEM, A);
}

cudaError_t launch_simt_grad(glm_ctx* c) {
    const Problem& P = c->pb;
    const int ns = grad_nsplit(c);
    SimtGArgs A;
    A.n = P.n;
    A.Tpad = P.Tpad;
    A.k_per_split = grad_split_bins(c);
    A.E = reinterpret_cast<const float*>(c->buf.E);
    A.X = reinterpret_cast<const float*>(c->buf.X);
    A.part_g = c->buf.part_g;
    const unsigned st = (unsigned)(P.n + 31) / 32;
    const int64_t blocks = (int64_t)st * st * ns;
    if (blocks <= 2 * (int64_t)c->sm_count)
        return launch_pdl(c, true, simt_grad_small_kernel<2, 2>, dim3(st, st, ns), dim3(GS_T<2, 2>), 0, A);
    if (blocks <= 6 * (int64_t)c->sm_count)
        return launch_pdl(c, true, simt_grad_small_kernel<4, 4>, dim3(st, st, ns), dim3(GS_T<4, 4>), 0, A);
    dim3 grid((P.n + SB - 1) / SB, (P.n + SB - 1) / SB, ns);
    const cudaError_t e = cudaFuncSetAttribute(simt_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G_SMEM);
    if (e != cudaSuccess) return e;
    return launch_pdl(c, true, simt_grad_kernel, grid, ST, G_SMEM, A);
}

}  // namespace glm

// The FP32 form's e^v - 1 (expm1_acc.cuh), evaluated on the host by the same code as the epilogue's.
extern "C" int glm_expm1(const float* v_host, int64_t n, float* out_host) {
    if (n < 0 || (n > 0 && (!v_host || !out_host))) return GLM_ERR_INVALID_ARG;
    for (int64_t k = 0; k < n; ++k) out_host[k] = glm::expm1_acc(v_host[k]);
    return GLM_OK;
}
