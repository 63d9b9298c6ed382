// Rayleigh-Ritz (LABPSD step 9, remark 6) over the whole GPU, for reduced problems of some dozens of
// columns and more: the same method as the one-cluster kernel of rr.cu, with every step that is bound by
// FP64 throughput (2 lanes per clock per SM) spread over all SMs and only the tridiagonalisation, whose two
// barriers per column need the latency of a cluster, on 16.
//
//   1. A = D S_R D, D = diag(S_R)^{-1/2}; blocked Cholesky A = L L^T, 32 columns at a time: k_rg_panel (every
//      CTA factors the diagonal block for itself, then its rows), k_rg_syrk.
//      A pivot below RG_PIVOT_MIN (or NaN) sets info[3]: the later kernels return at once and the host runs
//      the single-CTA kernel with the rank-revealing branch.
//   2. C = L^{-1} (D H_R D) L^{-T}: two blocked forward substitutions, one warp per column (k_rg_fwd); the
//      second stops at the diagonal (C is symmetric).
//   3. Householder tridiagonalisation of C on a cluster (k_rg_tridiag): rows dealt out cyclically, so that
//      every CTA keeps its share of the shrinking matrix; reflectors to global memory, no Q.
//   4. FP32 Sturm multisection (k_rg_bisect) and FP64 inverse iteration (k_rg_invit), one warp per pair.
//   5. CholeskyQR of the vectors with the kernels of 1 and 2, a second pass when they were far from
//      orthonormal; Rayleigh quotients.
//   6. W = D L^{-T} H_0 H_1 ... z, one CTA per vector (k_rg_back).
//
// One call, one cluster for everything before: q = 149, k = 85: 1.43 ms (2.46), of which tridiagonalisation 0.58,
// inverse iteration 0.15, Cholesky panels 0.19; q = 538, k = 282: 8.0 ms (44.7), of which tridiagonalisation 4.8,
// inverse iteration 0.77, panels 0.62, substitutions 0.6, back-transformation 0.48.
#include <cooperative_groups.h>

#include <cfloat>
#include <cmath>
#include <mutex>

#include "common.h"
#include "rr_math.h"

namespace cg = cooperative_groups;

namespace hbsd {
namespace {

using namespace rrm;

constexpr int RG_NB = 32;
constexpr double RG_PIVOT_MIN = 1e-14;
constexpr double RG_SECOND_PASS = 1e-2;   // max |V^T V - I| above which CholeskyQR runs twice
constexpr int RG_CLUSTER = 16;
constexpr int RG_TRI_THREADS = 512;
constexpr size_t RG_SMEM_MAX = 225 * 1024;

// info[3] set: a pivot of S_R failed, nothing below is wanted.  gate (nullable): max |G - I| of the first
// CholeskyQR pass; the kernels of the second return unless it is needed.  Every thread may ask for itself, except in
// k_rg_panel, which sets info[3].
__device__ __forceinline__ bool rg_stop(const int* info, const unsigned long long* gate) {
    if (__ldcg(info + 3)) return true;
    return gate && !(__longlong_as_double((long long)__ldcg(gate)) > RG_SECOND_PASS);
}

// A = D S D (lower and upper), dv = diag(S)^{-1/2}
__global__ void __launch_bounds__(256) k_rg_scale(const double* __restrict__ S, int q, double* __restrict__ A,
                                                  double* __restrict__ dv) {
    __shared__ double di[32], dj[32];
    const int i0 = blockIdx.y * 32, j0 = blockIdx.x * 32;
    if (threadIdx.x < 64) {
        const int r = (threadIdx.x < 32 ? i0 : j0) + (threadIdx.x & 31);
        const double v = r < q ? rsqrt(S[(int64_t)r * q + r]) : 0.0;
        (threadIdx.x < 32 ? di : dj)[threadIdx.x & 31] = v;
        if (threadIdx.x < 32 && blockIdx.x == 0 && r < q) dv[r] = v;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < 1024; t += 256) {
        const int i = i0 + (t >> 5), j = j0 + (t & 31);
        if (i < q && j < q) A[(int64_t)i * q + j] = S[(int64_t)i * q + j] * di[t >> 5] * dj[t & 31];
    }
}

// One panel (columns p0 .. p0 + nb - 1) of A = L L^T (row-major, lower): every CTA factors the diagonal block
// in shared memory, then each warp solves one row below it.  L, its transpose LT and rl = 1 / L_cc.
// clamp: pivots below DBL_MIN are raised to it (CholeskyQR) instead of stopping.
__global__ void __launch_bounds__(256) k_rg_panel(const double* __restrict__ A, int n, int p0, int clamp,
                                                  double* __restrict__ L, double* __restrict__ LT, double* __restrict__ rl,
                                                  int* __restrict__ info, const unsigned long long* gate) {
    __shared__ double D[RG_NB][RG_NB + 1], ri[RG_NB];   // D[j][i]: column j of the block's factor
    __shared__ int s_bad, s_stop;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nb = min(RG_NB, n - p0), p1 = p0 + nb;
    // this warp's row is on its way while the block is factored
    const int row = p1 + (int)blockIdx.x * 8 + warp;
    double a = row < n && lane < nb ? A[(int64_t)row * n + p0 + lane] : 0.0;
    // one reading for the CTA: another CTA of this launch may set info[3] meanwhile, and warps that left would be
    // missed at the barriers below
    if (tid == 0) {
        s_bad = 0;
        s_stop = rg_stop(info, gate);
    }
    __syncthreads();
    if (s_stop) return;
    if (warp < 4) {
        // columns 4 t + warp in this warp's registers, lane = row; columns and rows beyond nb are those of I
        double r[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const int j = 4 * t + warp;
            r[t] = lane < nb && j <= lane ? A[(int64_t)(p0 + lane) * n + p0 + j] : (lane == j ? 1.0 : 0.0);
        }
        // column c scaled by its pivot and published (integer comparisons: an FP64 one takes 170 clocks)
        auto finish = [&](int c, double& rc) {
            double piv = __shfl_sync(0xffffffffu, rc, c);
            const unsigned long long least = (unsigned long long)__double_as_longlong(clamp ? DBL_MIN : RG_PIVOT_MIN);
            const bool ok = (unsigned long long)__double_as_longlong(piv) - least <= 0x7FF0000000000000ull - least;   // least .. inf
            if (!ok) {
                if (clamp) piv = DBL_MIN;
                else s_bad = 1;
            }
            const double inv = rsqrt(piv);
            rc = lane >= c ? (lane == c ? piv : rc) * inv : 0.0;
            D[c][lane] = rc;
            if (lane == 0) ri[c] = inv;
        };
        if (warp == 0) finish(0, r[0]);
#pragma unroll
        for (int c = 0; c < RG_NB; ++c) {
            asm volatile("bar.sync 1, 128;" ::: "memory");
            const double lc = D[c][lane];
            // the owner of column c + 1 updates and publishes it before its other columns
            if (c + 1 < RG_NB && warp == ((c + 1) & 3)) {
                r[(c + 1) >> 2] = fma(-lc, D[c][c + 1], r[(c + 1) >> 2]);
                finish(c + 1, r[(c + 1) >> 2]);
            }
#pragma unroll
            for (int t = c >> 2; t < 8; ++t) {
                const int j = 4 * t + warp;
                if (j > c + 1) r[t] = fma(-lc, D[c][j], r[t]);
            }
        }
    }
    __syncthreads();
    if (s_bad) {   // the same block in every CTA
        if (tid == 0) atomicExch(info + 3, 1);
        return;
    }
    for (int c = 0; c < nb; ++c) {
        const double xc = __shfl_sync(0xffffffffu, a, c) * ri[c];
        if (lane == c) a = xc;
        else if (lane > c) a = fma(-D[c][lane], xc, a);
    }
    if (row < n && lane < nb) {
        L[(int64_t)row * n + p0 + lane] = a;
        LT[(int64_t)(p0 + lane) * n + row] = a;
    }
    if (blockIdx.x == 0) {
        for (int t = tid; t < nb * nb; t += 256) {
            const int i = t / nb, j = t % nb;
            if (j <= i) {
                L[(int64_t)(p0 + i) * n + p0 + j] = D[j][i];
                LT[(int64_t)(p0 + j) * n + p0 + i] = D[j][i];
            }
        }
        if (tid < nb) rl[p0 + tid] = ri[tid];
    }
}

// A(i, j) -= sum_c L(i, c) L(j, c) over the panel's columns, i >= j >= p1; one 16 x 16 tile per CTA
__global__ void __launch_bounds__(256) k_rg_syrk(double* __restrict__ A, const double* __restrict__ L, int n, int p0,
                                                 const int* __restrict__ info, const unsigned long long* gate) {
    if (rg_stop(info, gate)) return;
    __shared__ double li[16][RG_NB + 1], lj[16][RG_NB + 1];
    int ti, tj;
    tri_index((int)blockIdx.x, ti, tj);
    const int p1 = p0 + RG_NB, i0 = p1 + 16 * ti, j0 = p1 + 16 * tj;
    for (int t = threadIdx.x; t < 2 * 16 * RG_NB; t += 256) {
        const int r = (t >> 5) & 15, c = t & 31, i = (t < 512 ? i0 : j0) + r;
        (t < 512 ? li : lj)[r][c] = i < n ? L[(int64_t)i * n + p0 + c] : 0.0;
    }
    __syncthreads();
    const int r = threadIdx.x >> 4, c = threadIdx.x & 15, i = i0 + r, j = j0 + c;
    if (i >= n || j > i) return;
    double s0 = 0.0, s1 = 0.0;
#pragma unroll
    for (int k = 0; k < RG_NB; k += 2) {
        s0 = fma(li[r][k], lj[c][k], s0);
        s1 = fma(li[r][k + 1], lj[c][k + 1], s1);
    }
    A[(int64_t)i * n + j] -= s0 + s1;
}

// L x = b for nrhs right-hand sides, four per CTA, in blocks of 32 rows: warp w solves the block's triangle for
// right-hand side w by shuffles, then the four warps share the rows below, each entry of L read once for the
// four.  b(i) of right-hand side j at B[i * bs + j * br], the solution at X[i * xs + j * xr].  sv (nullable): b
// is scaled by sv[i] sv[j].  half: only the rows up to the last of the CTA's right-hand sides.
__global__ void __launch_bounds__(128) k_rg_fwd(const double* __restrict__ LT, const double* __restrict__ rl, int n, int nrhs,
                                                const double* __restrict__ B, int64_t bs, int64_t br,
                                                const double* __restrict__ sv, double* __restrict__ X, int64_t xs, int64_t xr,
                                                int half, const int* __restrict__ info, const unsigned long long* gate) {
    if (rg_stop(info, gate)) return;
    extern __shared__ double fsm[];   // [n][4]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int j0 = (int)blockIdx.x * 4;
    const int rows = half ? min(n, j0 + 4) : n;
    for (int t = tid; t < 4 * rows; t += 128) {
        // consecutive threads on consecutive addresses of B
        const int c = br == 1 ? t & 3 : t / rows, i = br == 1 ? t >> 2 : t - c * rows, j = j0 + c;
        double b = j < nrhs ? B[i * bs + j * br] : 0.0;
        if (sv && j < nrhs) b = b * sv[i] * sv[j];
        fsm[4 * i + c] = b;
    }
    __syncthreads();
    for (int b0 = 0; b0 < rows; b0 += 32) {
        const int r = b0 + lane, nb = min(32, rows - b0);
        {
            double lv[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) lv[i] = (i < nb && r < rows) ? LT[(int64_t)(b0 + i) * n + r] : 0.0;
            const double rv = r < rows ? rl[r] : 0.0;
            double xv = r < rows ? fsm[4 * r + warp] : 0.0;
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                const double xi = __shfl_sync(0xffffffffu, xv * rv, i);   // lane i's is final
                if (lane == i) xv = xi;
                else if (lane > i) xv = fma(-lv[i], xi, xv);
            }
            if (r < rows) fsm[4 * r + warp] = xv;
        }
        __syncthreads();
        for (int r2 = b0 + 32 + tid; r2 < rows; r2 += 128) {   // nb = 32 when there are rows below
            const double* lc = LT + (int64_t)b0 * n + r2;
            double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 16
            for (int i = 0; i < 32; ++i) {
                const double l = lc[(int64_t)i * n];
#pragma unroll
                for (int c = 0; c < 4; ++c) s[c] = fma(l, fsm[4 * (b0 + i) + c], s[c]);
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) fsm[4 * r2 + c] -= s[c];
        }
        __syncthreads();
    }
    for (int t = tid; t < 4 * rows; t += 128) {
        const int c = xr == 1 ? t & 3 : t / rows, i = xr == 1 ? t >> 2 : t - c * rows, j = j0 + c;
        if (j < nrhs) X[i * xs + j * xr] = fsm[4 * i + c];
    }
}

// Householder tridiagonalisation of C (its lower triangle, element (i, j <= i) at C[i q + j]) on one
// cluster.  Row i lives in CTA i % NC (cyclic), in shared memory when it fits (arows = NULL), else in the
// CTA's part of arows.  One cluster barrier per column: p = tau A v of the owned rows is pushed to every CTA
// and the owner of the next row leaves it in global memory, barrier, and then every CTA forms w = p -
// (tau/2)(p.v) v, the next row and its reflector for itself (warps 0-3), while warps 4-15 apply the rank-2
// update to the owned rows.  q = 149: 0.58 ms, a chain of about 3.9 us per column (barrier 0.5, dot product
// 0.8, reflector 1.4, p 0.9); q = 538: 4.8 ms, bound by the FP64 units of 16 SMs in the update and p.  The FP64
// unit of an SM sub-partition takes 64 clocks per warp instruction, so short vector steps run on four warps, in
// loops over shared memory: unrolled over registers, the compiler issues the FP64 instructions of the absent
// entries too (about 100 clocks each).
__global__ void __launch_bounds__(RG_TRI_THREADS, 1) k_rg_tridiag(const double* __restrict__ C, int q, int lda,
                                                                  double* __restrict__ arows, double* __restrict__ rowbuf,
                                                                  double* __restrict__ VH, double* __restrict__ tau,
                                                                  double* __restrict__ dg, double* __restrict__ eg,
                                                                  const int* __restrict__ info) {
    cg::cluster_group cluster = cg::this_cluster();
    constexpr int NC = RG_CLUSTER;
    const int rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (rg_stop(info, nullptr)) return;   // the same in every CTA
    extern __shared__ __align__(16) double tsm[];
    const int nrows = rank < q ? (q - rank + NC - 1) / NC : 0, maxrows = (q + NC - 1) / NC;
    double* vb2 = tsm;                      // [2][q + 1]: reflector, tau at [q]
    double* pb2 = vb2 + 2 * (q + 1);        // [2][q]: p, then w
    double* rb = pb2 + 2 * q;               // [q]: the row that becomes a reflector (entry j by thread (j - i) % 128)
    double* red = rb + q;                   // [8]
    double* A = arows ? arows + (int64_t)rank * maxrows * lda : red + 8;
    for (int t = tid; t < nrows * q; t += RG_TRI_THREADS) {
        const int li = t / q, j = t - li * q, i = rank + NC * li;
        A[(int64_t)li * lda + j] = j <= i ? C[(int64_t)i * q + j] : C[(int64_t)j * q + i];
    }
    // sum over the first four warps' lanes; the result in all of their lanes (warps 0-3 only)
    auto sum4 = [&](double v) {
        v = wsum(v);
        if (lane == 0) red[warp] = v;
        asm volatile("bar.sync 1, 128;" ::: "memory");
        const double s = (red[0] + red[1]) + (red[2] + red[3]);
        asm volatile("bar.sync 1, 128;" ::: "memory");
        return s;
    };
    // reflector of row i from its entries rb[i ..] (warps 0-3 of every CTA); rank 0 records it
    auto make_v = [&](int i) {
        double* vb = vb2 + (i & 1) * (q + 1);
        // the squares behind x0 on their own: taken from the whole sum by subtraction, entries below 1e-8 |x0| would
        // be lost, and dropped from T instead of eliminated
        double tail = 0.0;
        for (int j = i + tid; j < q; j += 128) tail = fma(j > i + 1 ? rb[j] : 0.0, rb[j], tail);
        tail = sum4(tail);
        const double x0 = rb[i + 1];   // thread 1's entry: visible after sum4's barriers
        const double s2 = fma(x0, x0, tail);
        double alpha = x0, t = 0.0;
        if (mag(tail) >= mag(RR_TAIL_MIN)) {   // NaN too
            alpha = -copysign(s2 * rsqrt(s2), x0);
            t = rcp64(fma(-alpha, x0, s2));   // 2 / v^T v with v^T v = 2 (s2 - alpha x0)
        }
        for (int j = i + 1 + tid; j < q; j += 128) {
            const double v = t == 0.0 ? 0.0 : (j == i + 1 ? x0 - alpha : rb[j]);
            vb[j] = v;
            if (rank == 0) VH[(int64_t)i * q + j] = v;
        }
        if (tid == 0) {
            vb[q] = t;
            if (rank == 0) {
                tau[i] = t;
                dg[i] = rb[i];
                eg[i] = alpha;
            }
        }
    };
    // p = tau A v_i on the owned rows below i (16 lanes per row), to every CTA; row i + 1 to global memory
    auto push_p = [&](int i) {
        const double* vb = vb2 + (i & 1) * (q + 1);
        double* pb = pb2 + (i & 1) * q;
        const double t = vb[q];
        const int li0 = i + 1 <= rank ? 0 : (i + 1 - rank + NC - 1) / NC;   // first owned row > i
        if (rank == (i + 1) % NC)
            for (int j = i + 1 + tid; j < q; j += RG_TRI_THREADS) rowbuf[((i + 1) & 1) * q + j] = A[(int64_t)li0 * lda + j];
        const int l = tid & 15;
        const unsigned hm = 0xFFFFu << (lane & 16);
        for (int li = li0 + (tid >> 4); li < nrows; li += RG_TRI_THREADS / 16) {
            const double* ai = A + (int64_t)li * lda;
            double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
            int j = i + 1 + l;
            for (; j + 48 < q; j += 64) {
                s0 = fma(ai[j], vb[j], s0);
                s1 = fma(ai[j + 16], vb[j + 16], s1);
                s2 = fma(ai[j + 32], vb[j + 32], s2);
                s3 = fma(ai[j + 48], vb[j + 48], s3);
            }
            for (; j < q; j += 16) s0 = fma(ai[j], vb[j], s0);
            s0 = (s0 + s1) + (s2 + s3);
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) s0 += __shfl_xor_sync(hm, s0, o);
            s0 *= t;
            if (l < NC) cluster.map_shared_rank(pb, l)[rank + NC * li] = s0;
        }
    };
    cluster.sync();   // every CTA is there before the first remote store
    if (warp < 4) {
        for (int j = tid; j < q; j += 128) rb[j] = C[(int64_t)j * q];
        make_v(0);
    }
    __syncthreads();
    push_p(0);
    for (int kk = 0; kk + 2 < q; ++kk) {
        cluster.sync();                                           // p and row kk + 1 are everywhere
        const double* vb = vb2 + (kk & 1) * (q + 1);
        double* pb = pb2 + (kk & 1) * q;
        const int i = kk + 1;
        if (warp < 4) {
            double pv = 0.0;
            for (int j = i + tid; j < q; j += 128) pv = fma(pb[j], vb[j], pv);
            const double K = 0.5 * vb[q] * sum4(pv);
            for (int j = i + tid; j < q; j += 128) pb[j] = fma(-K, vb[j], pb[j]);   // w
        } else {
            for (int j = i + tid - 128; j < q; j += RG_TRI_THREADS - 128) rb[j] = __ldcg(rowbuf + (i & 1) * q + j);   // row i
        }
        __syncthreads();
        if (warp < 4) {
            const double vi = vb[i], wi = pb[i];
            for (int j = i + tid; j < q; j += 128) rb[j] = fma(-vi, pb[j], fma(-wi, vb[j], rb[j]));
            if (i + 2 < q) {
                make_v(i);
            } else if (rank == 0) {   // the last 2 x 2 block
                if (tid == 0) dg[i] = rb[i];
                if (tid == 1) eg[i] = rb[i + 1];
            }
        } else {
            const int li0 = i + 1 <= rank ? 0 : (i + 1 - rank + NC - 1) / NC;   // first owned row > i
            const int nch = (q - i - 1 + 63) / 64, ntask = (nrows - li0) * nch;   // (row, 64 columns) over the warps
            for (int t = warp - 4; t < ntask; t += RG_TRI_THREADS / 32 - 4) {
                const int tr = t / nch, j = i + 1 + 64 * (t - tr * nch) + lane;
                const int ri = rank + NC * (li0 + tr);
                const double vr = vb[ri], wr = pb[ri];
                double* a = A + (int64_t)(li0 + tr) * lda + j;
                const bool on0 = j < q, on1 = j + 32 < q;
                double a0 = 0.0, a1 = 0.0, v0 = 0.0, v1 = 0.0, w0 = 0.0, w1 = 0.0;
                if (on0) { a0 = a[0]; v0 = vb[j]; w0 = pb[j]; }
                if (on1) { a1 = a[32]; v1 = vb[j + 32]; w1 = pb[j + 32]; }
                a0 = fma(-wr, v0, a0);
                a1 = fma(-wr, v1, a1);
                a0 = fma(-vr, w0, a0);
                a1 = fma(-vr, w1, a1);
                if (on0) a[0] = a0;
                if (on1) a[32] = a1;
            }
        }
        __syncthreads();
        if (i + 2 < q) push_p(i);
    }
    cluster.sync();                                               // no CTA leaves while others still write to it
    if (rank == (q - 1) % NC && tid == 0) {
        dg[q - 1] = A[(int64_t)((q - 1) / NC) * lda + q - 1];
        eg[q - 1] = 0.0;
    }
}

// Gershgorin interval and ||T|| by one warp
struct TriBounds {
    double gl, gu, tnorm, pivmin;
};
__device__ __forceinline__ TriBounds tri_bounds(const double* dd, const double* ee, int q, int lane) {
    TriBounds b{DBL_MAX, -DBL_MAX, 0.0, 0.0};
    for (int i = lane; i < q; i += 32) {
        const double r = (i > 0 ? fabs(ee[i - 1]) : 0.0) + (i < q - 1 ? fabs(ee[i]) : 0.0);
        b.gl = fmin(b.gl, dd[i] - r);
        b.gu = fmax(b.gu, dd[i] + r);
        b.tnorm = fmax(b.tnorm, fabs(dd[i]) + r);
    }
    for (int o = 16; o > 0; o >>= 1) {
        b.gl = fmin(b.gl, __shfl_xor_sync(0xffffffffu, b.gl, o));
        b.gu = fmax(b.gu, __shfl_xor_sync(0xffffffffu, b.gu, o));
        b.tnorm = fmax(b.tnorm, __shfl_xor_sync(0xffffffffu, b.tnorm, o));
    }
    b.pivmin = DBL_MIN * fmax(1.0, b.tnorm * b.tnorm);
    return b;
}

// The k lowest eigenvalues of T, coarse: FP32 Sturm multisection, one warp each (32 points per round)
__global__ void __launch_bounds__(128) k_rg_bisect(const double* __restrict__ dg, const double* __restrict__ eg, int q, int k,
                                                   double* __restrict__ lam, const int* __restrict__ info) {
    if (rg_stop(info, nullptr)) return;
    extern __shared__ float bsm[];
    float* df = bsm;
    float* e2f = df + q;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < q; i += 128) {
        df[i] = (float)dg[i];
        const double e = i < q - 1 ? eg[i] : 0.0;
        e2f[i] = (float)(e * e);
    }
    __syncthreads();
    const int j = (int)blockIdx.x * 4 + warp;
    if (j >= k) return;
    const TriBounds tb = tri_bounds(dg, eg, q, lane);
    const float pivf = FLT_MIN * (float)fmax(1.0, fmin(tb.tnorm * tb.tnorm, 1e30));
    const double span = fmax(tb.gu - tb.gl, DBL_MIN);
    double lo = tb.gl - (1e-5 * span + tb.pivmin), hi = tb.gu + (1e-5 * span + tb.pivmin);   // count(lo) <= j < count(hi)
    for (int it = 0; it < 6; ++it) {
        const float x = (float)(lo + (hi - lo) * (double)(lane + 1) / 33.0);
        int c = 0;
        float qq = df[0] - x;
        if (fabsf(qq) < pivf) qq = -pivf;
        c += qq < 0.f;
        for (int i = 1; i < q; ++i) {
            qq = df[i] - x - __fdividef(e2f[i - 1], qq);   // 2 ulp: the eigenvalue is coarse
            if (fabsf(qq) < pivf) qq = -pivf;
            c += qq < 0.f;
        }
        const int nb = __popc(__ballot_sync(0xffffffffu, c <= j));
        const double nlo = nb > 0 ? lo + (hi - lo) * (double)nb / 33.0 : lo;
        const double nhi = nb < 32 ? lo + (hi - lo) * (double)(nb + 1) / 33.0 : hi;
        lo = nlo;
        hi = nhi;
    }
    if (lane == 0) lam[j] = 0.5 * (lo + hi);
}

// Eigenvector j of T on one warp (rr_math.h), to Vt[j q + i].  vdiag[3][k]: solves after the first, last shift, coarse
// eigenvalue (read by the host under HBSD_RRDBG=2)
__global__ void __launch_bounds__(32) k_rg_invit(const double* __restrict__ dg, const double* __restrict__ eg, int q, int k,
                                                 const double* __restrict__ lam, double* __restrict__ Vt, double* gscr,
                                                 double* __restrict__ vdiag, const int* __restrict__ info) {
    if (rg_stop(info, nullptr)) return;
    extern __shared__ double ism[];
    const int lane = threadIdx.x, j = (int)blockIdx.x;
    double* dd = ism;
    double* ee = dd + q;
    double* scr = gscr ? gscr + (int64_t)j * 4 * q : ee + q;
    for (int i = lane; i < q; i += 32) {
        dd[i] = dg[i];
        ee[i] = i < q - 1 ? eg[i] : 0.0;
    }
    __syncwarp();
    const TriBounds tb = tri_bounds(dd, ee, q, lane);
    double th;
    const int solves = tri_eigenvector(dd, ee, q, k, j, lam, tb.tnorm, tb.pivmin, scr, lane, [&](const double* x) {
        for (int i = lane; i < q; i += 32) Vt[(int64_t)j * q + i] = x[i];
    }, &th);
    if (lane == 0) {
        vdiag[j] = (double)solves;
        vdiag[k + j] = th;
        vdiag[2 * k + j] = lam[j];
    }
}

// G = V^T V (lower triangle) from the rows of Vt (k x q), one 16 x 16 tile per CTA; off = max |G - I|
__global__ void __launch_bounds__(256) k_rg_vgram(const double* __restrict__ Vt, int q, int k, double* __restrict__ G,
                                                  unsigned long long* __restrict__ off, const int* __restrict__ info,
                                                  const unsigned long long* gate) {
    if (rg_stop(info, gate)) return;
    __shared__ double va[16][33], vb[16][33];
    __shared__ double smax[8];
    int ta, tb;
    tri_index((int)blockIdx.x, ta, tb);
    const int r = threadIdx.x >> 4, c = threadIdx.x & 15, a = 16 * ta + r, b = 16 * tb + c;
    double s0 = 0.0, s1 = 0.0;
    for (int i0 = 0; i0 < q; i0 += 32) {
        for (int t = threadIdx.x; t < 1024; t += 256) {
            const int rr = (t >> 5) & 15, cc = t & 31, v = 16 * (t < 512 ? ta : tb) + rr;
            (t < 512 ? va : vb)[rr][cc] = v < k && i0 + cc < q ? Vt[(int64_t)v * q + i0 + cc] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int t = 0; t < 32; t += 2) {
            s0 = fma(va[r][t], vb[c][t], s0);
            s1 = fma(va[r][t + 1], vb[c][t + 1], s1);
        }
        __syncthreads();
    }
    double o = 0.0;
    if (a < k && b <= a) {
        G[(int64_t)a * k + b] = s0 + s1;
        o = fabs((s0 + s1) - (a == b ? 1.0 : 0.0));
    }
    if (off) {
        if (!(o == o)) o = 0.0;   // a NaN is caught at the output
        for (int d = 16; d > 0; d >>= 1) o = fmax(o, __shfl_xor_sync(0xffffffffu, o, d));
        if ((threadIdx.x & 31) == 0) smax[threadIdx.x >> 5] = o;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < 8; ++w) o = fmax(o, smax[w]);
            atomicMax(off, (unsigned long long)__double_as_longlong(o));   // non-negative doubles order as integers
        }
    }
}

// Rayleigh quotients of the orthonormal vectors
__global__ void __launch_bounds__(128) k_rg_quotients(const double* __restrict__ dg, const double* __restrict__ eg, int q, int k,
                                                      const double* __restrict__ V1, const double* __restrict__ V2,
                                                      double* __restrict__ lamr, const int* __restrict__ info,
                                                      const unsigned long long* off) {
    if (rg_stop(info, nullptr)) return;
    const int lane = threadIdx.x & 31, j = (int)blockIdx.x * 4 + (threadIdx.x >> 5);
    if (j >= k) return;
    const double* v = (rg_stop(info, off) ? V1 : V2) + (int64_t)j * q;
    double acc = 0.0;
    for (int i = lane; i < q; i += 32) {
        acc = fma(dg[i] * v[i], v[i], acc);
        if (i + 1 < q) acc = fma(2.0 * eg[i] * v[i], v[i + 1], acc);
    }
    acc = wsum(acc);
    if (lane == 0) lamr[j] = acc;
}

// Products of the reflectors of a block (columns 32 b .. 32 b + 31): GV[b][i][j] = v_i . v_j for i < j, one 16 x 16
// tile per CTA
__global__ void __launch_bounds__(256) k_rg_vhgram(const double* __restrict__ VH, int q, double* __restrict__ GV,
                                                   const int* __restrict__ info) {
    if (rg_stop(info, nullptr)) return;
    __shared__ double va[16][33], vb[16][33];
    const int b0 = 32 * (int)blockIdx.x, ta = blockIdx.y == 2, tb = blockIdx.y >= 1;   // tiles (0,0), (0,1), (1,1)
    const int r = threadIdx.x >> 4, c = threadIdx.x & 15;
    double s0 = 0.0, s1 = 0.0;
    for (int i0 = b0 & ~31; i0 < q; i0 += 32) {
        for (int t = threadIdx.x; t < 1024; t += 256) {
            const int v = b0 + 16 * (t < 512 ? ta : tb) + ((t >> 5) & 15), j = i0 + (t & 31);
            (t < 512 ? va : vb)[(t >> 5) & 15][t & 31] = v + 2 < q && j > v && j < q ? VH[(int64_t)v * q + j] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int t = 0; t < 32; t += 2) {
            s0 = fma(va[r][t], vb[c][t], s0);
            s1 = fma(va[r][t + 1], vb[c][t + 1], s1);
        }
        __syncthreads();
    }
    GV[((int64_t)blockIdx.x * 32 + 16 * ta + r) * 32 + 16 * tb + c] = s0 + s1;
}

// One CTA per vector: y = H_0 H_1 ... H_{q-3} z, then x = D L^{-T} y, both in blocks of 32 from the last to the
// first.  A block of reflectors is applied as I - V T V^T (compact WY): s = V^T z (lanes over the entries, 8
// reflectors per warp), s' = T s from T^{-1} = diag(1/tau) + the strict upper triangle of V^T V by back
// substitution on one warp, z -= V s'.  The triangle of L^T likewise on one warp, the rows above by all.
// Column and eigenvalue go to their place in ascending order (ties by index).
__global__ void __launch_bounds__(128) k_rg_back(const double* __restrict__ VH, const double* __restrict__ GV,
                                                 const double* __restrict__ tau, const double* __restrict__ L,
                                                 const double* __restrict__ rl, int q, int k, const double* __restrict__ V1,
                                                 const double* __restrict__ V2, const double* __restrict__ lamr,
                                                 const double* __restrict__ dv, double* __restrict__ theta,
                                                 double* __restrict__ W, int* __restrict__ info, const unsigned long long* off) {
    if (rg_stop(info, nullptr)) return;
    extern __shared__ double xsm[];
    __shared__ double ss[32];
    __shared__ int s_rank;
    double* x = xsm;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, j = (int)blockIdx.x;
    const double* y = (rg_stop(info, off) ? V1 : V2) + (int64_t)j * q;
    for (int i = tid; i < q; i += 128) x[i] = y[i];
    __syncthreads();
    for (int b0 = ((q - 3) / 32) * 32; b0 >= 0; b0 -= 32) {
        const int nv = min(32, q - 2 - b0);
        double s[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) s[u] = 0.0;
        for (int i0 = b0; i0 < q; i0 += 32) {
            const int i = i0 + lane;
            const double xi = i < q ? x[i] : 0.0;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int v = 8 * warp + u;
                const double h = v < nv && i > b0 + v && i < q ? VH[(int64_t)(b0 + v) * q + i] : 0.0;
                s[u] = fma(h, xi, s[u]);
            }
        }
        // sums over the lanes of 8 values: three halvings leave one value per 4 lanes
#pragma unroll
        for (int o = 16, w = 4; o > 2; o >>= 1, w >>= 1) {
#pragma unroll
            for (int u = 0; u < w; ++u) {
                const bool up = (lane & o) != 0;
                const double give = up ? s[u] : s[u + w], keep = up ? s[u + w] : s[u];
                s[u] = keep + __shfl_xor_sync(0xffffffffu, give, o);
            }
        }
        s[0] += __shfl_xor_sync(0xffffffffu, s[0], 2);
        s[0] += __shfl_xor_sync(0xffffffffu, s[0], 1);
        // lane bits 4, 3, 2 chose the upper half of 8, 4, 2 values
        if ((lane & 3) == 0) ss[8 * warp + ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1)] = s[0];
        __syncthreads();
        if (warp == 0) {
            const double* g = GV + ((int64_t)(b0 / 32) * 32 + lane) * 32;   // row lane: v_lane . v_j
            double gv[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) gv[i] = i > lane && i < nv && lane < nv ? g[i] : 0.0;
            const double tl = lane < nv ? tau[b0 + lane] : 0.0;
            double sv = lane < nv ? ss[lane] : 0.0;
#pragma unroll
            for (int i = 31; i >= 0; --i) {
                const double si = __shfl_sync(0xffffffffu, sv * tl, i);   // lane i's is final
                if (lane == i) sv = si;
                else if (lane < i) sv = fma(-gv[i], si, sv);
            }
            ss[lane] = lane < nv ? sv : 0.0;
        }
        __syncthreads();
        for (int i = b0 + 1 + tid; i < q; i += 128) {
            double a0 = 0.0, a1 = 0.0;
            if (i > b0 + 32 && nv == 32) {
                const double* h = VH + (int64_t)b0 * q + i;
#pragma unroll 16
                for (int v = 0; v < 32; v += 2) {
                    a0 = fma(h[(int64_t)v * q], ss[v], a0);
                    a1 = fma(h[(int64_t)(v + 1) * q], ss[v + 1], a1);
                }
            } else {
                for (int v = 0; v < nv && b0 + v < i; ++v) a0 = fma(VH[(int64_t)(b0 + v) * q + i], ss[v], a0);
            }
            x[i] -= a0 + a1;
        }
        __syncthreads();
    }
    for (int b0 = ((q - 1) / 32) * 32; b0 >= 0; b0 -= 32) {
        const int r = b0 + lane, nb = min(32, q - b0);
        if (warp == 0) {
            double lv[32];   // L(b0 + i, r): row i of the block's triangle
#pragma unroll
            for (int i = 0; i < 32; ++i) lv[i] = (i < nb && lane <= i) ? L[(int64_t)(b0 + i) * q + r] : 0.0;
            const double rv = r < q ? rl[r] : 0.0;
            double xv = r < q ? x[r] : 0.0;
#pragma unroll
            for (int i = 31; i >= 0; --i) {
                const double xi = __shfl_sync(0xffffffffu, xv * rv, i);
                if (lane == i) xv = xi;
                else if (lane < i) xv = fma(-lv[i], xi, xv);   // rows beyond nb have lv = 0
            }
            if (r < q) x[r] = xv;
        }
        __syncthreads();
        for (int r2 = tid; r2 < b0; r2 += 128) {
            const double* lc = L + (int64_t)b0 * q + r2;
            double a0 = 0.0, a1 = 0.0;
            if (nb == 32) {
#pragma unroll 16
                for (int i = 0; i < 32; i += 2) {
                    a0 = fma(lc[(int64_t)i * q], x[b0 + i], a0);
                    a1 = fma(lc[(int64_t)(i + 1) * q], x[b0 + i + 1], a1);
                }
            } else {
                for (int i = 0; i < nb; ++i) a0 = fma(lc[(int64_t)i * q], x[b0 + i], a0);
            }
            x[r2] -= a0 + a1;
        }
        __syncthreads();
    }
    if (warp == 0) {
        const unsigned long long kj = dkey(lamr[j]);
        int rank = 0;
        for (int i = lane; i < k; i += 32) {
            const unsigned long long ki = dkey(lamr[i]);
            rank += (ki < kj) || (ki == kj && i < j);
        }
        for (int o = 16; o > 0; o >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
        if (lane == 0) {
            s_rank = rank;
            theta[rank] = lamr[j];
        }
    }
    __syncthreads();
    const int rank = s_rank;
    bool bad = !isfinite(lamr[j]);
    for (int i = tid; i < q; i += 128) {
        const double v = dv[i] * x[i];
        bad |= !isfinite(v);
        W[(int64_t)i * k + rank] = v;
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(info + 2, 1);
}

}  // namespace

size_t rr_grid_ws_doubles(int q, int k) {
    const int lda = q + 20, maxrows = (q + RG_CLUSTER - 1) / RG_CLUSTER;
    return (size_t)6 * q * q + (size_t)RG_CLUSTER * maxrows * lda + (size_t)2 * q * k + (size_t)3 * k * k +
           (size_t)4 * q * k + 42 * (size_t)q + 7 * (size_t)k + 1200;
}
size_t rr_grid_vdiag(int q, int k) { return rr_grid_ws_doubles(q, k) - 3 * (size_t)k; }

// Launches the whole reduced solve (info must be zero); *launched = false: the cluster cannot be scheduled here and
// nothing was launched.  ev (nullable): 8 events, recorded before the first launch and after each phase.
int rayleigh_ritz_grid(Session* s, const double* HR, const double* SR, int q, int k, double* theta, double* W, double* ws,
                       int* info, cudaStream_t st, bool* launched, cudaEvent_t* ev) {
    *launched = false;
    auto mark = [&](int i) {
        if (ev) (void)cudaEventRecord(ev[i], st);
    };
    const size_t qq = (size_t)q * q, kk = (size_t)k * k, qk = (size_t)q * k;
    double* A = ws;
    double* L = A + qq;
    double* LT = L + qq;
    double* T = LT + qq;
    double* C = T + qq;
    double* VH = C + qq;
    double* V1 = VH + qq;
    double* V2 = V1 + qk;
    double* G = V2 + qk;
    double* LG = G + kk;
    double* LGT = LG + kk;
    double* dv = LGT + kk;
    double* rl = dv + q;
    double* tau = rl + q;
    double* dg = tau + q;
    double* eg = dg + q;
    double* lam = eg + q;
    double* lamr = lam + k;
    double* rlg = lamr + k;
    unsigned long long* off = reinterpret_cast<unsigned long long*>(rlg + k);
    double* scr = rlg + k + 8;               // 4 q k: inverse iteration when q is too large for shared memory
    double* rowbuf = scr + 4 * qk;           // 2 q
    double* GV = rowbuf + 2 * q;             // 32 per reflector
    double* arows = GV + (size_t)32 * (q + 32);
    // rows of the tridiagonalisation: a leading dimension of 4 mod 16 puts eight rows on distinct banks
    const int lda = (int)round_up(q, 16) + 4;
    const int maxrows = ceil_div(q, RG_CLUSTER);
    const size_t tri_fixed = (size_t)(5 * q + 2 + 8) * sizeof(double);
    const bool in_sm = tri_fixed + (size_t)maxrows * lda * sizeof(double) <= RG_SMEM_MAX;
    const size_t tri_sm = tri_fixed + (in_sm ? (size_t)maxrows * lda * sizeof(double) : 0);
    const size_t fwd_sm = (size_t)4 * q * sizeof(double), back_sm = (size_t)q * sizeof(double);
    const bool inv_in = (size_t)6 * q * sizeof(double) <= 100 * 1024;
    const size_t inv_sm = (size_t)(inv_in ? 6 : 2) * q * sizeof(double);
    const size_t bis_sm = (size_t)2 * q * sizeof(float);
    if (q < 3 || tri_sm > RG_SMEM_MAX || fwd_sm > RG_SMEM_MAX || inv_sm > RG_SMEM_MAX) return 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(RG_CLUSTER, 1, 1);
    cfg.blockDim = dim3(RG_TRI_THREADS, 1, 1);
    cfg.dynamicSmemBytes = tri_sm;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = RG_CLUSTER;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    {
        static std::mutex mu;   // sessions of a server call this from several threads
        static int ok = 0;
        std::lock_guard<std::mutex> lk(mu);
        if (ok == 0) {   // once: shared-memory limits, and whether a full-size cluster can be scheduled
            HBSD_CUDA(cudaFuncSetAttribute(k_rg_tridiag, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RG_SMEM_MAX));
            HBSD_CUDA(cudaFuncSetAttribute(k_rg_tridiag, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
            HBSD_CUDA(cudaFuncSetAttribute(k_rg_fwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RG_SMEM_MAX));
            HBSD_CUDA(cudaFuncSetAttribute(k_rg_invit, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RG_SMEM_MAX));
            HBSD_CUDA(cudaFuncSetAttribute(k_rg_bisect, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RG_SMEM_MAX));
            HBSD_CUDA(cudaFuncSetAttribute(k_rg_back, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RG_SMEM_MAX));
            cudaLaunchConfig_t full = cfg;
            full.dynamicSmemBytes = RG_SMEM_MAX;
            int nclusters = 0;
            const cudaError_t e = cudaOccupancyMaxActiveClusters(&nclusters, k_rg_tridiag, &full);
            if (e != cudaSuccess) (void)cudaGetLastError();
            ok = e == cudaSuccess && nclusters >= 1 ? 1 : -1;
        }
        if (ok < 0) return 0;
    }
    auto cholesky = [&](double* M, int n, int clamp, double* Lo, double* Lt, double* r, const unsigned long long* gate) -> int {
        for (int p0 = 0; p0 < n; p0 += RG_NB) {
            const int below = std::max(0, n - p0 - RG_NB);
            k_rg_panel<<<std::max(1, ceil_div(below, 8)), 256, 0, st>>>(M, n, p0, clamp, Lo, Lt, r, info, gate);
            HBSD_LAUNCHED(s);
            if (below > 0) {
                const int t = ceil_div(below, 16);
                k_rg_syrk<<<t * (t + 1) / 2, 256, 0, st>>>(M, Lo, n, p0, info, gate);
                HBSD_LAUNCHED(s);
            }
        }
        return 0;
    };
    HBSD_CUDA(cudaMemsetAsync(off, 0, 2 * sizeof(*off), st));
    *launched = true;
    mark(0);
    const int tq = ceil_div(q, 32);
    k_rg_scale<<<dim3(tq, tq), 256, 0, st>>>(SR, q, A, dv);
    HBSD_LAUNCHED(s);
    HBSD_TRY(cholesky(A, q, 0, L, LT, rl, nullptr));
    mark(1);
    // T(:, j) = L^{-1} Hd(:, j) at T[j q + i]; C(:, j) = L^{-1} T(j, :)^T, rows up to j's block, at C[j q + i]
    k_rg_fwd<<<ceil_div(q, 4), 128, fwd_sm, st>>>(LT, rl, q, q, HR, 1, q, dv, T, 1, q, 0, info, nullptr);
    HBSD_LAUNCHED(s);
    k_rg_fwd<<<ceil_div(q, 4), 128, fwd_sm, st>>>(LT, rl, q, q, T, q, 1, nullptr, C, 1, q, 1, info, nullptr);
    HBSD_LAUNCHED(s);
    mark(2);
    HBSD_CUDA(cudaLaunchKernelEx(&cfg, k_rg_tridiag, (const double*)C, q, lda, in_sm ? (double*)nullptr : arows, rowbuf, VH, tau, dg, eg,
                                 (const int*)info));
    HBSD_LAUNCHED(s);
    mark(3);
    k_rg_bisect<<<ceil_div(k, 4), 128, bis_sm, st>>>(dg, eg, q, k, lam, info);
    HBSD_LAUNCHED(s);
    mark(4);
    k_rg_invit<<<k, 32, inv_sm, st>>>(dg, eg, q, k, lam, V1, inv_in ? nullptr : scr, ws + rr_grid_vdiag(q, k), info);
    HBSD_LAUNCHED(s);
    mark(5);
    // CholeskyQR: V1 -> V2, and V2 -> V1 when the first pass found the vectors far from orthonormal
    const int tk = ceil_div(k, 16);
    for (int pass = 0; pass < 2; ++pass) {
        const unsigned long long* gate = pass ? off : nullptr;
        double* from = pass ? V2 : V1;
        double* to = pass ? V1 : V2;
        k_rg_vgram<<<tk * (tk + 1) / 2, 256, 0, st>>>(from, q, k, G, pass ? nullptr : off, info, gate);
        HBSD_LAUNCHED(s);
        HBSD_TRY(cholesky(G, k, 1, LG, LGT, rlg, gate));
        k_rg_fwd<<<ceil_div(q, 4), 128, (size_t)4 * k * sizeof(double), st>>>(LGT, rlg, k, q, from, q, 1, nullptr, to, q, 1, 0, info,
                                                                            gate);
        HBSD_LAUNCHED(s);
    }
    mark(6);
    // the vectors are in V2, or in V1 after a second pass (rg_stop(info, off) chooses)
    k_rg_quotients<<<ceil_div(k, 4), 128, 0, st>>>(dg, eg, q, k, V2, V1, lamr, info, off);
    HBSD_LAUNCHED(s);
    k_rg_vhgram<<<dim3(ceil_div(q - 2, 32), 3), 256, 0, st>>>(VH, q, GV, info);
    HBSD_LAUNCHED(s);
    k_rg_back<<<k, 128, back_sm, st>>>(VH, GV, tau, L, rl, q, k, V2, V1, lamr, dv, theta, W, info, off);
    HBSD_LAUNCHED(s);
    mark(7);
    return 0;
}

}  // namespace hbsd
