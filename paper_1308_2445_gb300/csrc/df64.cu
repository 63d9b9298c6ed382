// Double-float ("df64") block products for the mixed form: steps 8 (Gram) and 10-11 (update).
//
// GB300 issues FP32 FMAs at 128 lanes per clock per SM and FP64 FMAs at 2, so a product whose
// FP64 rate is the bound runs faster as pairs of floats (hi + lo, Dekker 1971; Knuth's
// TwoSum): a product of two pairs is hi*hi exactly (TwoProd by FMA) plus the two cross terms,
// and the running sum is a pair kept by TwoSum and renormalised every few terms.  About 48
// significant bits per term; the Gram sums go over to FP64 every 64 rows, so their long sums
// carry FP64 accuracy.  Large products run on the tensor cores instead (gram_tc.cu, update_tc.cu).
//
// The pair arithmetic (split, TwoProd + TwoSum, renormalisation) is in df64.h.
#include <algorithm>
#include <cmath>
#include <mutex>

#include "common.h"
#include "df64.h"
#include "gram_tile.h"

namespace hbsd {

namespace {

using df::Seg2d;
using df::split_d;
using df::dfma;
using df::renorm;
using df::to_d;

// One CTA: a tile (a-block <= b-block, tw = 4 nb columns wide) of Z^T H Z (warps 0-1) and Z^T S Z
// (warps 2-3) over a chunk of rows.  Bound by the FP32 pipe (10 instructions per multiply-add of
// pairs, on two packed lanes).  32-wide tiles of 4 x 4 outputs per thread keep the padding of the
// triangle at 8% for q = 538 (64-wide tiles: 27%) and the warps of a CTA equally loaded; one matrix
// per warp pair keeps a thread at 128 registers without spills (both matrices in one thread: 24
// bytes spilled, 49 ms).  Stages of 4 rows, the next one's loads in flight during the sums; FP64
// sums in shared memory, flushed every 64 rows (with the 10-instruction multiply-add 64 rows are at
// least as accurate as 128 rows with the 12-instruction one).  n = 47,620, q = 149: 0.64 ms against
// 0.89 ms for 2 x 2 outputs per thread and scalar instructions; n = 646, q = 35: 33 against 64 us.
__global__ void __launch_bounds__(GTHREADS, GCTAS) k_gram_df64(Seg2d Z, Seg2d ZH, Seg2d ZS, int q, int64_t n,
                                                           int64_t rows_per_chunk, int ntile, int nb, df::f32x2 nz,
                                                           double* __restrict__ partial) {
    __shared__ GramTile sm;
    // tile pair: the off-diagonal ones first, then the diagonal ones (half the work)
    const int noff = ntile * (ntile - 1) / 2;
    int ta, tb;
    if ((int)blockIdx.x < noff) {
        tri_index((int)blockIdx.x, tb, ta);   // ta <= tb of the strict triangle
        ++tb;
    } else {
        ta = tb = (int)blockIdx.x - noff;
    }
    const int64_t r0 = (int64_t)blockIdx.y * rows_per_chunk;
    const int64_t qq = (int64_t)q * q;
    double* ph = partial + (int64_t)blockIdx.y * 2 * qq;
    gram_df64_tile(sm, Z, ZH, ZS, q, ta * 4 * nb, tb * 4 * nb, nb, ta == tb, r0, min(n, r0 + rows_per_chunk), nz,
                   [&](int m, int a, int b, double v) { ph[m * qq + (int64_t)a * q + b] = v; });
}

// Sum the chunks in order; entry (a, b), a <= b, of Z^T X Z is used for both (a, b) and (b, a).
__global__ void __launch_bounds__(256) k_gram_final_upper(const double* __restrict__ partial, int nchunks, int q,
                                                          double* __restrict__ HR, double* __restrict__ SR) {
    // 32 entries per block (lanes), the chunks split over the 8 warps, then summed in warp order:
    // the order is fixed, so the result is deterministic.  Entries a <= b are summed and mirrored.
    __shared__ double rh[8][33], rs[8][33];
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
    const int64_t qq = (int64_t)q * q;
    const int64_t idx = (int64_t)blockIdx.x * 32 + lane;
    const int a = (int)(idx / q), b = (int)(idx - (int64_t)(idx / q) * q);
    const bool on = idx < qq && a <= b;
    double h = 0.0, sv = 0.0;
    if (on)
        for (int c = g; c < nchunks; c += 8) {
            const double* ph = partial + (int64_t)c * 2 * qq;
            h += ph[idx];
            sv += ph[qq + idx];
        }
    rh[g][lane] = h;
    rs[g][lane] = sv;
    __syncthreads();
    if (g == 0 && on) {
        double H = 0.0, S = 0.0;
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            H += rh[t][lane];
            S += rs[t][lane];
        }
        HR[idx] = H;
        SR[idx] = S;
        HR[(int64_t)b * q + a] = H;
        SR[(int64_t)b * q + a] = S;
    }
}

// W (q x k, FP64) -> pairs
__global__ void k_split_w(const double* __restrict__ W, int64_t cnt, float2* __restrict__ W2, const unsigned* gate,
                          unsigned cap) {
    if (gate && __ldcg(gate) <= cap) return;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < cnt; t += (int64_t)gridDim.x * blockDim.x)
        W2[t] = split_d(W[t]);
}

// Y(:, 0:k) <- [Z0 Z1] W, Y = Z0 allowed (a CTA writes only the rows it has staged).  With gate, only when *gate >
// cap.  Threads are flattened over (row group, column): kc = min(k, 256)
// columns per pass, ng = min(256 / kc, 8) row groups of UR rows, so a CTA covers ng * UR rows;
// the rows (split) and W (q x k pairs) are staged in shared memory, W shared by the row groups.
// Every output sums its q terms in column order, the running pair renormalised after each
// term whose index is 7 mod 8 (the loops run in blocks of RN = 8 terms and a short tail).
constexpr int UR = 8;
constexpr int RN = 8;

__global__ void __launch_bounds__(256) k_update_df64(const double* Z0, int64_t ld0, int q0,
                                                     const double* __restrict__ Z1, int64_t ld1, int q1, int64_t n,
                                                     const float2* __restrict__ W2, int k, int ng, double* Y,
                                                     int64_t ldy, const unsigned* gate, unsigned cap) {
    if (gate && __ldcg(gate) <= cap) return;
    extern __shared__ __align__(16) float2 smu[];
    const int q = q0 + q1;
    const int rows = ng * UR;
    float2* zrow = smu;                      // [rows][q]
    float2* wsm = smu + (int64_t)rows * q;   // [q][k]
    const int64_t i0 = (int64_t)blockIdx.x * rows;
    for (int t = threadIdx.x; t < rows * q; t += 256) {
        const int rr = t / q, c = t % q;
        const int64_t i = i0 + rr;
        double v = 0.0;
        if (i < n) v = c < q0 ? Z0[i * ld0 + c] : Z1[i * ld1 + (c - q0)];
        zrow[t] = split_d(v);
    }
    for (int t = threadIdx.x; t < q * k; t += 256) wsm[t] = W2[t];
    __syncthreads();
    const int kc = min(k, 256);
    const int g = threadIdx.x / kc, cl = threadIdx.x % kc;
    if (g >= ng) return;
    const float2* zr = zrow + (int64_t)g * UR * q;
    for (int jb = 0; jb < k; jb += kc) {
        const int j = jb + cl;
        if (j >= k) continue;
        float ah[UR], al[UR];
#pragma unroll
        for (int u = 0; u < UR; ++u) { ah[u] = 0.f; al[u] = 0.f; }
        const float2* wc = wsm + j;
        int c = 0;
        for (; c + RN <= q; c += RN) {
#pragma unroll
            for (int cc = 0; cc < RN; ++cc) {
                const float2 wv = wc[(c + cc) * k];
#pragma unroll
                for (int u = 0; u < UR; ++u) dfma(zr[u * q + c + cc], wv, ah[u], al[u]);
            }
#pragma unroll
            for (int u = 0; u < UR; ++u) renorm(ah[u], al[u]);
        }
        for (; c < q; ++c) {
            const float2 wv = wc[c * k];
#pragma unroll
            for (int u = 0; u < UR; ++u) dfma(zr[u * q + c], wv, ah[u], al[u]);
        }
#pragma unroll
        for (int u = 0; u < UR; ++u) {
            const int64_t i = i0 + g * UR + u;
            if (i < n) Y[i * ldy + j] = to_d(ah[u], al[u]);
        }
    }
}

// The same product for q too large to stage W with the rows: UR rows per CTA staged once
// (split), one output column per thread (blockDim.x columns per pass, a multiple of 32 chosen so
// the passes are even), each thread reading its own column of W straight from L2, RN terms at a
// time (no other thread of the CTA reads it, so staging it would buy nothing).  Same term order
// and renormalisation as above.  In place: the outputs are written only after every row of the
// CTA was staged, and only the staged copy is read.
__global__ void __launch_bounds__(512) k_update_df64_kt(const double* Z0, int64_t ld0, int q0,
                                                        const double* __restrict__ Z1, int64_t ld1, int q1, int64_t n,
                                                        const float2* __restrict__ W2, int k, double* Y, int64_t ldy,
                                                        const unsigned* gate, unsigned cap) {
    if (gate && __ldcg(gate) <= cap) return;
    extern __shared__ __align__(16) float2 smu[];
    const int q = q0 + q1;
    const int nt = blockDim.x;
    float2* zrow = smu;                     // [UR][q]
    const int64_t i0 = (int64_t)blockIdx.x * UR;
    for (int t = threadIdx.x; t < UR * q; t += nt) {
        const int rr = t / q, c = t % q;
        const int64_t i = i0 + rr;
        double v = 0.0;
        if (i < n) v = c < q0 ? Z0[i * ld0 + c] : Z1[i * ld1 + (c - q0)];
        zrow[t] = split_d(v);
    }
    __syncthreads();
    for (int jb = 0; jb < k; jb += nt) {
        const int j = jb + threadIdx.x;
        if (j >= k) break;   // no barrier follows
        float ah[UR], al[UR];
#pragma unroll
        for (int u = 0; u < UR; ++u) { ah[u] = 0.f; al[u] = 0.f; }
        const float2* wc = W2 + j;
        int c = 0;
        for (; c + RN <= q; c += RN) {
            float2 wv[RN];
#pragma unroll
            for (int cc = 0; cc < RN; ++cc) wv[cc] = __ldg(wc + (int64_t)(c + cc) * k);
#pragma unroll
            for (int cc = 0; cc < RN; ++cc) {
#pragma unroll
                for (int u = 0; u < UR; ++u) dfma(zrow[u * q + c + cc], wv[cc], ah[u], al[u]);
            }
#pragma unroll
            for (int u = 0; u < UR; ++u) renorm(ah[u], al[u]);
        }
        for (; c < q; ++c) {
            const float2 wv = __ldg(wc + (int64_t)c * k);
#pragma unroll
            for (int u = 0; u < UR; ++u) dfma(zrow[u * q + c], wv, ah[u], al[u]);
        }
#pragma unroll
        for (int u = 0; u < UR; ++u) {
            const int64_t i = i0 + u;
            if (i < n) Y[i * ldy + j] = to_d(ah[u], al[u]);
        }
    }
}

}  // namespace

// Under capture nothing may be allocated, and a graph keeps the address of its scratch.  The tensor-core forms' scratch
// grows with the rows, so captured calls run the pairs, with scratch that a call of fewer rows has left and a call of
// more rows does not move: the update's copy of W, and for the Gram s->ws, which stops growing at CAPTURED_CTAS CTAs
// per SM and which other calls of the Gram reserve without using it.
static bool stream_captured(cudaStream_t st) {
    cudaStreamCaptureStatus c = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &c) != cudaSuccess) {   // the legacy stream beside another thread's capture
        (void)cudaGetLastError();
        return false;
    }
    return c != cudaStreamCaptureStatusNone;
}
constexpr int CAPTURED_CTAS = 8;
static int captured_chunks(int64_t n, int q) {
    const int ntile = ceil_div(q, GW), npair = ntile * (ntile + 1) / 2;
    return (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, ceil_div(152 * CAPTURED_CTAS, npair)));
}

int gram_df64_reserve(Session* s, int64_t n, int q) { return s->ws.alloc((size_t)captured_chunks(n, q) * 2 * q * q + 64); }

// Tensor cores from n q^2 = 8e7 on: below it the exponent pass, the lists and the fix-up launch (50 us at
// the least) outweigh the products.  Not below 48 columns, whatever the rows: a tile of 128 x (32 + 32) columns is
// then mostly padding.  Measured on both sides, us (k_gram_df64 / tensor cores): q = 71, n = 5,951: 57 / 69,
// n = 15,869: 108 / 92; q = 149, n = 2,252: 57 / 72, n = 5,855: 108 / 75; q = 538, n = 449: 101 / 105, n = 1,036:
// 177 / 142; q = 48, n = 34,722: 115 / 101, n = 434,027: 1,007 / 884; q = 40, n = 81,250: 194 / 196, n = 625,000:
// 1,116 / 1,264; q = 33, n = 275,482: 564 / 580; q = 24, n = 225,694: 249 / 336; q = 19, n = 360,110: 406 / 515.
static bool gram_tc_pays(int64_t n, int q) { return q >= 48 && (double)n * q * q >= 8e7; }

// chunks of rows for the pairs: several waves of CTAs, at least 128 rows each
static int gram_chunks(int64_t n, int q) {
    const int ntile = ceil_div(q, GW), npair = ntile * (ntile + 1) / 2;
    return (int)std::max<int64_t>(1, std::min<int64_t>((n + 127) / 128, ceil_div(GWAVES * 152 * GCTAS, npair)));
}

int gram2_df64(Session* s, const double* Z0, int64_t ld0, int q0, const double* Z1, int64_t ld1, int q1,
               const double* H0, int64_t ldh0, const double* H1, int64_t ldh1, const double* S0, int64_t lds0,
               const double* S1, int64_t lds1, int64_t n, double* HR, double* SR, cudaStream_t st) {
    const int q = q0 + q1;
    if (q <= 0) return 0;
    const bool captured = stream_captured(st);
    if (!captured && gram_tc_pays(n, q))
        return gram2_tc(s, Z0, ld0, q0, Z1, ld1, q1, H0, ldh0, H1, ldh1, S0, lds0, S1, lds1, n, HR, SR, st);
    // tiles of equal width, a multiple of 4 columns up to GW
    const int ntile = ceil_div(q, GW);
    const int nb = ceil_div(ceil_div(q, ntile), 4);
    const int npair = ntile * (ntile + 1) / 2;
    int nch = captured ? captured_chunks(n, q) : gram_chunks(n, q);
    int64_t rpc = round_up((n + nch - 1) / nch, GR);
    nch = (int)((n + rpc - 1) / rpc);
    DBuf<double>& ws = captured ? s->ws : s->df_ws;
    HBSD_TRY(ws.alloc((size_t)nch * 2 * q * q + 64));
    Seg2d Z{Z0, ld0, q0, Z1, ld1}, ZH{H0, ldh0, q0, H1, ldh1}, ZS{S0, lds0, q0, S1, lds1};
    k_gram_df64<<<dim3(npair, nch), GTHREADS, 0, st>>>(Z, ZH, ZS, q, n, rpc, ntile, nb, df::NEG_ZERO2, ws.p);
    HBSD_LAUNCHED(s);
    const int64_t qq = (int64_t)q * q;
    k_gram_final_upper<<<ceil_div(qq, 32), 256, 0, st>>>(ws.p, nch, q, HR, SR);
    HBSD_LAUNCHED(s);
    return 0;
}

// The update on the tensor cores where it is the faster one.  Otherwise one CTA's chain of column tiles and the passes
// over Z for exponents and guard cost more than they save; and a wave of row tiles costs the same however few rows are in
// it, so that blocks of q k < 12000 have to fill theirs (fill) or to be large.  us (pairs / digit slices; n, q, k) below
// the line: 4728, 282, 150: 129 / 172; 3295, 538, 282: 293 / 341; 21701, 128, 72: 123 / 144; 41700, 100, 72: 173 / 184;
// 59000, 96, 84: 255 / 271; 318877, 56, 56: 534 / 756; 233100, 66, 65: 587 / 700; 178571, 80, 70: 541 / 600; 162760, 96,
// 64: 496 / 469.  Above: 7092, 282, 150: 186 / 174; 6591, 538, 282: 548 / 348; 19773, 538, 282: 1,448 / 743; 16276, 128,
// 96: 133 / 108; 32552, 128, 72: 177 / 154; 44500, 112, 81: 231 / 194; 100000, 91, 90: 503 / 385; 334272, 100, 80: 1,390 /
// 1,141.  On 300 measured sizes the slower side is taken by at most 5%.
static bool update_tc_pays(int64_t n, int q, int k) {
    const double qk = (double)q * k, waves = (double)n / UPDATE_TC_WAVE, fill = waves / std::ceil(waves);
    if (n < 6144 || k < 56 || qk < 7200 || n * qk < 2e8) return false;
    return qk >= 12000 || fill >= 0.8 || (qk >= 9000 && n * qk >= 3e8);
}

// The scratch of one call, and the most of a solve whose Grams and updates have q_lo to q_hi columns, the first q_lo of
// them in one block and k of them updated: reserved before the loop, so that nothing is reallocated (and the
// device synchronised) while other sessions run.  Uncaptured calls.
size_t gram_df64_doubles(int64_t n, int q) {
    return gram_tc_pays(n, q) ? gram_tc_doubles(n, q) : (size_t)gram_chunks(n, q) * 2 * q * q + 64;
}
size_t update_df64_doubles(int64_t n, int q0, int q1, int k) {
    return update_tc_pays(n, q0 + q1, k) && k <= UPDATE_TC_MAX_K ? update_tc_doubles(n, q0, q1, k) : 0;
}
size_t df64_solve_doubles(int64_t n, int q_lo, int q_hi, int k) {
    size_t most = 0;
    for (int q = q_lo; q <= q_hi; ++q)
        most = std::max({most, gram_df64_doubles(n, q), update_df64_doubles(n, q_lo, q - q_lo, k)});
    return most;
}

int update2_df64(Session* s, double* Z0, int64_t ld0, int q0, const double* Z1, int64_t ld1, int q1, int64_t n,
                 const double* W, int k, cudaStream_t st, bool split_w) {
    const int q = q0 + q1;
    if (k > q0) return fail(HBSD_ERR_ARG, "update: k must not exceed the first segment width");
    if (update_tc_pays(n, q, k)) {
        if (!stream_captured(st) && (size_t)UR * q * sizeof(float2) <= 220 * 1024 && update_tc_fits(Z0, ld0, Z1, ld1, q1, k))
            return update2_tc(s, Z0, ld0, q0, Z1, ld1, q1, n, W, k, st);
        split_w = true;   // an earlier block of the same step may have gone the other way and left df_w alone
    }
    return update_df64_rows(s, Z0, ld0, q0, Z1, ld1, q1, n, W, k, Z0, ld0, nullptr, 0, st, split_w);
}

int update_df64_rows(Session* s, const double* Z0, int64_t ld0, int q0, const double* Z1, int64_t ld1, int q1, int64_t n,
                     const double* W, int k, double* Y, int64_t ldy, const unsigned* cnt, unsigned cap, cudaStream_t st,
                     bool split_w) {
    const int q = q0 + q1;
    // W staged whole when it fits with the rows (kernel k_update_df64), else read by each
    // thread from L2 (k_update_df64_kt: passes of nt <= 512 columns, as even as multiples of 32
    // allow, one pass for k <= 512)
    const int kc0 = std::min(k, 256);
    const int ng = std::max(1, std::min(256 / kc0, 8));
    const int rows = ng * UR;
    const size_t smem_whole = ((size_t)rows * q + (size_t)q * k) * sizeof(float2);
    const bool whole = smem_whole <= 220 * 1024;
    const int npass = ceil_div(k, 512);
    const int nt = (int)round_up(ceil_div(k, npass), 32);
    const size_t smem = whole ? smem_whole : (size_t)UR * q * sizeof(float2);
    if (smem > 220 * 1024) return fail(HBSD_ERR_ARG, "update: q too large for the double-float kernel");
    {
        static std::mutex attr_mu;
        static size_t attr = 0;
        std::lock_guard<std::mutex> lk(attr_mu);
        if (smem > 48 * 1024 && smem > attr) {
            HBSD_CUDA(cudaFuncSetAttribute(k_update_df64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            HBSD_CUDA(cudaFuncSetAttribute(k_update_df64_kt, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
            attr = smem;
        }
    }
    HBSD_TRY(s->df_w.alloc((size_t)q * k));
    if (split_w) {
        const int64_t wcnt = (int64_t)q * k;
        k_split_w<<<ceil_div(wcnt, 256), 256, 0, st>>>(W, wcnt, s->df_w.p, cnt, cap);
        HBSD_LAUNCHED(s);
    }
    if (whole) k_update_df64<<<ceil_div(n, rows), 256, smem, st>>>(Z0, ld0, q0, Z1, ld1, q1, n, s->df_w.p, k, ng, Y, ldy, cnt, cap);
    else k_update_df64_kt<<<ceil_div(n, UR), nt, smem, st>>>(Z0, ld0, q0, Z1, ld1, q1, n, s->df_w.p, k, Y, ldy, cnt, cap);
    HBSD_LAUNCHED(s);
    return 0;
}

}  // namespace hbsd
