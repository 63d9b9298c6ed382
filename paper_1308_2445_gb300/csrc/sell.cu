// SELL-C-sigma storage of the shared (H, S) pattern and the fused block SpMM that produces
// H X and S X in one pass over the pattern (LABPSD steps 3 and 7; Sec. 4 footnote: H and S
// share one sparsity pattern, so one column index serves two values).
//
// Layout: rows are sorted by length (descending) inside windows of sigma rows, grouped into
// slices of C rows and padded to the slice's longest row.  Entry j of slot t of slice s is at
// slice_ptr[s] + j*C + t, so the C rows of a slice read their j-th entries from one contiguous
// segment.  Values are interleaved as (h - sigma0 s, s): one 16-byte (FP64) or 8-byte (FP32)
// load yields both.
//
// Block vectors are row-major, so the X-row that a nonzero needs is one contiguous vector.
// A row is handled by lpr lanes; each lane owns VW consecutive columns per pass (one 16-byte
// vector load), so the gather of an X row is coalesced and vectorised.
#include <algorithm>
#include <cmath>
#include <numeric>

#include "common.h"
#include "df64.h"

namespace hbsd {

// D = diag(S)^{-1/2} and its inverse, a warp per row (the last positive diagonal entry; 1 without one)
__global__ void __launch_bounds__(256) k_sell_dscale(int64_t n, const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ col_idx,
                                                     const double* __restrict__ sval, double* __restrict__ dscale,
                                                     double* __restrict__ dinv) {
    const int64_t r = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (r >= n) return;
    const int64_t e0 = row_ptr[r];
    const int len = (int)(row_ptr[r + 1] - e0);
    int last = -1;
    for (int j = lane; j < len; j += 32)
        if (col_idx[e0 + j] == r && sval[e0 + j] > 0.0) last = j;
    last = __reduce_max_sync(0xffffffffu, last);
    if (lane == 0) {
        const double d = last >= 0 ? __ddiv_rn(1.0, __dsqrt_rn(sval[e0 + last])) : 1.0;
        dscale[r] = d;
        dinv[r] = __ddiv_rn(1.0, d);
    }
}

// A warp per slice, lanes over consecutive stored positions (8 rows x 4 entries at C = 8, so that the CSR reads
// are whole sectors): column indices and S values; padding repeats the row's last column with zeros.
__global__ void __launch_bounds__(256) k_sell_pattern(int64_t n_slices, int C, const int64_t* __restrict__ slice_ptr,
                                                      const int32_t* __restrict__ slot_row, const int64_t* __restrict__ row_ptr,
                                                      const int32_t* __restrict__ col_idx, const double* __restrict__ sval,
                                                      int32_t* __restrict__ cols, double2* __restrict__ hs) {
    const int64_t sl = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (sl >= n_slices) return;
    const int64_t base = slice_ptr[sl];
    const int count = (int)(slice_ptr[sl + 1] - base);
    for (int i = threadIdx.x & 31; i < count; i += 32) {
        const int j = i / C, r = slot_row[sl * C + i - j * C];
        int col = 0;
        double s = 0.0;
        if (r >= 0) {
            const int64_t e0 = row_ptr[r], e1 = row_ptr[r + 1];
            if (e0 + j < e1) {
                col = col_idx[e0 + j];
                s = sval[e0 + j];
            } else if (e1 > e0) {
                col = col_idx[e1 - 1];
            }
        }
        cols[base + i] = col;
        hs[base + i] = make_double2(0.0, s);
    }
}

// The H values in the same way, with the scaled pencil (D Hs D, D S D) in FP32 for the FP32 step entry points (FP32
// works only on this pencil: the unscaled basis spans ~30 orders of magnitude) and as float pairs, the nearest
// float and the nearest float to the remainder.  On the host this took 21 ms per matrix of 2.95 M entries, the copies
// of the finished arrays included; here the copy of the CSR values is most of it.
__global__ void __launch_bounds__(256) k_sell_values(int64_t n_slices, int C, const int64_t* __restrict__ slice_ptr,
                                                     const int32_t* __restrict__ slot_row, const int64_t* __restrict__ row_ptr,
                                                     const double* __restrict__ hval, double sigma0, const int32_t* __restrict__ cols,
                                                     const double* __restrict__ dscale, double2* __restrict__ hs,
                                                     float2* __restrict__ hs32, float4* __restrict__ hsdf) {
    const int64_t sl = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (sl >= n_slices) return;
    const int64_t base = slice_ptr[sl];
    const int count = (int)(slice_ptr[sl + 1] - base);
    for (int i = threadIdx.x & 31; i < count; i += 32) {
        const int j = i / C, r = slot_row[sl * C + i - j * C];
        const int64_t p = base + i;
        const int64_t e = r >= 0 ? row_ptr[r] + j : 0;
        if (r < 0 || e >= row_ptr[r + 1]) {
            hs32[p] = make_float2(0.f, 0.f);
            hsdf[p] = make_float4(0.f, 0.f, 0.f, 0.f);
            continue;
        }
        const double s = hs[p].y, h = fma(-sigma0, s, hval[e]), f = __dmul_rn(dscale[r], dscale[cols[p]]);
        const double fh = __dmul_rn(f, h), fs = __dmul_rn(f, s);
        const float h0 = (float)fh, s0 = (float)fs;
        hs[p] = make_double2(h, s);
        hs32[p] = make_float2(h0, s0);
        hsdf[p] = make_float4(h0, (float)(fh - (double)h0), s0, (float)(fs - (double)s0));
    }
}

int sell_build(Sell& m, int64_t n, const int64_t* row_ptr, const int32_t* col_idx,
               const double* hval, const double* sval, double sigma0) {
    const int C = m.C;
    const int sigma = m.sigma;
    m.n = n;
    m.nnz = row_ptr[n];
    std::vector<int32_t> order(n);
    std::iota(order.begin(), order.end(), 0);
    for (int64_t w0 = 0; w0 < n; w0 += sigma) {
        int64_t w1 = std::min<int64_t>(n, w0 + sigma);
        std::stable_sort(order.begin() + w0, order.begin() + w1, [&](int32_t a, int32_t b) {
            return (row_ptr[a + 1] - row_ptr[a]) > (row_ptr[b + 1] - row_ptr[b]);
        });
    }
    m.n_slots = round_up(n, C);
    m.n_slices = m.n_slots / C;
    std::vector<int32_t> slot_row(m.n_slots, -1);
    for (int64_t i = 0; i < n; ++i) slot_row[i] = order[i];
    std::vector<int64_t> sptr(m.n_slices + 1, 0);
    std::vector<int32_t> slen(m.n_slices, 0);
    for (int64_t s = 0; s < m.n_slices; ++s) {
        int64_t mx = 0;
        for (int t = 0; t < C; ++t) {
            int32_t r = slot_row[s * C + t];
            if (r >= 0) mx = std::max<int64_t>(mx, row_ptr[r + 1] - row_ptr[r]);
        }
        slen[s] = (int32_t)mx;
        sptr[s + 1] = sptr[s] + mx * C;
    }
    m.stored = sptr[m.n_slices];
    m.h_slice_ptr = sptr;
    m.h_slot_row = slot_row;
    HBSD_TRY(m.slice_ptr.alloc(m.n_slices + 1));
    HBSD_TRY(m.slice_len.alloc(m.n_slices));
    HBSD_TRY(m.cols.alloc(m.stored));
    HBSD_TRY(m.hs.alloc(m.stored));
    HBSD_TRY(m.hs32.alloc(m.stored));
    HBSD_TRY(m.hsdf.alloc(m.stored));
    HBSD_TRY(m.slot_row.alloc(m.n_slots));
    HBSD_TRY(m.row_ptr.alloc(n + 1));
    HBSD_TRY(m.val.alloc(m.nnz));
    HBSD_TRY(m.dscale.alloc(n));
    HBSD_TRY(m.dinv.alloc(n));
    HBSD_CUDA(cudaMemcpy(m.slice_ptr.p, sptr.data(), sptr.size() * 8, cudaMemcpyHostToDevice));
    HBSD_CUDA(cudaMemcpy(m.slice_len.p, slen.data(), slen.size() * 4, cudaMemcpyHostToDevice));
    HBSD_CUDA(cudaMemcpy(m.slot_row.p, slot_row.data(), slot_row.size() * 4, cudaMemcpyHostToDevice));
    HBSD_CUDA(cudaMemcpy(m.row_ptr.p, row_ptr, (n + 1) * 8, cudaMemcpyHostToDevice));
    int32_t* ci = reinterpret_cast<int32_t*>(m.hsdf.p);   // until the values are filled in
    HBSD_CUDA(cudaMemcpy(ci, col_idx, m.nnz * 4, cudaMemcpyHostToDevice));
    HBSD_CUDA(cudaMemcpy(m.val.p, sval, m.nnz * 8, cudaMemcpyHostToDevice));
    const int gs = ceil_div(m.n_slices, 8);
    k_sell_dscale<<<ceil_div(n, 8), 256>>>(n, m.row_ptr.p, ci, m.val.p, m.dscale.p, m.dinv.p);
    HBSD_LAUNCHED((Session*)nullptr);
    k_sell_pattern<<<gs, 256>>>(m.n_slices, m.C, m.slice_ptr.p, m.slot_row.p, m.row_ptr.p, ci, m.val.p, m.cols.p, m.hs.p);
    HBSD_LAUNCHED((Session*)nullptr);
    m.h_dscale.resize(n);
    HBSD_CUDA(cudaMemcpy(m.h_dscale.data(), m.dscale.p, n * 8, cudaMemcpyDeviceToHost));
    return sell_update_h(m, hval, sigma0);
}

// The stored H values from CSR values in host memory; S, the pattern and the scaling stay.  On the legacy default
// stream and complete on return, as the copies are.
int sell_update_h(Sell& m, const double* hval, double sigma0) {
    HBSD_CUDA(cudaMemcpy(m.val.p, hval, m.nnz * 8, cudaMemcpyHostToDevice));
    k_sell_values<<<ceil_div(m.n_slices, 8), 256>>>(m.n_slices, m.C, m.slice_ptr.p, m.slot_row.p, m.row_ptr.p, m.val.p, sigma0,
                                                    m.cols.p, m.dscale.p, m.hs.p, m.hs32.p, m.hsdf.p);
    HBSD_LAUNCHED((Session*)nullptr);
    HBSD_CUDA(cudaStreamSynchronize(cudaStreamLegacy));
    return 0;
}

// ---- kernels ------------------------------------------------------------------------
template <class T> struct VecOf;
template <> struct VecOf<double> { using V = double2; using P = double2; static constexpr int W = 2; };
template <> struct VecOf<float> { using V = float4; using P = float2; static constexpr int W = 4; };

template <class T>
__device__ __forceinline__ void vload(const T* p, T (&v)[VecOf<T>::W]);
template <>
__device__ __forceinline__ void vload<double>(const double* p, double (&v)[2]) {
    double2 t = __ldg(reinterpret_cast<const double2*>(p));
    v[0] = t.x; v[1] = t.y;
}
template <>
__device__ __forceinline__ void vload<float>(const float* p, float (&v)[4]) {
    float4 t = __ldg(reinterpret_cast<const float4*>(p));
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}

template <class T>
__device__ __forceinline__ void vstore(T* p, const T (&v)[VecOf<T>::W], int valid);
template <>
__device__ __forceinline__ void vstore<double>(double* p, const double (&v)[2], int valid) {
    if (valid >= 2) *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
    else if (valid == 1) p[0] = v[0];
}
template <>
__device__ __forceinline__ void vstore<float>(float* p, const float (&v)[4], int valid) {
    if (valid >= 4) *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    else for (int i = 0; i < valid; ++i) p[i] = v[i];
}

__device__ __forceinline__ void ldhs(const double2* hs, int64_t e, double& h, double& s) {
    double2 t = __ldg(hs + e);
    h = t.x; s = t.y;
}
__device__ __forceinline__ void ldhs(const float2* hs, int64_t e, float& h, float& s) {
    float2 t = __ldg(hs + e);
    h = t.x; s = t.y;
}

// MODE 0: pair (HX, SX).  MODE 1: shifted, Y = HX - e_j SX.  A row is worked by 1 << parts_log2 groups of
// 1 << lpr_log2 lanes of one warp, a lane one vector, a group every 1 << parts_log2-th entry; blockIdx.y counts
// passes of (1 << lpr_log2) vectors.
// Bound by the FP64 pipe (a multiply-add of a warp takes it 64 clocks, idle lanes included) and on small
// matrices by the chain of index and X loads.  One vector per lane: with up to four, 85 columns of the 32^3
// problem (47,620 rows, 62 entries each) took 1,042 us instead of 988, 64 columns of the 16^3 one 72 instead of 52.
template <class T, int MODE, bool SPLIT>
__global__ void __launch_bounds__(256) k_spmm(
    const int64_t* __restrict__ slice_ptr, const int32_t* __restrict__ slice_len,
    const int32_t* __restrict__ cols, const typename VecOf<T>::P* __restrict__ hs,
    const int32_t* __restrict__ slot_row, int64_t n_slots, int C, const T* __restrict__ X,
    int64_t ldx, int k, int lpr_log2, int parts_log2, T* __restrict__ Y0, int64_t ld0,
    T* __restrict__ Y1, int64_t ld1, const T* __restrict__ shifts) {
    constexpr int VW = VecOf<T>::W;
    const int lpr = 1 << lpr_log2, parts = SPLIT ? 1 << parts_log2 : 1, row_log2 = lpr_log2 + (SPLIT ? parts_log2 : 0);
    const int lane = threadIdx.x & (lpr - 1), part = SPLIT ? (threadIdx.x >> lpr_log2) & (parts - 1) : 0;
    const int64_t slot = (int64_t)blockIdx.x * (blockDim.x >> row_log2) + (threadIdx.x >> row_log2);
    const int cc = VW * ((int)blockIdx.y * lpr + lane);
    const bool on = slot < n_slots && cc < k;
    const int64_t sl = on ? slot / C : 0;
    const int64_t base = on ? slice_ptr[sl] + (slot - sl * C) : 0;
    const int len = on ? slice_len[sl] : 0;
    T ah[VW], as[VW];
#pragma unroll
    for (int v = 0; v < VW; ++v) { ah[v] = T(0); as[v] = T(0); }
#pragma unroll 4
    for (int j = part; j < len; j += parts) {
        const int64_t e = base + (int64_t)j * C;
        const int cj = __ldg(cols + e);
        T hv, sv, x[VW];
        ldhs(hs, e, hv, sv);
        vload<T>(X + (int64_t)cj * ldx + cc, x);
#pragma unroll
        for (int v = 0; v < VW; ++v) {
            ah[v] = fma(hv, x[v], ah[v]);
            as[v] = fma(sv, x[v], as[v]);
        }
    }
    for (int o = lpr; SPLIT && o < (1 << row_log2); o <<= 1) {
#pragma unroll
        for (int v = 0; v < VW; ++v) {
            ah[v] += __shfl_xor_sync(0xffffffffu, ah[v], o);
            as[v] += __shfl_xor_sync(0xffffffffu, as[v], o);
        }
    }
    const int row = on && part == 0 ? slot_row[slot] : -1;
    if (row < 0) return;
    const int valid = min(VW, k - cc);
    if (MODE == 0) {
        vstore<T>(Y0 + (int64_t)row * ld0 + cc, ah, valid);
        vstore<T>(Y1 + (int64_t)row * ld1 + cc, as, valid);
    } else {
        T y[VW];
#pragma unroll
        for (int v = 0; v < VW; ++v) {
            T ev = (cc + v < k) ? shifts[cc + v] : T(0);
            y[v] = ah[v] - ev * as[v];
        }
        vstore<T>(Y0 + (int64_t)row * ld0 + cc, y, valid);
    }
}

template <class T>
static const typename VecOf<T>::P* values_of(const Sell& m);
template <>
const double2* values_of<double>(const Sell& m) { return m.hs.p; }
template <>
const float2* values_of<float>(const Sell& m) { return m.hs32.p; }

constexpr int64_t SPMM_SPLIT_ROWS = 8192;   // rows x groups up to which FP64 rows are split

// most lanes per row: the autotuner's choice for the session, else 32
static int spmm_lanes(const Session* s) {
    const int v = s ? s->tune_spmm_lpr : 0;
    return (v == 4 || v == 8 || v == 16) ? v : 32;
}

static int ceil_log2(int v) {
    int g = 0;
    while ((1 << g) < v) ++g;
    return g;
}

// Small CTAs where large ones would leave SMs idle: 19 columns of the 16^3 problem 31 us with 64 threads, 39 with 256
// (FP32, bound by latencies alone, 25 and 21)
static int spmm_threads(int64_t n_slots, int row_log2, int passes) {
    return ceil_div(n_slots, 256 >> row_log2) * passes < 8 * 152 ? 64 : 256;
}

template <class T, int MODE>
static int spmm_launch(Session* s, const Sell& m, const T* X, int64_t ldx, int k, T* Y0, int64_t ld0,
                       T* Y1, int64_t ld1, const T* e, cudaStream_t st) {
    constexpr int VW = VecOf<T>::W;
    if (k <= 0) return 0;
    if ((ldx % VW) || (ld0 % VW) || (MODE == 0 && (ld1 % VW)))
        return fail(HBSD_ERR_ARG, "spmm: leading dimensions must be multiples of the vector width");
    // FP64 rows of a small matrix are split over 2 to 8 groups of lanes: 19 columns of the 8^3 problem (646 rows)
    // took 28.7 us on one group, its 38 (up to 77) entries one after another, and 11 us on 8.  By the matrix alone, so that a
    // column's sums do not depend on the block it is in; from 4,797 rows on (16^3) the pipe is busy without.
    int parts_log2 = 0;
    if (sizeof(T) == 8)
        while (parts_log2 < 3 && (m.n_slots << (parts_log2 + 1)) <= SPMM_SPLIT_ROWS) ++parts_log2;
    // lanes per row (4 or more, up to the session's limit) with the fewest idle over all passes, each pass worth half
    // a lane: 24 columns of the 32^3 problem 307 us in 3 passes of 4 lanes, 371 in one of 16; 85 columns 988 in 3
    // of 16, 1,335 in one of 32 with a second vector on every lane
    const int vecs = ceil_div(k, VW), lmax = std::min(ceil_log2(spmm_lanes(s)), 5 - parts_log2);
    int lg = std::min(lmax, ceil_log2(std::min(vecs, 4))), best = 0x7FFFFFFF;
    for (int g = lg; g <= lmax; ++g) {
        const int cost = ceil_div(vecs, 1 << g) * ((2 << g) + 1);
        if (cost <= best) { best = cost; lg = g; }
    }
    const int threads = sizeof(T) == 8 ? spmm_threads(m.n_slots, lg + parts_log2, ceil_div(vecs, 1 << lg)) : 256;
    const dim3 grid(ceil_div(m.n_slots, threads >> (lg + parts_log2)), ceil_div(vecs, 1 << lg));
    const auto kern = sizeof(T) == 8 && parts_log2 ? k_spmm<T, MODE, sizeof(T) == 8> : k_spmm<T, MODE, false>;
    kern<<<grid, threads, 0, st>>>(m.slice_ptr.p, m.slice_len.p, m.cols.p, values_of<T>(m), m.slot_row.p, m.n_slots, m.C,
                                   X, ldx, k, lg, parts_log2, Y0, ld0, Y1, ld1, e);
    HBSD_LAUNCHED(s);
    return 0;
}

// ---- double-float SpMM on the scaled pencil (mixed form) ------------------------------------------
// X2 = D^-1 X as double-float pairs (the FP64 scaling, then split_d's exact bit split), per two columns the two high
// parts and the two low parts: the packed operands of k_spmm_df64
__global__ void k_split_scaled(const double* __restrict__ X, int64_t ldx, int k, int64_t n,
                               const double* __restrict__ dinv, float4* __restrict__ X2, int pairs) {
    const int64_t total = n * pairs;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t / pairs;
        const int j = 2 * (int)(t - i * pairs);
        const double d = dinv[i];
        const float2 a = df::split_d(X[i * ldx + j] * d);
        const float2 b = j + 1 < k ? df::split_d(X[i * ldx + j + 1] * d) : make_float2(0.f, 0.f);
        X2[t] = make_float4(a.x, b.x, a.y, b.y);
    }
}

// Pair mode of k_spmm in double-float: per stored entry the (hi, lo) of D Hs D and of D S D, per column pair one
// float4 of X2.  Sums by df::dfma's steps on packed column pairs, renormalised every 8 entries; the row result is
// scaled back by D^-1 in FP64.
// Bound by the FP32 pipe (24 packed instructions, 48 pipe cycles of a warp, per entry and column pair: half of its cycles
// at 85 columns of the 32^3 problem) and the latency of the gathers.  Without the
// loads an entry ahead, and with scalar instructions, 85 columns of the 32^3 problem took 583 us (now 404); packed
// without them 517.
// nax = -ax; the product is kept negated, which saves negating it for its rounding error
__device__ __forceinline__ void dfma_packed(df::f32x2 ax, df::f32x2 nax, df::f32x2 ay, df::f32x2 bx, df::f32x2 by, df::f32x2& sh,
                                            df::f32x2& sl, df::f32x2 nz) {
    const df::f32x2 np = df::fma2(nax, bx, nz);   // minus the rounded product (df64.h: why not a multiplication)
    const df::f32x2 t = df::sub2(sh, np);
    const df::f32x2 bp = df::sub2(t, sh);
    df::f32x2 e = df::fma2(ax, bx, np);
    e = df::fma2(ax, by, e);
    e = df::fma2(ay, bx, e);
    const df::f32x2 err = df::sub2(df::sub2(sh, df::sub2(t, bp)), df::add2(np, bp));
    sl = df::add2(sl, df::add2(err, e));
    sh = t;
}

template <int CH>
__global__ void __launch_bounds__(256, CH <= 2 ? 3 : 2) k_spmm_df64(
    const int64_t* __restrict__ slice_ptr, const int32_t* __restrict__ slice_len, const int32_t* __restrict__ cols,
    const float4* __restrict__ hsdf, const int32_t* __restrict__ slot_row, int64_t n_slots, int C,
    const float4* __restrict__ X2, int pairs, int k, int lpr_log2, const double* __restrict__ dinv,
    double* __restrict__ Y0, int64_t ld0, double* __restrict__ Y1, int64_t ld1, df::f32x2 nz) {
    const int lpr = 1 << lpr_log2;
    const int lane = threadIdx.x & (lpr - 1);
    const int64_t slot = (int64_t)blockIdx.x * (blockDim.x >> lpr_log2) + (threadIdx.x >> lpr_log2);
    if (slot >= n_slots) return;
    const int64_t sl = slot / C;
    const int t = (int)(slot - sl * C);
    const int64_t base = slice_ptr[sl] + t;
    const int len = slice_len[sl];
    const int v0 = (int)blockIdx.y * lpr * CH + lane;
    df::f32x2 ah[CH][2], as[CH][2];   // [chunk][hi, lo] of two columns
#pragma unroll
    for (int c = 0; c < CH; ++c) ah[c][0] = ah[c][1] = as[c][0] = as[c][1] = 0;
    // entry j + 1's values and X vectors are loaded before entry j's sums, entry j + 2's index with them
    const float4* xv[CH];   // idle lanes repeat the last vector
#pragma unroll
    for (int c = 0; c < CH; ++c) xv[c] = X2 + min(v0 + c * lpr, pairs - 1);
    float4 hn = make_float4(0.f, 0.f, 0.f, 0.f), xn[CH];
    int64_t e = base;
    int cn = 0;
    if (len > 0) {
        hn = __ldg(hsdf + e);
        cn = __ldg(cols + e);
#pragma unroll
        for (int c = 0; c < CH; ++c) xn[c] = __ldg(xv[c] + (int64_t)cn * pairs);
        if (len > 1) cn = __ldg(cols + e + C);
    }
    for (int j = 0; j < len; ++j) {
        const float4 hv = hn;
        float4 x[CH];
#pragma unroll
        for (int c = 0; c < CH; ++c) x[c] = xn[c];
        e += C;
        if (j + 1 < len) {
            hn = __ldg(hsdf + e);
#pragma unroll
            for (int c = 0; c < CH; ++c) xn[c] = __ldg(xv[c] + (int64_t)cn * pairs);
            if (j + 2 < len) cn = __ldg(cols + e + C);
        }
        const df::f32x2 hx = df::pack2(hv.x, hv.x), hnx = df::pack2(-hv.x, -hv.x), hy = df::pack2(hv.y, hv.y);
        const df::f32x2 sx = df::pack2(hv.z, hv.z), snx = df::pack2(-hv.z, -hv.z), sy = df::pack2(hv.w, hv.w);
#pragma unroll
        for (int c = 0; c < CH; ++c) {
            const df::f32x2 bx = df::pack2(x[c].x, x[c].y), by = df::pack2(x[c].z, x[c].w);
            dfma_packed(hx, hnx, hy, bx, by, ah[c][0], ah[c][1], nz);
            dfma_packed(sx, snx, sy, bx, by, as[c][0], as[c][1], nz);
        }
        if ((j & 7) == 7) {
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                df::renorm2(ah[c][0], ah[c][1]);
                df::renorm2(as[c][0], as[c][1]);
            }
        }
    }
    const int row = slot_row[slot];
    if (row < 0) return;
    const double di = dinv[row];
#pragma unroll
    for (int c = 0; c < CH; ++c) {
        const int cc = 2 * (v0 + c * lpr);
        if (cc >= k) continue;
        float h0, h1, l0, l1, s0, s1, m0, m1;
        df::unpack2(ah[c][0], h0, h1);
        df::unpack2(ah[c][1], l0, l1);
        df::unpack2(as[c][0], s0, s1);
        df::unpack2(as[c][1], m0, m1);
        Y0[(int64_t)row * ld0 + cc] = df::to_d(h0, l0) * di;
        Y1[(int64_t)row * ld1 + cc] = df::to_d(s0, m0) * di;
        if (cc + 1 < k) {
            Y0[(int64_t)row * ld0 + cc + 1] = df::to_d(h1, l1) * di;
            Y1[(int64_t)row * ld1 + cc + 1] = df::to_d(s1, m1) * di;
        }
    }
}

int spmm_pair_df64(Session* s, const Sell& m, const double* X, int64_t ldx, int k, double* HX, int64_t ldhx,
                   double* SX, int64_t ldsx, cudaStream_t st) {
    if (k <= 0) return 0;
    const int pairs = ceil_div(k, 2);
    HBSD_TRY(s->x2.alloc((size_t)m.n * pairs));
    {
        const int g = (int)std::min<int64_t>(ceil_div(m.n * pairs, 256), 8192);
        k_split_scaled<<<g, 256, 0, st>>>(X, ldx, k, m.n, m.dinv.p, s->x2.p, pairs);
        HBSD_LAUNCHED(s);
    }
    // 4 lanes per row and up to 4 column pairs per lane, in as many passes as that takes (each worth one more pair):
    // 85 columns of the 32^3 problem 404 us in 3 passes of 4 x 4, 441 in one of 16 x 3, 552 in one of 16 x 2 and more;
    // 64 columns 279 us against 311 (16 x 2).  Few rows keep to 2 pairs: 64 columns of the 16^3 problem (4,796
    // rows) 33 us in 4 passes, 37 in 2
    const int lg = std::min(2, ceil_log2(pairs)), cmax = m.n_slots >= 152 * 128 ? 4 : 2;
    int ch = 1, best = 0x7FFFFFFF;
    for (int c = 1; c <= cmax; ++c) {
        const int cost = ceil_div(pairs, c << lg) * (c + 1);
        if (cost <= best) { best = cost; ch = c; }
    }
    const int threads = spmm_threads(m.n_slots, lg, ceil_div(pairs, ch << lg));
    const dim3 grid(ceil_div(m.n_slots, threads >> lg), ceil_div(pairs, ch << lg));
#define HBSD_SPMM_DF_CASE(CHV)                                                                                      \
    case CHV:                                                                                                       \
        k_spmm_df64<CHV><<<grid, threads, 0, st>>>(m.slice_ptr.p, m.slice_len.p, m.cols.p, m.hsdf.p, m.slot_row.p,      \
                                               m.n_slots, m.C, s->x2.p, pairs, k, lg, m.dinv.p, HX, ldhx, SX, ldsx, \
                                               df::NEG_ZERO2);                                                      \
        break;
    switch (ch) {
        HBSD_SPMM_DF_CASE(1)
        HBSD_SPMM_DF_CASE(2)
        HBSD_SPMM_DF_CASE(3)
        HBSD_SPMM_DF_CASE(4)
        default:
            return fail(HBSD_ERR_ARG, "spmm_df64: internal chunking error");
    }
#undef HBSD_SPMM_DF_CASE
    HBSD_LAUNCHED(s);
    return nl_apply_add<double>(s, X, ldx, k, HX, ldhx, st);
}

// Both add the nonlocal term F G F^T X of the session (Eq. fgf) to the H product.
template <class T>
int spmm_pair(Session* s, const Sell& m, const T* X, int64_t ldx, int k, T* HX, int64_t ldhx,
              T* SX, int64_t ldsx, cudaStream_t st) {
    HBSD_TRY((spmm_launch<T, 0>(s, m, X, ldx, k, HX, ldhx, SX, ldsx, nullptr, st)));
    return nl_apply_add<T>(s, X, ldx, k, HX, ldhx, st);
}

template <class T>
int spmm_shifted(Session* s, const Sell& m, const T* X, int64_t ldx, int k, const T* e, T* Y,
                 int64_t ldy, cudaStream_t st) {
    HBSD_TRY((spmm_launch<T, 1>(s, m, X, ldx, k, Y, ldy, nullptr, 0, e, st)));
    return nl_apply_add<T>(s, X, ldx, k, Y, ldy, st);
}

template int spmm_pair<double>(Session*, const Sell&, const double*, int64_t, int, double*, int64_t,
                               double*, int64_t, cudaStream_t);
template int spmm_pair<float>(Session*, const Sell&, const float*, int64_t, int, float*, int64_t,
                              float*, int64_t, cudaStream_t);
template int spmm_shifted<double>(Session*, const Sell&, const double*, int64_t, int, const double*,
                                  double*, int64_t, cudaStream_t);
template int spmm_shifted<float>(Session*, const Sell&, const float*, int64_t, int, const float*,
                                 float*, int64_t, cudaStream_t);

}  // namespace hbsd
