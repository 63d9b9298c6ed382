// Block update of steps 10-11 on the tensor cores by exact digit slices (slices.h), with the accuracy of the
// double-float form checked entry by entry (mixed form: Z0(:, 0:k) := [Z0 Z1] W in place).
//
// Column c of Z and row c of W are scaled by 2^(e_c) and 2^(-e_c), e_c the exponent of the largest entry of W's
// row: the search directions are large where their coefficients are small.  Then each row of Z and each column
// of W is a 62-bit fixed point against its own largest entry, and an output is the sum of the digit products,
// as in the Gram (gram_tc.cu).  With P the product of the row's and the column's leading powers of two, that leaves
// about sqrt(q) 2^-60 P and at most 2^-56 P per 256 terms, within the double-float form's 2^-48 sum|z||w| wherever
// sum|z||w| >= sqrt(q) 2^-11 P (for errors that do not all go one way, as there).  k_tu_guard evaluates
// sum|z||w| for every output (FP16 magnitudes, one MMA per 16 columns and 256 outputs of a row) and lists the entries
// below that line -- rows of a search block span many decades, and on the 16^3 case 0.4 to 1% of the outputs are that
// far below their row's largest term -- which k_tu_fix computes in FP64.  When more than a sixteenth of a slab's
// entries fail, the slab is computed by the double-float kernels.
//
// The rows are worked off in slabs: results go to a scratch block, since the tiles of a row read all of it, and
// are copied over Z0 when the slab is done.  One slab of 19,456 rows with q = 538, k = 282: exponents 26 us, guard
// 103, digits and products 230, entries in FP64 14, copy 15.  All 334,272 rows: 6.93 ms, 22.65 with pairs.  Bound
// by cutting Z (once per 64 columns; 16 clocks of four warps per value) and, in the guard, by the latency of the
// loads of one CTA per SM; the digit products alone are 1.8 ms.
#include <algorithm>
#include <mutex>

#include "common.h"
#include "df64.h"
#include "slices.h"
#include "tc.h"

namespace hbsd {
namespace {

using namespace slices;

constexpr int TU_NS = 3;                             // stage buffers of the main kernel
constexpr int TU_STAGE = DIG * (A_SLICE + B_SLICE);
constexpr int TU_MTHREADS = 576;                     // main kernel: 8 warps reading the accumulators, 8 slicing, MMAs, copies
constexpr int TU_SLICERS = 256;                      // the same of the guard
constexpr int TU_THREADS = TU_SLICERS + 64;
constexpr int TU_OUT_LD = 17;                        // doubles per row of a warp's 32 x 16 outputs in shared memory
constexpr size_t TU_SMEM = (size_t)TU_NS * TU_STAGE + (size_t)8 * 32 * (TU_OUT_LD + 4) * 8 + 1024;
constexpr int64_t TU_WAVE = UPDATE_TC_WAVE;
static_assert(TU_WAVE == 152 * ROWS, "one tile per SM");
constexpr int64_t TU_SLAB_BYTES = 88 << 20;          // Z rows of a slab: they stay in L2 between the passes
constexpr int64_t TU_SLAB_ROWS = 65536;              // a list entry holds 16 bits of row
constexpr int TU_GUARD_NS = 4;                       // stage buffers of the guard
constexpr int TU_GUARD_STAGE = 2 * (A_SLICE + UPDATE_TC_MAX_K * 32);   // 32 columns of Z and W
constexpr size_t TU_GUARD_SMEM = TU_GUARD_NS * (size_t)TU_GUARD_STAGE + 1024;

// [Z0 Z1] padded to steps of 16 columns: step t < t0 is columns 16 t of Z0, the later ones of Z1
struct Steps {
    const double* Z0;
    int64_t ld0;
    int q0;
    const double* Z1;
    int64_t ld1;
    int q1;
    int t0, total;
    // column of W's row of padded index kp, or -1
    __device__ __forceinline__ int wrow(int kp) const {
        const int c = kp < 16 * t0 ? kp : kp - 16 * t0;
        return kp < 16 * t0 ? (c < q0 ? c : -1) : (c < q1 ? q0 + c : -1);
    }
};

// entries 4 quarter .. + 3 of row i in step t; pairs, aligned (the caller checked pointers and strides)
__device__ __forceinline__ void load4(const Steps& S, int64_t i, int t, int quarter, double (&x)[4]) {
    const bool first = t < S.t0;
    const int c = 16 * (first ? t : t - S.t0) + 4 * quarter, q = first ? S.q0 : S.q1;
    const double* p = (first ? S.Z0 + i * S.ld0 : S.Z1 + i * S.ld1) + c;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        double2 v = make_double2(0.0, 0.0);
        if (c + 2 * h + 1 < q) v = *reinterpret_cast<const double2*>(p + 2 * h);
        else if (c + 2 * h < q) v.x = p[2 * h];
        x[2 * h] = v.x;
        x[2 * h + 1] = v.y;
    }
}

// ek[kp] = exponent field of W's row kp (0: padding or zero row)
__global__ void __launch_bounds__(256) k_tu_wrow(Steps S, const double* __restrict__ W, int k, int* __restrict__ ek) {
    const int kp = (int)blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (kp >= 16 * S.total) return;
    const int r = S.wrow(kp);
    int e = 0;
    if (r >= 0)
        for (int j = lane; j < k; j += 32) e = max(e, exp_field(W[(int64_t)r * k + j]));
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) ek[kp] = e;
}

// cw[j] = max over W's rows of the exponent field of W(r, j) minus ek
__global__ void __launch_bounds__(256) k_tu_wcol(Steps S, const double* __restrict__ W, int k, const int* __restrict__ ek,
                                                 int* __restrict__ cw) {
    __shared__ int red[8][32];
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5, j = (int)blockIdx.x * 32 + lane;
    int e = (int)0x80808080;
    if (j < k)
        for (int kp = g; kp < 16 * S.total; kp += 8) {
            const int r = S.wrow(kp);
            const int x = r >= 0 ? exp_field(W[(int64_t)r * k + j]) : 0;
            if (x != 0) e = max(e, x == 2047 ? BAD_EXP : x - ek[kp]);
        }
    red[g][lane] = e;
    __syncthreads();
    if (g == 0) {
        for (int t = 1; t < 8; ++t) e = max(e, red[t][lane]);
        if (j < k) cw[j] = e;
    }
}

// Digit slices of W per (64-column tile, step), each 16 KB as the main kernel's stage wants them, and the guard
// magnitudes per step of all kp64 = 64 gridDim.x columns
__global__ void __launch_bounds__(128) k_tu_wslice(Steps S, const double* __restrict__ W, int k, const int* __restrict__ ek,
                                                   const int* __restrict__ cw, uint8_t* __restrict__ Wsl,
                                                   uint8_t* __restrict__ Wg) {
    const int nl = threadIdx.x & 63, half = threadIdx.x >> 6, t = (int)blockIdx.y, j = (int)blockIdx.x * COLS + nl;
    const int c = j < k ? cw[j] : 0;
    double x[8];
    int off[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int kp = 16 * t + 8 * half + i, r = S.wrow(kp);
        x[i] = j < k && r >= 0 ? W[(int64_t)r * k + j] : 0.0;
        off[i] = c + ek[kp];
    }
    const int64_t cell = (int64_t)blockIdx.x * S.total + t;
    slice8(x, off, Wsl + cell * (DIG * B_SLICE) + half * 128 + (nl >> 3) * 256 + (nl & 7) * 16, B_SLICE);
    slice8_guard(x, off, Wg + (int64_t)t * gridDim.x * B_SLICE + half * 128 + (j >> 3) * 256 + (j & 7) * 16);
}

// rowexp[r] = max over the columns of the exponent field of Z(r, c) plus ek, one warp per row of the slab
__global__ void __launch_bounds__(256) k_tu_rowexp(Steps S, int64_t rbase, int rows, const int* __restrict__ ek,
                                                   int* __restrict__ rowexp) {
    const int r = (int)blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (r >= rows) return;
    int e = (int)0x80808080;
    const double* z0 = S.Z0 + (rbase + r) * S.ld0;
#pragma unroll 8
    for (int c = lane; c < S.q0; c += 32) {
        const int x = exp_field(z0[c]);
        if (x != 0) e = max(e, x == 2047 ? BAD_EXP : x + ek[c]);
    }
    if (S.q1 > 0) {
        const double* z1 = S.Z1 + (rbase + r) * S.ld1;
#pragma unroll 8
        for (int c = lane; c < S.q1; c += 32) {
            const int x = exp_field(z1[c]);
            if (x != 0) e = max(e, x == 2047 ? BAD_EXP : x + ek[16 * S.t0 + c]);
        }
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) rowexp[r] = e;
}

// bytes of W's slices or magnitudes to a stage, completing full
__device__ __forceinline__ void bulk_copy(void* dst, const void* src, uint32_t bytes, uint64_t* full) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(tc::smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(tc::smem_u32(full))
                 : "memory");
}
__device__ __forceinline__ void expect_bytes(uint64_t* full, uint32_t bytes) {   // with this thread's arrival
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(tc::smem_u32(full)), "r"(bytes) : "memory");
}
// the first `copies` copies, one after another into NS stages, have landed: the CTA may leave its shared memory
template <int NS>
__device__ __forceinline__ void drain_copies(uint64_t (&full)[NS], int copies) {
    for (int i = 0; i < NS; ++i) {
        const int c = (copies - i + NS - 1) / NS;   // into stage i
        if (c > 0) (void)tc::mbar_wait(&full[i], (uint32_t)((c - 1) & 1), WAIT_NS);
    }
}

// One CTA: sum|z||w| of 128 rows and all outputs, 32 columns of Z per stage (warps 0-7 the magnitudes of Z, warp
// 9 those of W, warp 8 the MMAs).  Entries below the line, and those of rows and columns with a non-finite
// entry, go to list[2 ..] as row << 16 | column; list[0] counts them (entries beyond cap are only counted).  A
// wait that gives up leaves the whole slab to the double-float kernels (list[0] above cap).
__global__ void __launch_bounds__(TU_THREADS, 1) k_tu_guard(Steps S, int64_t rbase, int rows, int k, int kp64,
                                                            const int* __restrict__ ek, const int* __restrict__ cw,
                                                            const uint8_t* __restrict__ Wg, const int* __restrict__ rowexp,
                                                            unsigned* __restrict__ list, unsigned cap) {
    extern __shared__ __align__(1024) uint8_t tu_smem[];
    __shared__ __align__(8) uint64_t full[TU_GUARD_NS], wfull[TU_GUARD_NS], empty[TU_GUARD_NS], done, drain;
    __shared__ uint32_t tslot;
    __shared__ int s_fail;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int r0 = (int)blockIdx.x * ROWS;   // row in the slab
    uint8_t* base = tu_smem + ((1024 - (tc::smem_u32(tu_smem) & 1023)) & 1023);
    if (tid == 0) {
        for (int i = 0; i < TU_GUARD_NS; ++i) {
            tc::mbar_init(&full[i], TU_SLICERS / 32);
            tc::mbar_init(&wfull[i], 1);
            tc::mbar_init(&empty[i], 1);
        }
        tc::mbar_init(&done, 1);
        tc::mbar_init(&drain, 1);
        s_fail = 0;
    }
    if (warp == 0) tc::tmem_alloc(&tslot, 512);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tbase = tslot;
    const int pairs = (S.total + 1) / 2;
    if (warp == 9) {
        if (lane == 0) {
            int st = 0, p = 0;
            uint32_t ph = 1;
            for (; p < pairs; ++p) {
                if (!tc::mbar_wait(&empty[st], ph, WAIT_NS)) { s_fail = 1; break; }
                const int nt = min(2, S.total - 2 * p);
                expect_bytes(&wfull[st], (uint32_t)(nt * kp64 * 32));
                for (int h = 0; h < nt; ++h)
                    bulk_copy(base + st * TU_GUARD_STAGE + 2 * A_SLICE + h * UPDATE_TC_MAX_K * 32,
                              Wg + (int64_t)(2 * p + h) * kp64 * 32, (uint32_t)(kp64 * 32), &wfull[st]);
                if (++st == TU_GUARD_NS) { st = 0; ph ^= 1u; }
            }
            drain_copies(wfull, p);
        }
    } else if (warp == 8) {
        if (lane == 0) {
            int st = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (int p = 0; p < pairs; ++p) {
                ok = tc::mbar_wait(&full[st], ph, WAIT_NS) && tc::mbar_wait(&wfull[st], ph, WAIT_NS);
                if (!ok) break;
                tc::fence_after_sync();
                const int nt = min(2, S.total - 2 * p);
                for (int h = 0; h < nt; ++h) {
                    const uint64_t a = tc::smem_desc(tc::smem_u32(base + st * TU_GUARD_STAGE + h * A_SLICE), 128, 256);
                    for (int c = 0; c < kp64; c += 256) {
                        const uint64_t b = tc::smem_desc(
                            tc::smem_u32(base + st * TU_GUARD_STAGE + 2 * A_SLICE + h * UPDATE_TC_MAX_K * 32 + c * 32), 128, 256);
                        const uint32_t id = tc::idesc_f16_f32(ROWS, min(256, kp64 - c));
                        if (p == 0 && h == 0) mma<0>(tbase + c, a, b, id);
                        else mma<1>(tbase + c, a, b, id);
                    }
                }
                tc::mma_commit(&empty[st]);
                if (++st == TU_GUARD_NS) { st = 0; ph ^= 1u; }
            }
            if (ok) tc::mma_commit(&done);
            else s_fail = 1;
            tc::mma_drain(&drain, WAIT_NS);
        }
    } else {
        const int quarter = lane & 3, row8 = warp * 16 + (lane >> 2);
        int ce[2];
        bool on[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            on[u] = r0 + row8 + 8 * u < rows;
            ce[u] = on[u] ? rowexp[r0 + row8 + 8 * u] : 0;
        }
        double x[2][2][2][4];   // [stage parity][step of the pair][row][column]
        int4 e[2][2];
        auto fetch = [&](int p, double (&xs)[2][2][4], int4 (&es)[2]) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int t = 2 * p + h;
                if (t >= S.total) return;
                es[h] = __ldg(reinterpret_cast<const int4*>(ek + 16 * t + 4 * quarter));
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    if (on[u]) load4(S, rbase + r0 + row8 + 8 * u, t, quarter, xs[h][u]);
                    else xs[h][u][0] = xs[h][u][1] = xs[h][u][2] = xs[h][u][3] = 0.0;
                }
            }
        };
        fetch(0, x[0], e[0]);
        fetch(1, x[1], e[1]);
        int st = 0;
        uint32_t ph = 1;
        auto step = [&](int p, double (&xs)[2][2][4], int4 (&es)[2]) {
            tc::warp_wait(&empty[st], ph, WAIT_NS, &s_fail);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (2 * p + h >= S.total) break;
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const double(&v)[4] = xs[h][u];
                    const uint32_t w0 = guard16(v[0], ce[u] - es[h].x) | (guard16(v[1], ce[u] - es[h].y) << 16);
                    const uint32_t w1 = guard16(v[2], ce[u] - es[h].z) | (guard16(v[3], ce[u] - es[h].w) << 16);
                    *reinterpret_cast<uint2*>(base + st * TU_GUARD_STAGE + h * A_SLICE + (quarter >> 1) * 128 + (row8 >> 3) * 256 +
                                              u * 256 + (row8 & 7) * 16 + (quarter & 1) * 8) = make_uint2(w0, w1);
                }
            }
            tc::fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(&full[st]);
            fetch(p + 2, xs, es);
            if (++st == TU_GUARD_NS) { st = 0; ph ^= 1u; }
        };
        for (int p = 0; p < pairs; p += 2) {
            step(p, x[0], e[0]);
            if (p + 1 < pairs) step(p + 1, x[1], e[1]);
        }
        tc::warp_wait(&done, 0u, WAIT_NS, &s_fail);
        __syncwarp();
        tc::fence_after_sync();
        const int r = (warp & 3) * 32 + lane;
        const int er = r0 + r < rows ? rowexp[r0 + r] : (int)0x80808080;
        const float need = sqrtf((float)(S.q0 + S.q1)) * 0x1p-11f;   // in units of the leading powers of two
        const bool row_on = er != (int)0x80808080, row_bad = er == BAD_EXP;
        for (int c0 = (warp >> 2) * 8; c0 < kp64; c0 += 16) {
            uint32_t v[8];
            tmem_ld8(tbase + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0, v);
            asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const int j = c0 + c;
                const int w = j < k ? cw[j] : (int)0x80808080;
                // a zero row or column gives exact zeros -- unless the other holds a non-finite entry
                const bool fail = j < k && r0 + r < rows &&
                                  (row_bad || w == BAD_EXP || (row_on && w != (int)0x80808080 && !(__uint_as_float(v[c]) >= need)));
                const unsigned m = __ballot_sync(0xffffffffu, fail);
                if (m) {
                    unsigned pos = 0;
                    if (lane == 0) pos = atomicAdd(list, __popc(m));
                    pos = __shfl_sync(0xffffffffu, pos, 0) + __popc(m & ((1u << lane) - 1u));
                    if (fail && pos < cap) list[2 + pos] = ((unsigned)(r0 + r) << 16) | (unsigned)j;
                }
            }
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == 0) tc::tmem_dealloc(tbase, 512);
    if (tid == 0 && s_fail) atomicAdd(list, cap + 1);
}

// One CTA: 128 rows of Y, 64 columns after 64 columns.  Warps 8-15 cut Z (one thread: 4 columns of two rows per
// step), warp 17 copies the W slices, warp 16 issues the MMAs; every 16 steps, and at the end of a column tile,
// warps 0-7 fold the accumulators into 64-bit integers in registers (32 columns of a row per thread).  Cutting
// and folding by the same warps, in turn, took 270 us (8 warps) and 325 us (16 warps, fewer registers) instead of
// 230 us for 19,456 rows, q = 538, k = 282 (the MMAs alone: 105 us).
__global__ void __launch_bounds__(TU_MTHREADS, 1) k_update_tc(Steps S, int64_t rbase, int rows, int k, int jt,
                                                             const int* __restrict__ ek, const int* __restrict__ cw,
                                                             const uint8_t* __restrict__ Wsl, const int* __restrict__ rowexp,
                                                             double* __restrict__ Y, unsigned* __restrict__ list, unsigned cap) {
    extern __shared__ __align__(1024) uint8_t tu_smem[];
    __shared__ __align__(8) uint64_t full[TU_NS], wfull[TU_NS], empty[TU_NS], phasedone, accfree, drain;
    __shared__ uint32_t tslot;
    __shared__ int s_fail;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) s_fail = __ldcg(list) > cap;   // one reading for the CTA: another CTA's failure may raise it
    __syncthreads();
    if (s_fail) return;                          // the slab is left to the double-float kernels
    __syncthreads();
    const int r0 = (int)blockIdx.x * ROWS;
    uint8_t* base = tu_smem + ((1024 - (tc::smem_u32(tu_smem) & 1023)) & 1023);
    if (tid == 0) {
        for (int i = 0; i < TU_NS; ++i) {
            tc::mbar_init(&full[i], 8);
            tc::mbar_init(&wfull[i], 1);
            tc::mbar_init(&empty[i], 1);
        }
        tc::mbar_init(&phasedone, 1);
        tc::mbar_init(&accfree, 8);
        tc::mbar_init(&drain, 1);
    }
    if (warp == 0) tc::tmem_alloc(&tslot, 512);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tbase = tslot;
    const int total = S.total, nph = (total + FLUSH_STEPS - 1) / FLUSH_STEPS, all = jt * total;

    if (warp == 17) {   // ---- W slices: one bulk copy per step, in the order of the steps
        if (lane == 0) {
            int st = 0, v = 0;
            uint32_t ph = 1;
            for (; v < all; ++v) {
                if (!tc::mbar_wait(&empty[st], ph, WAIT_NS)) { s_fail = 1; break; }
                expect_bytes(&wfull[st], DIG * B_SLICE);
                bulk_copy(base + st * TU_STAGE + DIG * A_SLICE, Wsl + (int64_t)v * (DIG * B_SLICE), DIG * B_SLICE, &wfull[st]);
                if (++st == TU_NS) { st = 0; ph ^= 1u; }
            }
            drain_copies(wfull, v);
        }
    } else if (warp == 16) {   // ---- MMA issuer
        if (lane == 0) {
            bool ok = true;
            int st = 0;
            uint32_t ph = 0;
            for (int p = 0; ok && p < jt * nph; ++p) {
                const int steps = min(FLUSH_STEPS, total - (p % nph) * FLUSH_STEPS);
                if (p > 0) ok = tc::mbar_wait(&accfree, (uint32_t)((p - 1) & 1), WAIT_NS);
                for (int t = 0; ok && t < steps; ++t) {
                    ok = tc::mbar_wait(&full[st], ph, WAIT_NS) && tc::mbar_wait(&wfull[st], ph, WAIT_NS);
                    if (!ok) break;
                    tc::fence_after_sync();
                    const uint64_t a = tc::smem_desc(tc::smem_u32(base + st * TU_STAGE), 128, 256);
                    const uint64_t b = a + (uint64_t)((DIG * A_SLICE) >> 4);
                    if (t == 0) mma_window<0, 0>(tbase, a, b);
                    else mma_window<0, 1>(tbase, a, b);
                    mma_window<1, 1>(tbase, a, b);
                    mma_window<2, 1>(tbase, a, b);
                    mma_window<3, 1>(tbase, a, b);
                    mma_window<4, 1>(tbase, a, b);
                    mma_window<5, 1>(tbase, a, b);
                    mma_window<6, 1>(tbase, a, b);
                    mma_window<7, 1>(tbase, a, b);
                    tc::mma_commit(&empty[st]);
                    if (++st == TU_NS) { st = 0; ph ^= 1u; }
                }
                if (ok) tc::mma_commit(&phasedone);
            }
            if (!ok) s_fail = 1;
            tc::mma_drain(&drain, WAIT_NS);
        }
    } else if (warp < 8) {   // ---- the accumulators: 32 rows and 32 columns per warp, kept over the phases of a column tile
        const uint32_t taddr = tbase + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * 32);
        const int fr = r0 + (warp & 3) * 32 + lane;
        const int fer = fr < rows ? rowexp[fr] : 0;
        double* o = reinterpret_cast<double*>(base + TU_NS * TU_STAGE) + (int64_t)warp * 32 * TU_OUT_LD;
        // [8][32]: fractions of this row's 32 sums, four columns in a word (in registers they would spill)
        uint32_t* low = reinterpret_cast<uint32_t*>(base + TU_NS * TU_STAGE + 8 * 32 * TU_OUT_LD * 8) + warp * 256 + lane;
        int p = 0;
        for (int tile = 0; tile < jt; ++tile) {
            long long acc[32];
#pragma unroll
            for (int c = 0; c < 32; ++c) acc[c] = 0;
#pragma unroll
            for (int c = 0; c < 8; ++c) low[32 * c] = 0;
            for (int u = 0; u < nph; ++u, ++p) {
                tc::warp_wait(&phasedone, (uint32_t)(p & 1), WAIT_NS, &s_fail);
                __syncwarp();
                tc::fence_after_sync();
#pragma unroll
                for (int c0 = 0; c0 < 32; c0 += 4) {
                    uint32_t v[8][4];
#pragma unroll
                    for (int l = 0; l < 8; ++l) tmem_ld4(taddr + (uint32_t)(COLS * l + c0), v[l]);
                    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
                    uint32_t w = low[8 * c0];
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const uint32_t l[8] = {v[0][c], v[1][c], v[2][c], v[3][c], v[4][c], v[5][c], v[6][c], v[7][c]};
                        acc[c0 + c] += fold_levels(l, w, c);
                    }
                    low[8 * c0] = w;
                }
                tc::fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(&accfree);
            }
            // through shared memory, 16 columns of two rows per store
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int j0 = tile * COLS + (warp >> 2) * 32 + 16 * h;
#pragma unroll
                for (int c = 0; c < 16; ++c)
                    o[lane * TU_OUT_LD + c] =
                        j0 + c < k ? scaled_sum(acc[16 * h + c], low[32 * (4 * h + c / 4)], c & 3, fer + cw[j0 + c] - 2056 - FRAC) : 0.0;
                __syncwarp();
                const int oc = lane & 15;
                if (j0 + oc < k)
                    for (int r = lane >> 4; r < 32; r += 2) {
                        const int yr = r0 + (warp & 3) * 32 + r;
                        if (yr < rows) Y[(int64_t)yr * k + j0 + oc] = o[r * TU_OUT_LD + oc];
                    }
                __syncwarp();
            }
        }
    } else {   // ---- slicers: rows row8 and row8 + 8, four columns of each step
        const int quarter = lane & 3, row8 = (warp - 8) * 16 + (lane >> 2);
        bool on[2];
        int ce[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            on[u] = r0 + row8 + 8 * u < rows;
            ce[u] = on[u] ? rowexp[r0 + row8 + 8 * u] : 0;
        }
        const uint32_t soff = (uint32_t)((quarter >> 1) * 128 + (row8 >> 3) * 256 + (row8 & 7) * 16 + (quarter & 1) * 8);
        double x[2][2][4];   // [step parity][row][column]
        int4 e[2];
        int ft = 0;          // step in the column tile of the next fetch
        auto fetch = [&](double (&xs)[2][4], int4& es) {   // past the last step: harmless loads of the first ones
            es = __ldg(reinterpret_cast<const int4*>(ek + 16 * ft + 4 * quarter));
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                if (on[u]) load4(S, rbase + r0 + row8 + 8 * u, ft, quarter, xs[u]);
                else xs[u][0] = xs[u][1] = xs[u][2] = xs[u][3] = 0.0;
            }
            if (++ft == total) ft = 0;
        };
        fetch(x[0], e[0]);
        fetch(x[1], e[1]);
        int st = 0;
        uint32_t ph = 1;
        auto step = [&](double (&xs)[2][4], int4& es) {
            tc::warp_wait(&empty[st], ph, WAIT_NS, &s_fail);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                uint8_t* dst = base + st * TU_STAGE + soff + u * 256;
                const int off[4] = {ce[u] - es.x, ce[u] - es.y, ce[u] - es.z, ce[u] - es.w};
                unsigned long long w[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) w[c] = fixed62(xs[u][c], off[c]);
                uint32_t sg[2], csg[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    sg[h] = signs2(xs[u][2 * h], xs[u][2 * h + 1]);
                    asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(csg[h]) : "r"(sg[h]), "r"(0xE480E480u));
                }
#pragma unroll
                for (int s = 0; s < DIG; ++s) {
                    uint32_t d[2];
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        d[h] = digits2(w[2 * h], w[2 * h + 1], s, sg[h], csg[h]);
                    *reinterpret_cast<uint2*>(dst + s * A_SLICE) = make_uint2(d[0], d[1]);
                }
            }
            tc::fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(&full[st]);
            fetch(xs, es);
            if (++st == TU_NS) { st = 0; ph ^= 1u; }
        };
        for (int v = 0; v < all; v += 2) {
            step(x[0], e[0]);
            if (v + 1 < all) step(x[1], e[1]);
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == 0) tc::tmem_dealloc(tbase, 512);
    if (tid == 0 && s_fail) atomicAdd(list, cap + 1);   // a wait gave up: the double-float kernels recompute the slab
}

// The listed entries in FP64, one warp each
__global__ void __launch_bounds__(256) k_tu_fix(Steps S, int64_t rbase, const double* __restrict__ W, int k, double* __restrict__ Y,
                                                const unsigned* __restrict__ list, unsigned cap) {
    const unsigned cnt = list[0];
    if (cnt > cap) return;
    const int lane = threadIdx.x & 31;
    for (unsigned w = blockIdx.x * 8 + (threadIdx.x >> 5); w < cnt; w += gridDim.x * 8) {
        const unsigned code = list[2 + w], r = code >> 16, j = code & 0xFFFFu;
        const double* z0 = S.Z0 + (rbase + r) * S.ld0;
        double s = 0.0;
        for (int c = lane; c < S.q0; c += 32) s = fma(z0[c], W[(int64_t)c * k + j], s);
        if (S.q1 > 0) {
            const double* z1 = S.Z1 + (rbase + r) * S.ld1;
            for (int c = lane; c < S.q1; c += 32) s = fma(z1[c], W[(int64_t)(S.q0 + c) * k + j], s);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) Y[(int64_t)r * k + j] = s;
    }
}

__global__ void __launch_bounds__(256) k_tu_copy(const double* __restrict__ Y, int k, int64_t rows, double* __restrict__ Z,
                                                 int64_t ld) {
    const int64_t total = rows * k;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = t / k;
        Z[i * ld + (t - i * k)] = Y[t];
    }
}

}  // namespace

bool update_tc_fits(const double* Z0, int64_t ld0, const double* Z1, int64_t ld1, int q1, int k) {
    auto ok = [](const double* p, int64_t ld) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && (ld & 1) == 0; };
    return k <= UPDATE_TC_MAX_K && ok(Z0, ld0) && (q1 == 0 || ok(Z1, ld1));
}

// slabs of whole waves whose Z rows stay in L2 from one pass to the next
struct TuPlan {
    int64_t slab;
    unsigned cap;                // entries of the list
    size_t y_b, sl_b, g_b;       // bytes of the workspace: results of a slab | slices of W | guard magnitudes of W
    size_t doubles;              // ... | exponents of rows, W's rows and columns | list
};
static TuPlan tu_plan(int64_t n, int q0, int q1, int k) {
    TuPlan p;
    const int total = ceil_div(q0, 16) + ceil_div(q1, 16), jt = ceil_div(k, COLS), kp64 = jt * COLS;
    const int64_t waves = std::max<int64_t>(1, std::min<int64_t>(TU_SLAB_BYTES / (TU_WAVE * (q0 + q1) * 8), TU_SLAB_ROWS / TU_WAVE));
    p.slab = std::min<int64_t>(waves * TU_WAVE, round_up(n, ROWS));
    p.cap = (unsigned)std::max<int64_t>(4096, p.slab * k / 16);
    auto kib = [](size_t b) { return (b + 1023) / 1024 * 1024; };
    p.y_b = kib((size_t)p.slab * k * 8);
    p.sl_b = kib((size_t)jt * total * DIG * B_SLICE);
    p.g_b = kib((size_t)total * kp64 * 32);
    const size_t ints = (size_t)p.slab + 16 * total + kp64 + 2 + p.cap;
    p.doubles = (p.y_b + p.sl_b + p.g_b + ints * 4 + 64) / 8 + 1;
    return p;
}
size_t update_tc_doubles(int64_t n, int q0, int q1, int k) { return tu_plan(n, q0, q1, k).doubles; }

int update2_tc(Session* s, double* Z0, int64_t ld0, int q0, const double* Z1, int64_t ld1, int q1, int64_t n, const double* W,
               int k, cudaStream_t st) {
    Steps S{Z0, ld0, q0, Z1, ld1, q1, ceil_div(q0, 16), 0};
    S.total = S.t0 + ceil_div(q1, 16);
    const int jt = ceil_div(k, COLS), kp64 = jt * COLS;
    const TuPlan p = tu_plan(n, q0, q1, k);
    const int64_t slab = p.slab;
    const unsigned cap = p.cap;
    HBSD_TRY(s->df_ws.alloc(p.doubles));
    uint8_t* ws = reinterpret_cast<uint8_t*>(s->df_ws.p);
    double* Y = reinterpret_cast<double*>(ws);
    uint8_t* Wsl = ws + p.y_b;
    uint8_t* Wg = Wsl + p.sl_b;
    int* ek = reinterpret_cast<int*>(Wg + p.g_b);          // 16-byte aligned, a multiple of 16 entries
    int* rowexp = ek + 16 * S.total;
    int* cw = rowexp + slab;
    unsigned* list = reinterpret_cast<unsigned*>(cw + kp64);
    static std::once_flag once;
    static cudaError_t attr = cudaSuccess;
    std::call_once(once, [] {
        attr = cudaFuncSetAttribute(k_update_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TU_SMEM);
        if (attr == cudaSuccess)
            attr = cudaFuncSetAttribute(k_tu_guard, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TU_GUARD_SMEM);
    });
    HBSD_CUDA(attr);
    k_tu_wrow<<<ceil_div(16 * S.total, 8), 256, 0, st>>>(S, W, k, ek);
    HBSD_LAUNCHED(s);
    k_tu_wcol<<<ceil_div(k, 32), 256, 0, st>>>(S, W, k, ek, cw);
    HBSD_LAUNCHED(s);
    k_tu_wslice<<<dim3(jt, S.total), 128, 0, st>>>(S, W, k, ek, cw, Wsl, Wg);
    HBSD_LAUNCHED(s);
    for (int64_t b = 0; b < n; b += slab) {
        const int rows = (int)std::min<int64_t>(slab, n - b), tiles = ceil_div(rows, ROWS);
        HBSD_CUDA(cudaMemsetAsync(list, 0, 2 * sizeof(unsigned), st));
        k_tu_rowexp<<<ceil_div(rows, 8), 256, 0, st>>>(S, b, rows, ek, rowexp);
        HBSD_LAUNCHED(s);
        k_tu_guard<<<tiles, TU_THREADS, TU_GUARD_SMEM, st>>>(S, b, rows, k, kp64, ek, cw, Wg, rowexp, list, cap);
        HBSD_LAUNCHED(s);
        k_update_tc<<<tiles, TU_MTHREADS, TU_SMEM, st>>>(S, b, rows, k, jt, ek, cw, Wsl, rowexp, Y, list, cap);
        HBSD_LAUNCHED(s);
        k_tu_fix<<<152 * 8, 256, 0, st>>>(S, b, W, k, Y, list, cap);
        HBSD_LAUNCHED(s);
        HBSD_TRY(update_df64_rows(s, Z0 + b * ld0, ld0, q0, q1 ? Z1 + b * ld1 : Z1, ld1, q1, rows, W, k, Y, k, list, cap, st));
        k_tu_copy<<<(int)std::min<int64_t>(152 * 16, ceil_div((int64_t)rows * k, 256)), 256, 0, st>>>(Y, k, rows, Z0 + b * ld0, ld0);
        HBSD_LAUNCHED(s);
    }
    return 0;
}

}  // namespace hbsd
