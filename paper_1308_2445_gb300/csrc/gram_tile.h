// The double-float Gram tile of k_gram_df64 (df64.cu) and, where its guard fails, of the tensor-core Gram
// (gram_tc.cu).
#pragma once
#include <stdint.h>

#include "df64.h"

namespace hbsd {

namespace df {
// a row-major block in two segments, Z = [Z0 Z1]
struct Seg2d {
    const double* p0;
    int64_t ld0;
    int q0;
    const double* p1;
    int64_t ld1;
    __device__ __forceinline__ double at(int64_t i, int c) const {
        return c < q0 ? p0[i * ld0 + c] : p1[i * ld1 + (c - q0)];
    }
    __device__ __forceinline__ const double* column(int c, int64_t& ld) const {   // first entry of column c
        ld = c < q0 ? ld0 : ld1;
        return c < q0 ? p0 + c : p1 + (c - q0);
    }
};
}  // namespace df

namespace {

// (hi, lo), lo <= hi, of the p-th entry of a packed lower triangle
__device__ __forceinline__ void tri_index(int p, int& hi, int& lo) {
    hi = (int)((sqrtf(8.0f * (float)p + 1.0f) - 1.0f) * 0.5f);
    while ((hi + 1) * (hi + 2) / 2 <= p) ++hi;
    while (hi * (hi + 1) / 2 > p) --hi;
    lo = p - hi * (hi + 1) / 2;
}

constexpr int GW = 32;          // widest output tile: 8 x 8 threads of 4 x 4 outputs, once for HZ and once for SZ
constexpr int GR = 4;           // rows per shared-memory stage
constexpr int GRENORM = 2;      // stages per renormalisation of the sums (8 rows)
constexpr int GFLUSH = 16;      // stages per FP64 flush (64 rows)
constexpr int GTHREADS = 128;
constexpr int GCTAS = 4;        // CTAs per SM (128 registers)
constexpr int GWAVES = 6;       // CTAs wanted, in waves of the whole GPU

// One row stage in shared memory, high and low parts apart: the Z columns twice over (one float
// pair per column, so that a packed operand is one aligned load), the HZ and SZ columns plain.
struct GStage {
    float2 zh[GR][GW], zl[GR][GW];
    float xh[2][GR][GW], xl[2][GR][GW];   // [0] HZ, [1] SZ
};

struct GramTile {
    __align__(16) GStage buf[2];
    double acc[16][GTHREADS];
};

// The tile of Z^T ZH (warps 0-1) and Z^T ZS (warps 2-3) at columns a0.. and b0.., 4 nb columns wide, over
// rows r0..r1; with diag only the 4 x 4 blocks on and above the diagonal.  out(m, a, b, value) takes the
// results (m = 0: ZH, 1: ZS; a, b < q).  Called by all GTHREADS threads; the caller synchronises before
// sm is used again.
template <class Out>
__device__ __forceinline__ void gram_df64_tile(GramTile& sm, const df::Seg2d& Z, const df::Seg2d& ZH, const df::Seg2d& ZS,
                                               int q, int a0, int b0, int nb, bool diag, int64_t r0, int64_t r1,
                                               df::f32x2 nz, Out&& out) {
    const int tid = threadIdx.x, tw = 4 * nb;
    // thread -> 4 x 4 outputs (ua, ub) of matrix m; on the diagonal only ua <= ub
    const int m = tid >> 6, t = tid & 63;
    int ua, ub;
    bool on;
    if (diag) {
        tri_index(t, ub, ua);
        on = ub < nb;
    } else {
        ua = t / nb;
        ub = t - ua * nb;
        on = ua < nb;
    }
    if (!on) ua = ub = 0;
    df::f32x2 sh[4][2], sl[4][2];   // [a][pair of b]
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 2; ++v) sh[u][v] = sl[u][v] = 0ull;
#pragma unroll
    for (int o = 0; o < 16; ++o) sm.acc[o][tid] = 0.0;
    // loads: column lc of the tile, row lr of the stage
    const int lc = tid & (GW - 1), lr = tid / GW;
    const bool lza = lc < tw && a0 + lc < q, lzb = lc < tw && b0 + lc < q;
    double rz, rh, rs;
    auto fetch = [&](int64_t i0) {
        const int64_t i = i0 + lr;
        const bool ok = i < r1;
        rz = ok && lza ? Z.at(i, a0 + lc) : 0.0;
        rh = ok && lzb ? ZH.at(i, b0 + lc) : 0.0;
        rs = ok && lzb ? ZS.at(i, b0 + lc) : 0.0;
    };
    fetch(r0);
    int stage = 0;
    for (int64_t i0 = r0; i0 < r1; i0 += GR, ++stage) {
        GStage& g = sm.buf[stage & 1];
        {
            const float2 z = df::split_d(rz), h = df::split_d(rh), s = df::split_d(rs);
            g.zh[lr][lc] = make_float2(z.x, z.x);
            g.zl[lr][lc] = make_float2(z.y, z.y);
            g.xh[0][lr][lc] = h.x;
            g.xl[0][lr][lc] = h.y;
            g.xh[1][lr][lc] = s.x;
            g.xl[1][lr][lc] = s.y;
        }
        __syncthreads();   // the other buffer's readers are past it too: one barrier per stage
        if (i0 + GR < r1) fetch(i0 + GR);
        if (on) {
#pragma unroll
            for (int rr = 0; rr < GR; ++rr) {
                const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(&g.xh[m][rr][4 * ub]);
                const ulonglong2 y = *reinterpret_cast<const ulonglong2*>(&g.xl[m][rr][4 * ub]);
#pragma unroll
                for (int u2 = 0; u2 < 2; ++u2) {
                    const ulonglong2 zx = *reinterpret_cast<const ulonglong2*>(&g.zh[rr][4 * ua + 2 * u2]);
                    const ulonglong2 zy = *reinterpret_cast<const ulonglong2*>(&g.zl[rr][4 * ua + 2 * u2]);
                    df::dfma2(zx.x, zy.x, x.x, y.x, sh[2 * u2][0], sl[2 * u2][0], nz);
                    df::dfma2(zx.x, zy.x, x.y, y.y, sh[2 * u2][1], sl[2 * u2][1], nz);
                    df::dfma2(zx.y, zy.y, x.x, y.x, sh[2 * u2 + 1][0], sl[2 * u2 + 1][0], nz);
                    df::dfma2(zx.y, zy.y, x.y, y.y, sh[2 * u2 + 1][1], sl[2 * u2 + 1][1], nz);
                }
            }
            const bool flush = (stage % GFLUSH) == GFLUSH - 1 || i0 + GR >= r1;
            if (flush || (stage % GRENORM) == GRENORM - 1) {
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int v = 0; v < 2; ++v) df::renorm2(sh[u][v], sl[u][v]);
            }
            if (flush) {
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int v = 0; v < 2; ++v) {
                        float x0, x1, y0, y1;
                        df::unpack2(sh[u][v], x0, x1);
                        df::unpack2(sl[u][v], y0, y1);
                        sm.acc[u * 4 + v * 2][tid] += df::widen(x0) + df::widen(y0);
                        sm.acc[u * 4 + v * 2 + 1][tid] += df::widen(x1) + df::widen(y1);
                        sh[u][v] = sl[u][v] = 0ull;
                    }
            }
        }
    }
    if (!on) return;
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int a = a0 + 4 * ua + u, b = b0 + 4 * ub + v;
            if (a < q && b < q) out(m, a, b, sm.acc[u * 4 + v][tid]);
        }
}

}  // namespace
}  // namespace hbsd
