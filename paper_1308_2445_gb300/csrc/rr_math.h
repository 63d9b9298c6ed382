// Pieces shared by the Rayleigh-Ritz kernels (rr.cu, rr_grid.cu): warp sums, the reciprocal, sorting keys and
// the eigenvectors of the tridiagonal matrix.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <cfloat>
#include <cmath>

namespace hbsd {
namespace rrm {

__device__ __forceinline__ double wsum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Squares of a reflector's entries below this are zero: their reciprocal would not be finite.
constexpr double RR_TAIL_MIN = 0x1p-1000;

// magnitude of a double as an integer that orders like it
__device__ __forceinline__ unsigned long long mag(double x) {
    return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}

// 1/d: the FP32 reciprocal of the leading 24 bits (relative error below 2^-21), then one third-order step
// r (1 + e + e^2), e = 1 - d r, whose error e^3 is below the last bit.  The conversions are integer
// operations: an FP64 instruction takes the unit of an SM sub-partition 64 clocks, a conversion included.
// Operands outside 2^-100 .. 2^100 use the IEEE division.
__device__ __forceinline__ double rcp64(double d) {
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    const unsigned ex = (hi >> 20) & 0x7FFu;
    if (ex - 923u > 200u) return 1.0 / d;
    const float f = __uint_as_float((hi & 0x80000000u) | ((ex - 896u) << 23) | ((hi & 0xFFFFFu) << 3) | (lo >> 29));
    float rf;
    asm("rcp.approx.f32 %0, %1;" : "=f"(rf) : "f"(f));
    const unsigned b = __float_as_uint(rf);
    const double r = __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7FFFFFFFu) >> 3) + 0x38000000u)), (int)(b << 29));
    const double e = fma(-d, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

// order-preserving integer key of a double (sorting on the integer pipe)
__device__ __forceinline__ unsigned long long dkey(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

// (a, b), b <= a, of the p-th entry of a packed lower triangle
__device__ __forceinline__ void tri_index(int p, int& a, int& b) {
    a = (int)((sqrtf(8.0f * (float)p + 1.0f) - 1.0f) * 0.5f);
    while ((a + 1) * (a + 2) / 2 <= p) ++a;
    while (a * (a + 1) / 2 > p) --a;
    b = p - a * (a + 1) / 2;
}

// Eigenvector j of T (diagonal dd, off-diagonal ee) by one warp: inverse iteration at the coarse eigenvalue
// lam[j] from a fixed pseudo-random start, then solves at the Rayleigh quotient theta = x^T T x.  Pivoted
// tridiagonal LU with reciprocal pivots, sequential on lane 0; pivots below eps ||T|| are raised to it, so
// that a shift on an eigenvalue amplifies the wanted direction by about 1/eps instead of overflowing.
// ee[q - 1] must be 0.  scr: 4 q doubles; store(x) is called by the whole warp with every accepted vector; *th_out: the last shift.
// Returns the number of solves after the first (0: the second failed).
template <class Store>
__device__ __forceinline__ int tri_eigenvector(const double* dd, const double* ee, int q, int k, int j, const double* lam,
                                               double tnorm, double pivmin, double* scr, int lane, Store&& store,
                                               double* th_out) {
    double* fdv = scr;             // reciprocals of the U diagonal; T's shifted diagonal before
    double* fuv = scr + q;         // first super-diagonal
    double* fu2v = scr + 2 * q;    // second super-diagonal
    double* x = scr + 3 * q;       // iterate
    const double ptd = fmax(DBL_EPSILON * tnorm, pivmin);
    const unsigned long long ptdm = mag(ptd);
    auto floor_piv = [&](double d) { return mag(d) < ptdm ? copysign(ptd, d) : d; };
    // x <- (T - sh I)^{-1} x.  Factorisation and forward substitution in one sweep on lane 0 (six FP64
    // instructions per row), the scaling by the reciprocals on all lanes, the backward sweep on lane 0 (two).
    auto solve64 = [&](double sh) {
        for (int i = lane; i < q; i += 32) fdv[i] = dd[i] - sh;
        __syncwarp();
        if (lane == 0) {
            double di = fdv[0], ui = ee[0], xi = x[0];
            for (int i = 0; i + 1 < q; ++i) {
                const double sub = ee[i], dn = fdv[i + 1], un = ee[i + 1], xn = x[i + 1];   // ee[q - 1] = 0
                if (mag(di) >= mag(sub)) {
                    const double ri = rcp64(floor_piv(di));
                    const double f = sub * ri;
                    fdv[i] = ri;
                    fuv[i] = ui;
                    fu2v[i] = 0.0;
                    x[i] = xi;
                    di = fma(-f, ui, dn);
                    xi = fma(-f, xi, xn);
                    ui = un;
                } else {
                    const double ri = rcp64(floor_piv(sub));
                    const double f = di * ri;
                    fdv[i] = ri;
                    fuv[i] = dn;
                    fu2v[i] = un;
                    x[i] = xn;
                    di = fma(-f, dn, ui);
                    xi = fma(-f, xn, xi);
                    ui = -f * un;
                }
            }
            fdv[q - 1] = rcp64(floor_piv(di));
            fuv[q - 1] = fu2v[q - 1] = 0.0;
            x[q - 1] = xi;
        }
        __syncwarp();
        for (int i = lane; i < q; i += 32) {
            const double r = fdv[i];
            fuv[i] *= r;
            fu2v[i] *= r;
            x[i] *= r;
        }
        __syncwarp();
        if (lane == 0) {
            double x1 = 0.0, x2 = 0.0;
            for (int i = q - 1; i >= 0; --i) {
                const double v = fma(-fuv[i], x1, fma(-fu2v[i], x2, x[i]));
                x[i] = v;
                x2 = x1;
                x1 = v;
            }
        }
        __syncwarp();
    };
    // x / ||x||; false (x untouched) when an entry of x is not finite or x is zero
    // (fmax drops NaN, so the entries are tested one by one)
    auto normalise = [&]() {
        double mx = 0.0;
        bool bad = false;
        for (int i = lane; i < q; i += 32) {
            bad |= !isfinite(x[i]);
            mx = fmax(mx, fabs(x[i]));
        }
        if (__any_sync(0xffffffffu, bad)) return false;
        for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (!(mx > 0.0 && isfinite(mx))) return false;
        const double sc = 1.0 / mx;
        double n2 = 0.0;
        for (int i = lane; i < q; i += 32) { x[i] *= sc; n2 = fma(x[i], x[i], n2); }
        const double inr = rsqrt(wsum(n2));
        for (int i = lane; i < q; i += 32) x[i] *= inr;
        __syncwarp();
        return true;
    };
    for (int i = lane; i < q; i += 32) {
        uint64_t h = 0x9E3779B97F4A7C15ull * (uint64_t)(j + 1) + 0xBF58476D1CE4E5B9ull * (uint64_t)(i + 1);
        h ^= h >> 31;
        h *= 0x94D049BB133111EBull;
        h ^= h >> 29;
        x[i] = 0.5 + (double)(h >> 11) * (1.0 / 9007199254740992.0);
    }
    __syncwarp();
    solve64(lam[j]);
    normalise();
    store(x);   // kept if the next solve fails
    double th = 0.0;
    for (int i = lane; i < q; i += 32) {
        th = fma(dd[i] * x[i], x[i], th);
        if (i + 1 < q) th = fma(2.0 * ee[i] * x[i], x[i + 1], th);
    }
    th = wsum(th);
    __syncwarp();
    solve64(th);
    bool ok2 = normalise();
    if (ok2)
        store(x);
    // Rayleigh-quotient iteration until the residual ||T x - theta x|| is below
    // 1e-12 ||T|| (a start vector nearly orthogonal to the wanted eigenvector leaves a
    // neighbour's component after the first solve): at most three more solves
    // only for a separated eigenvalue: inside a cluster narrower than 1e-6 ||T|| further
    // solves would pull several vectors onto one eigenvector, while the mixing they
    // remove there costs almost nothing (it is weighted by the cluster width).  A vector
    // is accepted only while its quotient stays in eigenvalue j's interval (midpoints to
    // the neighbouring coarse eigenvalues): unguarded, the iteration can settle on a
    // neighbour and duplicate its vector.
    double gapj = DBL_MAX;
    if (j > 0) gapj = fmin(gapj, fabs(lam[j] - lam[j - 1]));
    if (j + 1 < k) gapj = fmin(gapj, fabs(lam[j + 1] - lam[j]));
    const bool separated = gapj > 1e-6 * tnorm;
    const double lo_j = j > 0 ? 0.5 * (lam[j - 1] + lam[j]) : -DBL_MAX;
    const double hi_j = j + 1 < k ? 0.5 * (lam[j] + lam[j + 1]) : DBL_MAX;
    auto rayleigh = [&]() {
        double t2 = 0.0;
        for (int i = lane; i < q; i += 32) {
            t2 = fma(dd[i] * x[i], x[i], t2);
            if (i + 1 < q) t2 = fma(2.0 * ee[i] * x[i], x[i + 1], t2);
        }
        return wsum(t2);
    };
    int extra = 0;
    if (ok2 && separated) {
        double th2 = rayleigh();
        while (extra < 3 && th2 >= lo_j && th2 <= hi_j) {
            double r2 = 0.0;
            for (int i = lane; i < q; i += 32) {
                double ti = fma(dd[i] - th2, x[i], 0.0);
                if (i > 0) ti = fma(ee[i - 1], x[i - 1], ti);
                if (i + 1 < q) ti = fma(ee[i], x[i + 1], ti);
                r2 = fma(ti, ti, r2);
            }
            r2 = wsum(r2);
            __syncwarp();
            th = th2;
            if (r2 <= (1e-12 * tnorm) * (1e-12 * tnorm)) break;   // far below what the caller resolves
            solve64(th);
            ++extra;
            if (!normalise()) break;               // store keeps the last accepted vector
            th2 = rayleigh();
            __syncwarp();
            if (th2 < lo_j || th2 > hi_j) break;   // left the interval: rejected
            store(x);
            __syncwarp();
        }
    }
    *th_out = th;
    return ok2 ? 1 + extra : 0;
}

}  // namespace rrm
}  // namespace hbsd
