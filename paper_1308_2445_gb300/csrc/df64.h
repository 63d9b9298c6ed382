// Double-float arithmetic: a value as an unevaluated sum hi + lo of two floats (Dekker 1971;
// Knuth's TwoSum), for FP64-bound products on GB300's FP32 pipes (128 FP32 lanes per clock
// per SM against 2 FP64).
//
// split_d builds the pair without the FP64 pipe: hi = the FP64 value truncated to 24 bits, from
// its sign, exponent and top mantissa bits; lo = the remaining 29 mantissa bits converted by the
// integer-to-float unit and scaled by the exponent.  The pair carries ~47 bits for magnitudes
// above 2^-96; below that lo is an FP32 subnormal and the precision falls towards 24 bits, and
// magnitudes below 2^-126 enter as zero.  dfma adds the product of two pairs (TwoProd by FMA
// for hi*hi plus the two cross terms) to a running pair by TwoSum; renorm restores |lo| <= ulp(hi)/2.
// The _rn intrinsics are never contracted into FMAs, which would break the error-free steps.
#pragma once
#include <cuda_runtime.h>

namespace hbsd {
namespace df {

__device__ __forceinline__ float2 split_d(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned hi32 = (unsigned)(b >> 32);
    const unsigned sign = hi32 & 0x80000000u;
    const int e = (int)((hi32 >> 20) & 0x7FFu);
    float h = 0.f, l = 0.f;
    if (e >= 897) {
        if (e > 1150) {
            h = __uint_as_float(sign | 0x7F800000u);   // beyond the FP32 range: +-inf, never silent
        } else {
            const unsigned top23 = ((hi32 & 0xFFFFFu) << 3) | (unsigned)((b >> 29) & 7u);
            h = __uint_as_float(sign | ((unsigned)(e - 896) << 23) | top23);
            const unsigned low29 = (unsigned)(b & 0x1FFFFFFFull);
            if (e >= 949) {   // lo = low29 * 2^(e - 1075), the scale a normal float
                l = __fmul_rn(__uint_as_float(sign | ((unsigned)(e - 948) << 23)), __uint2float_rn(low29));
            } else {          // the same in two normal-range factors, 2^-64 and 2^(e - 1011)
                l = __fmul_rn(__fmul_rn(__uint2float_rn(low29), __uint_as_float(sign | (63u << 23))),
                              __uint_as_float((unsigned)(e - 884) << 23));
            }
        }
    }
    return make_float2(h, l);
}

// (sh, sl) += a * b for double-float a, b
__device__ __forceinline__ void dfma(const float2 a, const float2 b, float& sh, float& sl) {
    const float p = __fmul_rn(a.x, b.x);
    float e = fmaf(a.x, b.x, -p);   // rounding error of p, exact
    e = fmaf(a.x, b.y, e);
    e = fmaf(a.y, b.x, e);
    const float t = __fadd_rn(sh, p);   // TwoSum(sh, p)
    const float bp = __fsub_rn(t, sh);
    const float err = __fadd_rn(__fsub_rn(sh, __fsub_rn(t, bp)), __fsub_rn(p, bp));
    sl = __fadd_rn(sl, __fadd_rn(err, e));
    sh = t;
}

__device__ __forceinline__ void renorm(float& sh, float& sl) {   // FastTwoSum, |sh| >= |sl|
    const float t = __fadd_rn(sh, sl);
    sl = __fsub_rn(sl, __fsub_rn(t, sh));
    sh = t;
}

__device__ __forceinline__ double to_d(float sh, float sl) { return __dadd_rn((double)sh, (double)sl); }

// ---- the same on pairs of lanes: sm_103a executes one FP32 operation on two packed floats per
// instruction (add/fma.rn.f32x2, each half rounded as the scalar instruction rounds).  The FP32 pipe
// is as busy as with scalar instructions, but the issue slots are halved, which leaves room for the
// shared-memory loads and the splitting beside the sums. ----
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float x, float y) {
    f32x2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
    return d;
}
__device__ __forceinline__ void unpack2(f32x2 a, float& x, float& y) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a));
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
// x - y as the (exact) FMA y * -1 + x
__device__ __forceinline__ f32x2 sub2(f32x2 x, f32x2 y) { return fma2(y, 0xBF800000BF800000ull, x); }

// Multiply-add on two lanes: (sh, sl) += (ax + ay) (bx + by), the operands' high and low parts packed
// apart.  TwoSum(sh, p) gives t and two exact differences, sh - (t - bp) and p - bp; the second is
// taken together with the rounding error of p in one FMA, ax bx - bp: 10 instructions against dfma's
// 12, with two more roundings of the size of ulp(t).  Its users keep the sums short (64 terms between
// FP64 flushes), which leaves their error below that of 128 terms with dfma.
// nz is a pair of -0.0f that the compiler must not see through (a kernel argument, NEG_ZERO2): the
// rounded product is RN(ax bx + -0).  ptxas contracts mul.rn.f32x2 + add.rn.f32x2 into one fma.f32x2
// (measured; -fmad=false does not stop it), and an unrounded p would break the TwoSum.
constexpr f32x2 NEG_ZERO2 = 0x8000000080000000ull;
__device__ __forceinline__ void dfma2(f32x2 ax, f32x2 ay, f32x2 bx, f32x2 by, f32x2& sh, f32x2& sl, f32x2 nz) {
    const f32x2 p = fma2(ax, bx, nz);
    const f32x2 t = add2(sh, p);
    const f32x2 nbp = sub2(sh, t);           // -(t - sh)
    const f32x2 q = sub2(sh, add2(t, nbp));
    f32x2 e = fma2(ax, bx, nbp);
    e = fma2(ax, by, e);
    e = fma2(ay, bx, e);
    sl = add2(sl, add2(e, q));
    sh = t;
}
__device__ __forceinline__ void renorm2(f32x2& sh, f32x2& sl) {
    const f32x2 t = add2(sh, sl);
    sl = sub2(sl, sub2(t, sh));
    sh = t;
}

// FP64 value of a float without the conversion unit, which runs at the FP64 rate (normal floats and
// zero by their bits; subnormals, infinities and NaN by the conversion)
__device__ __forceinline__ double widen(float x) {
    const unsigned b = __float_as_uint(x), e = b & 0x7F800000u;
    if (e == 0x7F800000u || (e == 0 && (b & 0x7FFFFFu))) return (double)x;
    const unsigned hi = e ? ((b & 0x80000000u) | (((b & 0x7FFFFFFFu) >> 3) + 0x38000000u)) : (b & 0x80000000u);
    return __hiloint2double((int)hi, (int)(b << 29));
}

}  // namespace df
}  // namespace hbsd
