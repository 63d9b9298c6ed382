// Exact digit slices of FP64 values for the tensor cores (gram_tc.cu, update_tc.cu): a 62-bit fixed point in 8
// balanced base-256 digits, each exact in FP16; products of equal weight accumulated by tcgen05.mma in one FP32
// accumulator per level s + t = 0..7.  An operand tile is 16 deep; A has 128 rows, B 64 columns per slice.
#pragma once
#include <stdint.h>

#include "common.h"
#include "tc.h"

namespace hbsd {
namespace slices {

constexpr int DIG = 8;                    // base-256 digits per operand
constexpr int ROWS = 128;                 // rows of an A slice (M of every MMA)
constexpr int COLS = 64;                  // columns of a B slice; level L's accumulator begins at TMEM column 64 L
constexpr int A_SLICE = ROWS * 16 * 2;    // bytes of one 128 x 16 slice
constexpr int B_SLICE = COLS * 16 * 2;    // bytes of one 64 x 16 slice
constexpr int FLUSH_STEPS = 16;           // steps of 16 between readings of the accumulators: levels 0-4 stay exact
constexpr int FRAC = 37;                  // fraction bits of the 64-bit sums, in units of the leading digit product
constexpr int FRAC_LOW = 8;               // further fraction bits, kept beside the sums (fold_levels)
constexpr int BAD_EXP = 0x40000000;       // exponent of a row or column with a non-finite entry
constexpr uint64_t WAIT_NS = 2000000000ull;

__device__ __forceinline__ int exp_field(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }

__device__ __forceinline__ void mbar_arrive(uint64_t* mbar) {
    asm volatile("{\n.reg .b64 st;\nmbarrier.arrive.shared::cta.b64 st, [%0];\n}\n" ::"r"(tc::smem_u32(mbar)) : "memory");
}
template <int ACC>
__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc) {
    asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
                 "l"(a), "l"(b), "r"(idesc), "n"(ACC));
}
// slice s of A times the B slices 0 .. 7 - s into levels s .. 7
template <int S, int ACC>
__device__ __forceinline__ void mma_window(uint32_t tbase, uint64_t a, uint64_t b) {
    constexpr int N = (DIG - S) * COLS, N0 = N > 256 ? 256 : N;
    mma<ACC>(tbase + S * COLS, a + S * (A_SLICE >> 4), b, tc::idesc_f16_f32(ROWS, N0));
    if constexpr (N > 256)
        mma<ACC>(tbase + S * COLS + 256, a + S * (A_SLICE >> 4), b + 4 * (B_SLICE >> 4), tc::idesc_f16_f32(ROWS, N - 256));
}

// |x| as a 62-bit fixed-point integer, rounded to nearest, plus 0x0080808080808080: byte 7 - s is the digit d_s of
// |x| plus 128, the leading byte d_0 itself.  off: the column's exponent plus or minus the row's; off - exponent
// field >= 0 is the shift below the maximum.  The rounding takes one more bit, halved after the bias and a half are
// added; cut instead, same-signed columns lose up to a unit per row, all one way: 2^-44 of sum|z||h| over 8192 rows at
// the guard's line, 2^-48 rounded.  The digits of the sign are taken in digits2.
__device__ __forceinline__ unsigned long long fixed62(double x, int off) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int ex = (int)((hi >> 20) & 0x7FFu);
    const unsigned sh = ex ? (unsigned)(off - ex) : 64u;   // zeros and subnormals enter as zero
    const unsigned mh = __funnelshift_l(lo, (hi & 0xFFFFFu) | 0x100000u, 10), ml = lo << 10;
    unsigned long long v;
    asm("shr.b64 %0, %1, %2;" : "=l"(v) : "l"(((unsigned long long)mh << 32) | ml), "r"(sh));   // 0 from 64 on
    return (v + 0x0101010101010101ull) >> 1;
}

// FP16 digits s of two values from one byte of each biased integer: 1024 + byte by its bits (the leading byte, at most
// 64, with its bias put in here), then (1024 + byte) sg - 1152 sg = +-d exactly, with sg = +-1 the values' signs and
// csg = -1152 sg
__device__ __forceinline__ uint32_t digits2(unsigned long long u0, unsigned long long u1, int s, uint32_t sg, uint32_t csg) {
    const unsigned w0 = (unsigned)(s < 4 ? u0 >> 32 : u0), w1 = (unsigned)(s < 4 ? u1 >> 32 : u1), byte = 3 - (s & 3);
    const unsigned z = (__byte_perm(w0, w1, byte | ((4 + byte) << 8)) & 0x00FF00FFu) | (s == 0 ? 0x64806480u : 0x64006400u);
    uint32_t d;
    asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(z), "r"(sg), "r"(csg));
    return d;
}
__device__ __forceinline__ uint32_t signs2(double x0, double x1) {
    return (__byte_perm((unsigned)__double2hiint(x0), (unsigned)__double2hiint(x1), 0x7030) & 0x80008000u) | 0x3C003C00u;
}

// The 8 slices of 8 values (consecutive rows of one column): 16 bytes per slice at dst + s * stride
__device__ __forceinline__ void slice8(const double (&x)[8], const int (&off)[8], uint8_t* dst, int stride) {
    uint32_t w[DIG][4];
#pragma unroll
    for (int c = 0; c < 8; c += 2) {
        const unsigned long long u0 = fixed62(x[c], off[c]), u1 = fixed62(x[c + 1], off[c + 1]);
        const uint32_t sg = signs2(x[c], x[c + 1]);
        uint32_t csg;
        asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(csg) : "r"(sg), "r"(0xE480E480u));
#pragma unroll
        for (int s = 0; s < DIG; ++s)
            w[s][c >> 1] = digits2(u0, u1, s, sg, csg);
    }
#pragma unroll
    for (int s = 0; s < DIG; ++s)
        *reinterpret_cast<uint4*>(dst + s * stride) = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
}

// The guard slice: 8 values as FP16 magnitudes 1.m 2^-shift against the column's leading power of two
// (m truncated; 0 below 2^-14 of it)
__device__ __forceinline__ unsigned guard16(double x, int off) {
    const unsigned hi = (unsigned)__double2hiint(x);
    const int ex = (int)((hi >> 20) & 0x7FFu), sh = off - ex;
    return ex != 0 && sh < 15 ? (unsigned)((15 - sh) << 10) | ((hi >> 10) & 0x3FFu) : 0u;
}
__device__ __forceinline__ void slice8_guard(const double (&x)[8], const int (&off)[8], uint8_t* dst) {
    uint32_t w[4];
#pragma unroll
    for (int c = 0; c < 8; c += 2) w[c >> 1] = guard16(x[c], off[c]) | (guard16(x[c + 1], off[c + 1]) << 16);
    *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
}

__device__ __forceinline__ void tmem_ld8(uint32_t addr, uint32_t (&v)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(addr));
}

__device__ __forceinline__ void tmem_ld4(uint32_t addr, uint32_t (&v)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                 : "r"(addr));
}

// One output's levels as a 64-bit integer in units of 2^-37 of the leading digit product, to be added to the output's sum,
// and its fraction in units of 2^-45, added to byte i of low (the sum's own fraction) with the carry in the result: levels
// 0 and 1 (within 2^22) by adding 1.5 * 2^23, whose bits then hold the integer; levels 2-5 by conversion; levels 6 and
// 7 together, rounded to 2^-45 of level 0 (2^3 of level 6).  With levels 5-7 rounded to 2^-37 at every reading, entries
// that the guard accepts at its line were off by 2^-41 of sum|z||h|, now 2^-48; the fraction and the rounded operands
// take 2% of the Gram (n = 334,272, q = 538: 9.69 -> 9.89 ms) and 3% of the update (k = 282: 7.00 -> 7.19).
__device__ __forceinline__ long long fold_levels(const uint32_t (&l)[8], uint32_t& low, int i) {
    const int m0 = __float_as_int(__fadd_rn(__uint_as_float(l[0]), 12582912.0f)) - 0x4B400000;
    const int m1 = __float_as_int(__fadd_rn(__uint_as_float(l[1]), 12582912.0f)) - 0x4B400000;
    const int m2 = __float2int_rn(__uint_as_float(l[2]));
    const int m3 = __float2int_rn(__uint_as_float(l[3]));
    const int m4 = __float2int_rn(__uint_as_float(l[4]));
    const int m5 = __float2int_rn(__uint_as_float(l[5]));
    const float g = __fmaf_rn(__uint_as_float(l[7]), 0.00390625f, __uint_as_float(l[6]));
    const int m6 = __float_as_int(__fmaf_rn(g, 0.125f, 12582912.0f)) - 0x4B400000;
    const int w = m5 * 32 + m6 + (int)((low >> (8 * i)) & 255u);   // below 2^30
    low = __byte_perm(low, (uint32_t)w, 0x3210u + ((4u - i) << (4 * i)));
    return (((long long)m0 << 37) + ((long long)m1 << 29)) + (long long)m2 * (1 << 21) + (long long)m3 * (1 << 13) +
           (long long)m4 * 32 + (long long)(w >> FRAC_LOW);
}

// v 2^e without the FP64 pipe (normalise, round to nearest, set the exponent); results outside the normal
// range by ldexp
__device__ __forceinline__ double scaled_double(long long v, int e) {
    if (v == 0) return 0.0;
    const unsigned long long m = (unsigned long long)(v < 0 ? -v : v);
    const int z = __clzll((long long)m);
    const int ex = 1023 + 63 - z + e;   // exponent field of the leading bit
    if (ex < 1 || ex > 2045) return ldexp((double)v, e);
    const unsigned long long f = m << z;   // leading bit 63; the fraction is the next 52, rounded half up
    const unsigned long long bits = ((unsigned long long)ex << 52) + ((f << 1) >> 12) + ((f >> 10) & 1ull);
    return __longlong_as_double((long long)(bits | (v < 0 ? 0x8000000000000000ull : 0ull)));
}
// (v + byte i of low 2^-8) 2^e, rounded once: the fraction counts while v has fewer than 55 bits
__device__ __forceinline__ double scaled_sum(long long v, uint32_t low, int i, int e) {
    const bool small = v + (1ll << 54) >= 0 && v < (1ll << 54);
    return scaled_double(small ? (long long)(((unsigned long long)v << FRAC_LOW) | ((low >> (8 * i)) & 255u)) : v, small ? e - FRAC_LOW : e);
}

}  // namespace slices
}  // namespace hbsd
