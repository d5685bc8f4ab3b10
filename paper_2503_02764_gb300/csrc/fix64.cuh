// FP64 results with few FP64 instructions.
//
// An FP64 instruction of a warp holds this GPU's FP64 pipe for 16 to 19 cycles of an SM, in which its four
// schedulers can issue 64 other instructions. The routines here do the bulk of an operation in
// FP32 and integer arithmetic and leave to FP64 only what fixes the last bits:
//   fix_div, fix_sqrt   a double-FP32 approximation (~2^-39) from an FP32 reciprocal (square
//                       root), joined to an FP64 number by integer addition, then one
//                       residual and one correction in FP64 (two instructions in place of
//                       five or more, half a unit of rounding plus ~2^-61);
//   fix_stencil         the 4th-order difference E_-2 - 8 E_-1 + 8 E_+1 - E_+2 in 63-bit fixed
//                       point (no FP64 instruction in place of three): the sum is exact to
//                       2^-57 of the largest operand per operand and rounded once, where the
//                       FP64 form rounds a sum eight times as large as the operands.
// The operand of fix_sqrt is positive and within in_f32_range, those of fix_div pass div_ok.
#pragma once
#include "fld_internal.cuh"

namespace fld {

struct f32pair {
    float h, l;
};

// v = h + l to 2^-46: h the top 24 bits of the significand, l the next 23
__device__ __forceinline__ f32pair split_pos(double v) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const unsigned h = __funnelshift_l(lo, hi, 3) - (896u << 23);
    const float us = __uint_as_float((h & 0x7F800000u) - (23u << 23));     // one unit of h
    const float f = __uint_as_float(0x3F800000u | ((lo & 0x1FFFFFFFu) >> 6));
    return {__uint_as_float(h), __fmaf_rn(f, us, -us)};
}

// h + l as FP64 (h positive and normal, |l| below 64 units of h), l rounded to 2^-15 units of h:
// 2^-39 of the value, which the residual correction takes to 2^-61 (1.5 * 2^23 rounds to the
// integer). Where the sum leaves h's binade, the part beyond the power of two is in other units:
// half as large below it, twice as large above. (Left as it is, that part would be off by half or
// twice its size, up to 2^-23 of the value, and the quotient by 2^-46.)
__device__ __forceinline__ double join_pos(float h, float l) {
    const unsigned u = __float_as_uint(h);
    const float per = __uint_as_float((277u << 23) - (u & 0x7F800000u));   // 1 / unit of h
    const int r = __float_as_int(__fmaf_rn(l * per, 32768.f, 12582912.f)) - 0x4B400000;
    const long long hb = (long long)(((unsigned long long)u + (896ull << 23)) << 29);
    long long b = hb + ((long long)r << 14);
    if (__builtin_expect((((int)(b >> 32) ^ (int)(hb >> 32)) & 0x7FF00000) != 0, 0)) {
        asm volatile("");              // a branch: not executed by every cell
        const long long edge = (max(b, hb) >> 52) << 52;
        b = b < edge ? 2 * b - edge : (b + edge) >> 1;
    }
    return __longlong_as_double(b);
}

__device__ __forceinline__ float rcp_fast(float a) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(a));
    return y;
}
__device__ __forceinline__ float rsqrt_fast(float a) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(a));
    return y;
}

// n and d, and their quotient, positive and far enough inside the FP32 normal range
__device__ __forceinline__ bool div_ok(double n, double d) {
    const int en = __double2hiint(n) >> 20, ed = __double2hiint(d) >> 20;
    return (unsigned)(en - 924) < 198u && (unsigned)(ed - 924) < 198u && abs(en - ed) < 98;
}

// n / d for operands that pass div_ok
__device__ __forceinline__ double fix_div(double n, double d) {
    const f32pair a = split_pos(n), b = split_pos(d);
    const float y = rcp_fast(b.h);
    const float q = a.h * y;
    const float r = __fmaf_rn(-q, b.l, __fmaf_rn(-q, b.h, a.h)) + a.l;
    const double q0 = join_pos(q, r * y);
    return fma(fma(-q0, d, n), f64_of_pos(y), q0);
}

__device__ __forceinline__ double fix_sqrt(double x) {
    const f32pair a = split_pos(x);
    const float y = rsqrt_fast(a.h), hy = 0.5f * y;
    const float s = a.h * y;
    const float r = __fmaf_rn(-s, s, a.h) + a.l;
    const double s0 = join_pos(s, r * hy);
    return fma(fma(-s0, s0, x), f64_of_pos(hy), s0);
}

// the FP64 value as a 63-bit fixed-point number, its unit 2^(emax - 1080)
__device__ __forceinline__ long long fix_of(unsigned hi, unsigned lo, int emax) {
    const int e = (int)((hi >> 20) & 0x7FFu);
    const unsigned top = (hi & 0xFFFFFu) | (e ? 0x100000u : 0u);
    const unsigned long long m = ((((unsigned long long)top << 32) | lo) << 5) >> min(emax - e, 63);
    const long long s = (long long)(int)hi >> 63;
    return ((long long)m ^ s) - s;
}

// the same in FP64, for operands near the ends of the exponent range. Out of line: inlined, its
// three FP64 instructions are executed speculatively by every cell.
static __device__ __noinline__ double stencil_far(double a, double b, double c, double d) {
    return fma(d, -1.0, fma(8.0, c, fma(-8.0, b, a)));
}

// a - 8 b + 8 c - d
__device__ __forceinline__ double fix_stencil(double a, double b, double c, double d) {
    const unsigned ha = (unsigned)__double2hiint(a), hb = (unsigned)__double2hiint(b),
                   hc = (unsigned)__double2hiint(c), hd = (unsigned)__double2hiint(d);
    const unsigned m = 0x7FF00000u;
    const int emax = (int)(max(max(ha & m, hb & m), max(hc & m, hd & m)) >> 20);
    if (emax < 128 || emax > 2000) return stencil_far(a, b, c, d);
    const long long s = (fix_of(ha, (unsigned)__double2loint(a), emax) -
                         fix_of(hd, (unsigned)__double2loint(d), emax)) +
                        ((fix_of(hc, (unsigned)__double2loint(c), emax) -
                          fix_of(hb, (unsigned)__double2loint(b), emax)) << 3);
    if (s == 0) return 0.0;
    unsigned long long u = (unsigned long long)(s < 0 ? -s : s);
    const int z = __clzll((long long)u);
    u <<= z;
    // 53 bits rounded to nearest; the leading one and a carry count in the exponent field
    const unsigned long long r = (u >> 11) + ((u >> 10) & 1ull);
    return __longlong_as_double((long long)((((unsigned long long)(emax + 5 - z)) << 52) + r) |
                                (s & (long long)0x8000000000000000ull));
}

}  // namespace fld
