// trig_fixed.cuh -- FP64 sine and cosine with the polynomials in 64-bit fixed point
// on the integer pipe.
//
// GB300's FP64 unit takes a warp instruction every 19 cycles per SM (measured: 76 per
// scheduler with all four busy), so the ~28 FP64 instructions of the library's
// sincos were a sixth of an FP64 kernel's time. Here FP64 does the reduction and one
// multiply-add (7 instructions); the rest is about 130 integer instructions, which
// issue beside the FP64 unit.
//
// Reduction (Cody and Waite, "Software Manual for the Elementary Functions", 1980):
// k = nearest integer to x (2 / pi), r = x - k pi/2 with pi/2 split into three doubles,
// each product fused; |r| <= pi/4 up to rounding, and the first difference is exact
// where it cancels.
// With z = r^2 as a 64-bit fraction, the Taylor series
//     h = 1 - sin(r) / r = z/3! - z^2/5! + ...   (8 terms),
//     y = 1 - cos(r)     = z/2! - z^2/4! + ...   (9 terms)
// by Horner's rule in 64-bit fractions; the terms below 2^-25 (2^-28) of the leading
// one in 32 bits, where their rounding costs under 2^-60. First omitted terms:
// 2^-62 and 2^-61. Then sin r = r - r h in one multiply-add and cos r = 1 - y rounded
// from its fraction: both within 0.51 ulp of r's sine and cosine. r's own rounding
// is half an ulp of r, a whole one of a sine that lies in the binade below: at most 1.51
// ulp in all (the library: up to 2). Seen against 113- and 140-bit values: up to 1.35
// over one turn, 1.49 up to 2^30 rad, 0.3 on average.
// The sine of -0 is +0. Angles of 2^30 rad or more, infinities and NaN take the library.
#pragma once
#include <cuda_runtime.h>

#include "df_trig.cuh"

namespace rdyn {

// high half of a b, at most 3 units too small (the low halves' product is left out)
__device__ __forceinline__ unsigned long long fx_mulhi(unsigned long long a, unsigned long long b)
{
    const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a;
    const unsigned bh = (unsigned)(b >> 32), bl = (unsigned)b;
    return (unsigned long long)ah * bh + __umulhi(ah, bl) + __umulhi(al, bh);
}

// pi/2 less its head and tail (df_trig.cuh), nearest double
constexpr double kPio2Third = -1.4973849048591698e-33;

static __device__ __noinline__ void sincos_large(double x, double *s, double *c) { sincos(x, s, c); }

__device__ __forceinline__ void sincos_fixed(double x, double *s_out, double *c_out)
{
    if (((unsigned)__double2hiint(x) & 0x7fffffffu) >= 0x41d00000u) {  // |x| >= 2^30, inf, NaN
        double s, c;
        sincos_large(x, &s, &c);
        *s_out = s;
        *c_out = c;
        return;
    }
    const double kMagic = 6755399441055744.0;  // 1.5 * 2^52: leaves k in the low bits
    const double t = fma(x, kDfTwoOverPi, kMagic);
    const int quad = __double2loint(t);
    const double k = t - kMagic;
    const double r = fma(-k, kPio2Third, fma(-k, kDfPio2Tail, fma(-k, kDfPio2Head, x)));
    // |r| < 1 as a 64-bit fraction, then z = r^2
    const unsigned hi = (unsigned)__double2hiint(r) & 0x7fffffffu;
    const unsigned long long mant =
        ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | (unsigned)__double2loint(r);
    const int sh = (int)(hi >> 20) - 1011;
    const unsigned long long u = sh >= 0 ? mant << sh : mant >> (-sh < 63 ? -sh : 63);
    const unsigned long long z = fx_mulhi(u, u);
    const unsigned zh = (unsigned)(z >> 32);
    // h: 1/11!, 1/13!, ... in units of 2^-57, then 1/9!, ..., 1/3! in 2^-64
    unsigned p = 0x1ae7fu - __umulhi(zh, 0x195u);
    p = 0x1612461u - __umulhi(zh, p);
    p = 0xd7322b40u - __umulhi(zh, p);
    unsigned long long h = 0x2e3bc74aad8eull - (((unsigned long long)zh * p) >> 25);
    h = 0xd00d00d00d00dull - fx_mulhi(z, h);
    h = 0x222222222222222ull - fx_mulhi(z, h);
    h = 0x2aaaaaaaaaaaaaabull - fx_mulhi(z, h);
    h = fx_mulhi(z, h) | 1u;
    // y: 1/12!, 1/14!, ... in units of 2^-60, then 1/10!, ..., 1/2! in 2^-64
    p = 0xd740u - __umulhi(zh, 0xb4u);
    p = 0xc9cba5u - __umulhi(zh, p);
    p = 0x8f76c780u - __umulhi(zh, p);
    unsigned long long y = 0x49f93edde28ull - (((unsigned long long)zh * p) >> 28);
    y = 0x1a01a01a01a02ull - fx_mulhi(z, y);
    y = 0x5b05b05b05b05bull - fx_mulhi(z, y);
    y = 0xaaaaaaaaaaaaaabull - fx_mulhi(z, y);
    y = 0x8000000000000000ull - fx_mulhi(z, y);
    y = fx_mulhi(z, y);
    // h as a double (truncated), sin r = r - r h
    const int lz = __clzll((long long)h);
    const double hd = __longlong_as_double(((long long)(1021 - lz) << 52) + (long long)((h << lz) >> 11));
    const double sr = fma(-r, hd, r);
    // cos r in [0.7, 1]: a 63-bit fraction whose leading bit is 62 (63 at 1)
    const unsigned long long v = 0x8000000000000000ull - (y >> 1);
    const double cr = __longlong_as_double((1021ll << 52) + (long long)((v + 512) >> 10));
    const double a = (quad & 1) ? cr : sr, b = (quad & 1) ? sr : cr;
    *s_out = __hiloint2double(__double2hiint(a) ^ ((quad & 2) << 30), __double2loint(a));
    *c_out = __hiloint2double(__double2hiint(b) ^ (((quad + 1) & 2) << 30), __double2loint(b));
}

}  // namespace rdyn
