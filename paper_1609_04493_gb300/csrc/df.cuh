// df.cuh -- double-float arithmetic: a value is the unevaluated sum hi + lo of
// two FP32 numbers with |lo| <= ulp(hi) / 2, a significand of about 48 bits.
//
// Methods: the exact sum a + b = s + e is Knuth's branch-free two-sum (TAOCP
// vol. 2, Sec. 4.2.2) and, for |a| >= |b|, Dekker's fast two-sum (T. J.
// Dekker, Numer. Math. 18, 1971); the exact product a b = p + e takes its
// error from one fused multiply-add. The sum of two double-floats adds the
// two low parts to the error of the high parts and renormalises once (the
// cheaper of Dekker's two additions): its error is a few units of 2^-48
// times |x| + |y|, the bound a double sum of inputs that carry rounding
// errors of their own already has. Products are accurate to a few units of
// 2^-48 of the result.
//
// On GB300 the FP32 pipe executes 64 times as many fused multiply-adds per
// clock as the FP64 pipe, so a double-float multiply-add (about 15 FP32
// instructions) costs a quarter of an FP64 one in issue time.
//
// The same helpers are overloaded for double, so code templated on the scalar
// D runs in either.
#pragma once
#include <cuda_runtime.h>

namespace rdyn {
// The type and its operators sit in a namespace of their own so that calls
// to fma inside rdyn find this overload by argument-dependent lookup only and
// do not hide the global fma(double, double, double).
namespace dfloat {

// 8-byte aligned, so a pair moves with one 64-bit load or store
struct alignas(8) DF {
    float hi, lo;
    DF() = default;
    __host__ __device__ constexpr DF(float h, float l) : hi(h), lo(l) {}
    __host__ __device__ constexpr explicit DF(float h) : hi(h), lo(0.0f) {}
};

// exact a + b = s + e (Knuth)
__device__ __forceinline__ DF df_two_sum(float a, float b)
{
    const float s = a + b;
    const float bb = s - a;
    return DF(s, (a - (s - bb)) + (b - bb));
}

// exact a + b = s + e for |a| >= |b| or a = 0 (Dekker)
__device__ __forceinline__ DF df_fast_two_sum(float a, float b)
{
    const float s = a + b;
    return DF(s, b - (s - a));
}

__device__ __forceinline__ DF operator+(DF x, DF y)
{
    const DF s = df_two_sum(x.hi, y.hi);
    return df_fast_two_sum(s.hi, s.lo + (x.lo + y.lo));
}

__device__ __forceinline__ DF operator-(DF x) { return DF(-x.hi, -x.lo); }
__device__ __forceinline__ DF operator-(DF x, DF y) { return x + (-y); }

__device__ __forceinline__ DF operator*(DF x, DF y)
{
    const float p = x.hi * y.hi;
    const float e = fmaf(x.hi, y.lo, fmaf(x.lo, y.hi, fmaf(x.hi, y.hi, -p)));
    return df_fast_two_sum(p, e);
}

// x y + z: the product's exact high part and error terms, then one sum
__device__ __forceinline__ DF fma(DF x, DF y, DF z)
{
    const float p = x.hi * y.hi;
    const float e = fmaf(x.hi, y.lo, fmaf(x.lo, y.hi, fmaf(x.hi, y.hi, -p)));
    const DF s = df_two_sum(p, z.hi);
    return df_fast_two_sum(s.hi, s.lo + (e + z.lo));
}

__device__ __forceinline__ DF &operator+=(DF &x, DF y) { return x = x + y; }
__device__ __forceinline__ DF &operator-=(DF &x, DF y) { return x = x - y; }

// ---- sums formed as one: the errors of the products and of the partial sums
// of the high parts are added up beside the high part. Error: a
// few units of 2^-48 times the sum of the terms' magnitudes, no more than the
// same sum as a chain of multiply-adds, for fewer instructions (two products: 16
// against 22; three: 28 against 37; four terms: 24 against 33).

// high part and error of x y; of c y for a plain float c
__device__ __forceinline__ DF df_prod(DF x, DF y)
{
    const float p = x.hi * y.hi;
    return DF(p, fmaf(x.hi, y.lo, fmaf(x.lo, y.hi, fmaf(x.hi, y.hi, -p))));
}
__device__ __forceinline__ DF df_prod(float c, DF y)
{
    const float p = c * y.hi;
    return DF(p, fmaf(c, y.lo, fmaf(c, y.hi, -p)));
}

// The _raw forms leave the result unnormalised: hi is the rounded sum of the high
// parts, lo every error and low part. As an operand of a further sum of products
// it is as good (the neglected lo lo is 2^-48 of the magnitudes that went into
// it, as the value's own error is); what is carried on from link to link is
// renormalised (df_renorm).
__device__ __forceinline__ DF df_renorm(DF x) { return df_fast_two_sum(x.hi, x.lo); }

// x0 y0 + x1 y1 (S: DF or float)
template <typename S>
__device__ __forceinline__ DF ddot2_raw(S x0, DF y0, S x1, DF y1)
{
    const DF p = df_prod(x0, y0), r = df_prod(x1, y1);
    const DF s = df_two_sum(p.hi, r.hi);
    return DF(s.hi, s.lo + (p.lo + r.lo));
}

__device__ __forceinline__ DF ddot3_raw(DF x0, DF y0, DF x1, DF y1, DF x2, DF y2)
{
    const DF p = df_prod(x0, y0), r = df_prod(x1, y1), t = df_prod(x2, y2);
    const DF s = df_two_sum(p.hi, r.hi);
    const DF u = df_two_sum(s.hi, t.hi);
    return DF(u.hi, (s.lo + u.lo) + (p.lo + r.lo + t.lo));
}

// x y + z
__device__ __forceinline__ DF dfma_raw(DF x, DF y, DF z)
{
    const DF p = df_prod(x, y);
    const DF s = df_two_sum(p.hi, z.hi);
    return DF(s.hi, s.lo + (p.lo + z.lo));
}

__device__ __forceinline__ DF dsum2_raw(DF x, DF y)
{
    const DF s = df_two_sum(x.hi, y.hi);
    return DF(s.hi, s.lo + (x.lo + y.lo));
}

__device__ __forceinline__ DF dsum3_raw(DF x, DF y, DF z)
{
    const DF s = df_two_sum(x.hi, y.hi);
    const DF u = df_two_sum(s.hi, z.hi);
    return DF(u.hi, (s.lo + u.lo) + (x.lo + y.lo + z.lo));
}

__device__ __forceinline__ DF dsum4_raw(DF x, DF y, DF z, DF w)
{
    const DF s = df_two_sum(x.hi, y.hi), t = df_two_sum(z.hi, w.hi);
    const DF u = df_two_sum(s.hi, t.hi);
    return DF(u.hi, (s.lo + t.lo + u.lo) + ((x.lo + y.lo) + (z.lo + w.lo)));
}

__device__ __forceinline__ DF dmul_raw(DF x, DF y) { return df_prod(x, y); }
__device__ __forceinline__ DF dmul_raw(float c, DF y) { return df_prod(c, y); }

}  // namespace dfloat
using dfloat::ddot2_raw;
using dfloat::ddot3_raw;
using dfloat::DF;
using dfloat::df_renorm;
using dfloat::df_two_sum;
using dfloat::dfma_raw;
using dfloat::dmul_raw;
using dfloat::dsum2_raw;
using dfloat::dsum3_raw;
using dfloat::dsum4_raw;

// the same in FP64
__device__ __forceinline__ double df_renorm(double x) { return x; }
__device__ __forceinline__ double ddot2_raw(double x0, double y0, double x1, double y1)
{
    return fma(x0, y0, x1 * y1);
}
__device__ __forceinline__ double ddot3_raw(double x0, double y0, double x1, double y1, double x2,
                                            double y2)
{
    return fma(x0, y0, fma(x1, y1, x2 * y2));
}
__device__ __forceinline__ double dfma_raw(double x, double y, double z) { return fma(x, y, z); }
__device__ __forceinline__ double dsum2_raw(double x, double y) { return x + y; }
__device__ __forceinline__ double dsum3_raw(double x, double y, double z) { return (x + y) + z; }
__device__ __forceinline__ double dsum4_raw(double x, double y, double z, double w)
{
    return (x + y) + (z + w);
}
__device__ __forceinline__ double dmul_raw(double x, double y) { return x * y; }

// ---- helpers overloaded for double and DF

// x / 2 and 2 x (exact)
__device__ __forceinline__ double dhalf(double x) { return 0.5 * x; }
__device__ __forceinline__ DF dhalf(DF x) { return DF(0.5f * x.hi, 0.5f * x.lo); }
__device__ __forceinline__ double dtwice(double x) { return 2.0 * x; }
__device__ __forceinline__ DF dtwice(DF x) { return DF(2.0f * x.hi, 2.0f * x.lo); }
// 2 x + y: one FMA in double; the exact doubling and one sum in double-float
__device__ __forceinline__ double dtwice_add(double x, double y) { return fma(2.0, x, y); }
__device__ __forceinline__ DF dtwice_add(DF x, DF y) { return dtwice(x) + y; }

// 1 / x. DF: the FP32 reciprocal r refined by one Newton step
// r + r (1 - x r), which doubles its correct bits.
__device__ __forceinline__ double drecip(double x) { return 1.0 / x; }
__device__ __forceinline__ DF drecip(DF x)
{
    const float r = 1.0f / x.hi;
    const DF e = DF(1.0f) - x * DF(r);
    return fma(DF(r), e, DF(r));
}

__device__ __forceinline__ bool dpositive(double x) { return x > 0.0; }
__device__ __forceinline__ bool dpositive(DF x) { return x.hi > 0.0f; }
__device__ __forceinline__ bool disnan(double x) { return !(x == x); }
__device__ __forceinline__ bool disnan(DF x) { return !(x.hi == x.hi); }

// a - b of two data values in D: exact for FP32 data (a double, or a
// double-float, holds the difference of two floats exactly), one rounding for
// FP64 data
template <typename D>
struct DSub;
template <>
struct DSub<double> {
    __device__ __forceinline__ static double sub(float a, float b) { return (double)a - (double)b; }
    __device__ __forceinline__ static double sub(double a, double b) { return a - b; }
};
template <>
struct DSub<DF> {
    __device__ __forceinline__ static DF sub(float a, float b) { return df_two_sum(a, -b); }
};

template <typename D, typename T>
__device__ __forceinline__ D dsub_exact(T a, T b)
{
    return DSub<D>::sub(a, b);
}

// the value of lane src
__device__ __forceinline__ DF df_shfl(DF x, int src)
{
    return DF(__shfl_sync(0xffffffffu, x.hi, src), __shfl_sync(0xffffffffu, x.lo, src));
}

// conversions between the data types (float, double) and D
template <typename To>
struct DCvt;
template <>
struct DCvt<double> {
    __device__ __forceinline__ static double from(float x) { return (double)x; }
    __device__ __forceinline__ static double from(double x) { return x; }
    __device__ __forceinline__ static double from(DF x) { return (double)x.hi + (double)x.lo; }
};
template <>
struct DCvt<float> {
    __device__ __forceinline__ static float from(float x) { return x; }
    __device__ __forceinline__ static float from(double x) { return (float)x; }
    __device__ __forceinline__ static float from(DF x) { return x.hi + x.lo; }
};
template <>
struct DCvt<DF> {
    __device__ __forceinline__ static DF from(float x) { return DF(x); }
    __device__ __forceinline__ static DF from(DF x) { return x; }
};

template <typename To, typename From>
__device__ __forceinline__ To dcvt(From x)
{
    return DCvt<To>::from(x);
}

// A plain factor (the sine or cosine of a joint angle) beside values of type D: an FP32
// factor stays a float next to double-floats, where its products take one
// multiply-add less.
template <typename D>
struct DScalar;
template <>
struct DScalar<double> {
    __device__ __forceinline__ static double from(double x) { return x; }
};
template <>
struct DScalar<DF> {
    __device__ __forceinline__ static float from(float x) { return x; }
    __device__ __forceinline__ static DF from(DF x) { return x; }
};
template <typename D, typename From>
__device__ __forceinline__ auto dscalar(From x)
{
    return DScalar<D>::from(x);
}

// nearest double-float of a double (host side: records are split once;
// constexpr, so constant tables split at compile time)
constexpr DF df_split_host(double v)
{
    return DF((float)v, (float)(v - (double)(float)v));
}

// double <-> double-float on the device (conversions on the FP64 path)
__device__ __forceinline__ DF df_from_double(double v)
{
    const float hi = __double2float_rn(v);
    return DF(hi, __double2float_rn(v - (double)hi));
}

__device__ __forceinline__ double df_to_double(DF x) { return (double)x.hi + (double)x.lo; }

}  // namespace rdyn
