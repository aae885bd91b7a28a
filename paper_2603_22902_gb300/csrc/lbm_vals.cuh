// lbm_vals.cuh -- the value types that the arithmetic of one lattice update is written in
// (lbm_cell.cuh): d1 (FP64), df64 (double words) and f1 (FP32).
//
// d1 and f1 round every operation as it is written: their sums and products are the
// round-to-nearest intrinsics, which the compiler neither contracts nor reorders, and a fused
// multiply-add is there only where rfma says so (df64 is written likewise).  A cell therefore
// gets the same bits from any kernel that computes it, whatever its tile shape.
#pragma once

#include <type_traits>

#include "lbm_df64.cuh"

namespace lbm {

struct f1 {
    float v;
    f1() = default;
    __device__ __forceinline__ constexpr f1(float a) : v(a) {}
    __device__ __forceinline__ explicit constexpr operator float() const { return v; }
    __device__ __forceinline__ explicit constexpr operator double() const { return (double)v; }
};
__device__ __forceinline__ f1 operator+(f1 a, f1 b) { return f1(__fadd_rn(a.v, b.v)); }
__device__ __forceinline__ f1 operator-(f1 a, f1 b) { return f1(__fsub_rn(a.v, b.v)); }
__device__ __forceinline__ f1 operator*(f1 a, f1 b) { return f1(__fmul_rn(a.v, b.v)); }
__device__ __forceinline__ f1 operator-(f1 a) { return f1(-a.v); }
__device__ __forceinline__ bool operator>(f1 a, f1 b) { return a.v > b.v; }
__device__ __forceinline__ bool operator==(f1 a, f1 b) { return a.v == b.v; }
__device__ __forceinline__ bool operator==(df64 a, df64 b) { return a.hi == b.hi && a.lo == b.lo; }
__device__ __forceinline__ f1 rfma(f1 a, f1 b, f1 c) { return f1(__fmaf_rn(a.v, b.v, c.v)); }

struct d1 {
    double v;
    d1() = default;
    __device__ __forceinline__ constexpr d1(double a) : v(a) {}
    __device__ __forceinline__ explicit constexpr operator double() const { return v; }
};
__device__ __forceinline__ d1 operator+(d1 a, d1 b) { return d1(__dadd_rn(a.v, b.v)); }
__device__ __forceinline__ d1 operator-(d1 a, d1 b) { return d1(__dsub_rn(a.v, b.v)); }
__device__ __forceinline__ d1 operator*(d1 a, d1 b) { return d1(__dmul_rn(a.v, b.v)); }
__device__ __forceinline__ d1 operator-(d1 a) { return d1(-a.v); }
__device__ __forceinline__ bool operator>(d1 a, d1 b) { return a.v > b.v; }
__device__ __forceinline__ bool operator==(d1 a, d1 b) { return a.v == b.v; }
__device__ __forceinline__ d1 rfma(d1 a, d1 b, d1 c) { return d1(__fma_rn(a.v, b.v, c.v)); }

// Fused multiply-adds of the other types, and the reciprocal and the reciprocal square root.
__device__ __forceinline__ double rfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float rfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double rrsqrt(double a) { return rsqrt(a); }
__device__ __forceinline__ float rrsqrt(float a) { return rsqrtf(a); }
__device__ __forceinline__ f1 rrsqrt(f1 a) { return f1(rsqrtf(a.v)); }
__device__ __forceinline__ d1 rrsqrt(d1 a) { return d1(rsqrt(a.v)); }
__device__ __forceinline__ d1 rinv(d1 a) { return d1(__drcp_rn(a.v)); }
__device__ __forceinline__ df64 rinv(df64 a) { return df64(1) / a; }
__device__ __forceinline__ f1 rinv(f1 a) { return f1(__frcp_rn(a.v)); }

// Type of a constant that FP32 holds exactly (2, 3, 0.5, 4.5, ...) in arithmetic of type V:
// V itself, except float for double words (a product with a float costs 3 FP32 instructions
// instead of 4) and for FP32.
template <class V>
using exact_t =
    typename std::conditional<std::is_same<V, double>::value || std::is_same<V, d1>::value, double, float>::type;
// Type of any other constant, and of the coefficients: df64 for double words, else the same.
template <class V>
using const_t = typename std::conditional<std::is_same<V, df64>::value, df64, exact_t<V>>::type;

// The value type of a policy's arithmetic type R.
template <class R>
using val_t = typename std::conditional<std::is_same<R, float>::value, f1,
                                        typename std::conditional<std::is_same<R, double>::value, d1, R>::type>::type;

// The leading FP32 part of a value, for the screens of eq. H.  For a double: its sign, exponent
// and 23 leading fraction bits, put together with integer instructions, since a conversion
// would run on the 2-lane FP64 unit; magnitudes below FP32's normal range become 0 (or a value
// below 2^-126), magnitudes above it, infinities and NaN become infinite.
__device__ __forceinline__ float lead(f1 a) { return a.v; }
__device__ __forceinline__ float lead(float a) { return a; }
__device__ __forceinline__ float lead(df64 a) { return a.hi; }
__device__ __forceinline__ float lead(d1 a)
{
    const int hi = __double2hiint(a.v), lo = __double2loint(a.v);
    int e = (hi & 0x7fffffff) - 0x38000000;        // exponent bias 1023 -> 127
    const bool none = e < 0, most = e >= 0x0ff00000;
    unsigned m = __funnelshift_l((unsigned)lo, (unsigned)e, 3);
    m = none ? 0u : most ? 0x7f800000u : m;
    return __uint_as_float(m | ((unsigned)hi & 0x80000000u));
}

}  // namespace lbm
