// lbm_num.cuh -- arithmetic types of the collision kernels.
//
// The collision rules are written once over a number type T:
//   double  FP64 path: Newton reciprocal (below) and table logarithm (lbm_f64.cuh).
//   F2      FP32 path, two nodes per value: the packed FP32x2 instructions of
//           sm_100+ (__fadd2_rn, __fmul2_rn, __ffma2_rn) do both nodes in one
//           issue; reciprocals and logarithms run per lane on the MUFU unit.
// The compiler may fuse a packed product whose only use is a following
// packed add into one packed FMA (it does so even for the _rn forms), which
// scalar __fmul_rn / __fadd_rn never are.  All step kernels use F2 with the same
// collision code and agree bit for bit with each other.
//
// FP32 transcendental choice: ln(p/W) is needed as log(1 + delta) with
// |delta| < 1 typically; the FP32 path evaluates log2(1 + delta) with the
// hardware approximation (absolute error about 2^-22) and folds ln 2 into the
// final scale factor; reciprocals use the hardware approximation (about 1 ulp).
// Both errors stay at the FP32 rounding level of the populations (the tests
// bound the FP32 results against the FP64 oracle).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace lbm {

__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float lg2_approx(float x) {
    float r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// 1 / x in FP64: the FP32 reciprocal of x cut to 24 bits (error below 2^-21.9)
// as the seed and one third-order Newton step, r (1 + e + e^2) with e = 1 - x r:
// 3 FP64 instructions instead of an IEEE division's 8.  The error before the
// last rounding is e^3 < 2^-65, so that about one result in 10^5 differs
// from the IEEE quotient, by one unit, and none is off by more than 0.501 ulp
// (the 20-bit FP64 seed left 2^-60: one result in 100).  The seed's conversions
// run on the integer pipe.  Operands or results outside FP32's normal range,
// zeros, infinities and NaN take the division.
__device__ __noinline__ static double rcp_f64_slow(double x) { return 1.0 / x; }
__device__ __forceinline__ double rcp_f64(double x) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    if (((hi >> 20) & 0x7ffu) - 899u >= 249u) return rcp_f64_slow(x);  // |x| in [2^-124, 2^125)
    const uint32_t m = __funnelshift_l(lo, hi, 3);  // exponent and leading 23 bits, FP64's bias
    const uint32_t s = __float_as_uint(
        rcp_approx(__uint_as_float(((m - 0xc0000000u) & 0x7fffffffu) | (hi & 0x80000000u))));
    const double r = __hiloint2double(
        (int)((s & 0x80000000u) | (((s & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(s << 29));
    const double e = fma(-x, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

struct F2 {
    float2 v;
    F2() = default;
    __device__ __forceinline__ constexpr F2(float a) : v{a, a} {}
    __device__ __forceinline__ constexpr F2(float a, float b) : v{a, b} {}
    __device__ __forceinline__ F2(float2 a) : v(a) {}
};
__device__ __forceinline__ F2 operator+(F2 a, F2 b) { return F2(__fadd2_rn(a.v, b.v)); }
__device__ __forceinline__ F2 operator-(F2 a) { return F2(-a.v.x, -a.v.y); }
__device__ __forceinline__ F2 operator-(F2 a, F2 b) {
    return F2(__fadd2_rn(a.v, make_float2(-b.v.x, -b.v.y)));
}
__device__ __forceinline__ F2 operator*(F2 a, F2 b) { return F2(__fmul2_rn(a.v, b.v)); }

// Per-lane predicate.
struct B2 {
    bool x, y;
};

template <typename T> struct Num;

template <> struct Num<double> {
    using Pred = bool;
    static constexpr int LANES = 1;
    __device__ static __forceinline__ double mad(double a, double b, double c) { return fma(a, b, c); }
    __device__ static __forceinline__ double rcp(double x) { return rcp_f64(x); }
    __device__ static __forceinline__ double lane(double v, int) { return v; }
    __device__ static __forceinline__ void set_lane(double& v, int, double x) { v = x; }
};

template <> struct Num<F2> {
    using Pred = B2;
    static constexpr int LANES = 2;
    static constexpr float LOG_SCALE = 0.693147180559945309f;
    __device__ static __forceinline__ F2 mad(F2 a, F2 b, F2 c) { return F2(__ffma2_rn(a.v, b.v, c.v)); }
    __device__ static __forceinline__ F2 rcp(F2 x) { return F2(rcp_approx(x.v.x), rcp_approx(x.v.y)); }
    __device__ static __forceinline__ F2 lnp(F2, F2 y) { return F2(lg2_approx(y.v.x), lg2_approx(y.v.y)); }
    __device__ static __forceinline__ F2 vmin(F2 a, F2 b) {
        return F2(fminf(a.v.x, b.v.x), fminf(a.v.y, b.v.y));
    }
    __device__ static __forceinline__ Pred gt(F2 a, F2 b) { return {a.v.x > b.v.x, a.v.y > b.v.y}; }
    __device__ static __forceinline__ F2 sel(Pred p, F2 a, F2 b) {
        return F2(p.x ? a.v.x : b.v.x, p.y ? a.v.y : b.v.y);
    }
    __device__ static __forceinline__ float lane(F2 v, int i) { return i ? v.v.y : v.v.x; }
    __device__ static __forceinline__ void set_lane(F2& v, int i, float x) {
        if (i) v.v.y = x;
        else v.v.x = x;
    }
};

// Scalar type of one lane.
template <typename T> struct LaneOf { using type = T; };
template <> struct LaneOf<F2> { using type = float; };

// 4x4 symmetric positive definite solve A x = b by an LDL^T factorisation:
// A = L D L^T with unit lower-triangular L, then L z = b, x = L^-T D^-1 z.
// Four reciprocals (of the pivots) and 32 multiply-adds; A is given as its
// 10 unique entries, unknown order (1, 2, 3, 4).
template <typename T>
__device__ __forceinline__ void spd4_solve(T a11, T a21, T a22, T a31, T a32, T a33, T a41, T a42,
                                           T a43, T a44, T b1, T b2, T b3, T b4, T& x1, T& x2,
                                           T& x3, T& x4) {
    using N = Num<T>;
    const T r1 = N::rcp(a11);
    const T l21 = a21 * r1, l31 = a31 * r1, l41 = a41 * r1;
    const T r2 = N::rcp(N::mad(-l21, a21, a22));
    const T t32 = N::mad(-l31, a21, a32), t42 = N::mad(-l41, a21, a42);
    const T l32 = t32 * r2, l42 = t42 * r2;
    const T r3 = N::rcp(N::mad(-l32, t32, N::mad(-l31, a31, a33)));
    const T t43 = N::mad(-l42, t32, N::mad(-l41, a31, a43));
    const T l43 = t43 * r3;
    const T r4 = N::rcp(N::mad(-l43, t43, N::mad(-l42, t42, N::mad(-l41, a41, a44))));
    const T z2 = N::mad(-l21, b1, b2);
    const T z3 = N::mad(-l32, z2, N::mad(-l31, b1, b3));
    const T z4 = N::mad(-l43, z3, N::mad(-l42, z2, N::mad(-l41, b1, b4)));
    x4 = z4 * r4;
    x3 = N::mad(-l43, x4, z3 * r3);
    x2 = N::mad(-l42, x4, N::mad(-l32, x3, z2 * r2));
    x1 = N::mad(-l41, x4, N::mad(-l31, x3, N::mad(-l21, x2, b1 * r1)));
}

}  // namespace lbm
