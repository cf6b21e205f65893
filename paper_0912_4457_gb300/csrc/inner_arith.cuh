// Arithmetic of the inner part on T = double (real, the Hermitian case) or
// double2 (complex): the helpers that inner_lanczos.cu and inner.cu share.
#pragma once

#include "nk_common.cuh"

namespace nk {

__device__ __forceinline__ double t_zero(double) { return 0.0; }
__device__ __forceinline__ double2 t_zero(double2) { return mk(0.0, 0.0); }
__device__ __forceinline__ double t_one(double) { return 1.0; }
__device__ __forceinline__ double2 t_one(double2) { return mk(1.0, 0.0); }
__device__ __forceinline__ double t_from(double2 a, double) { return a.x; }
__device__ __forceinline__ double2 t_from(double2 a, double2) { return a; }
__device__ __forceinline__ double2 t_to2(double a) { return mk(a, 0.0); }
__device__ __forceinline__ double2 t_to2(double2 a) { return a; }
__device__ __forceinline__ double t_conj(double a) { return a; }
__device__ __forceinline__ double2 t_conj(double2 a) { return cconj(a); }
__device__ __forceinline__ double t_mul(double a, double b) { return a * b; }
__device__ __forceinline__ double2 t_mul(double2 a, double2 b) { return cmul(a, b); }
__device__ __forceinline__ double t_add(double a, double b) { return a + b; }
__device__ __forceinline__ double2 t_add(double2 a, double2 b) { return cadd(a, b); }
__device__ __forceinline__ double t_sub(double a, double b) { return a - b; }
__device__ __forceinline__ double2 t_sub(double2 a, double2 b) { return csub(a, b); }
__device__ __forceinline__ double t_scale(double a, double s) { return a * s; }
__device__ __forceinline__ double2 t_scale(double2 a, double s) { return cscale(a, s); }
__device__ __forceinline__ double t_neg(double a) { return -a; }
__device__ __forceinline__ double2 t_neg(double2 a) { return mk(-a.x, -a.y); }
// a * b + c
__device__ __forceinline__ double t_fma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double2 t_fma(double2 a, double2 b, double2 c) {
    return mk(fma(a.x, b.x, fma(-a.y, b.y, c.x)), fma(a.x, b.y, fma(a.y, b.x, c.y)));
}
__device__ __forceinline__ double t_inv(double a) { return 1.0 / a; }
__device__ __forceinline__ double2 t_inv(double2 a) { return cinv(a); }
__device__ __forceinline__ double t_abs1(double a) { return fabs(a); }
__device__ __forceinline__ double t_abs1(double2 a) { return cabs1(a); }  // LAPACK CABS1
__device__ __forceinline__ double t_norm2(double a) { return a * a; }
__device__ __forceinline__ double t_norm2(double2 a) { return cnorm2(a); }
__device__ __forceinline__ bool t_iszero(double a) { return a == 0.0; }
__device__ __forceinline__ bool t_iszero(double2 a) { return a.x == 0.0 && a.y == 0.0; }
// s + conj(a) b
__device__ __forceinline__ double t_dot_add(double s, double a, double b) { return fma(a, b, s); }
__device__ __forceinline__ double2 t_dot_add(double2 s, double2 a, double2 b) {
    return mk(fma(a.x, b.x, fma(a.y, b.y, s.x)), fma(a.x, b.y, fma(-a.y, b.x, s.y)));
}

constexpr unsigned kFull = 0xffffffffu;
__device__ __forceinline__ double shup(double v, int o) { return __shfl_up_sync(kFull, v, o); }
__device__ __forceinline__ double2 shup(double2 v, int o) {
    return mk(__shfl_up_sync(kFull, v.x, o), __shfl_up_sync(kFull, v.y, o));
}
__device__ __forceinline__ double shdn(double v, int o) { return __shfl_down_sync(kFull, v, o); }
__device__ __forceinline__ double2 shdn(double2 v, int o) {
    return mk(__shfl_down_sync(kFull, v.x, o), __shfl_down_sync(kFull, v.y, o));
}
__device__ __forceinline__ double shfl_from(double v, int src) { return __shfl_sync(kFull, v, src); }
__device__ __forceinline__ double2 shfl_from(double2 v, int src) {
    return mk(__shfl_sync(kFull, v.x, src), __shfl_sync(kFull, v.y, src));
}

// 1/n for n in [1, 16): an FP32 reciprocal (its conversions on the integer
// pipe) and two Newton steps r <- r + r (1 - n r), four FP64 instructions where
// a division takes about ten.  About one ulp.
__device__ __forceinline__ double rcp_unit(double n) {
    double r = f2d_int(__frcp_rn(d2f_int(n)));
    r = fma(r, fma(-n, r, 1.0), r);
    return fma(r, fma(-n, r, 1.0), r);
}
// 1/a of a pivot.  Scaled by a power of two (exact) into the range of rcp_unit;
// complex as conj(a) / |a|^2, which then neither over- nor underflows.  Near
// the ends of the exponent range, and for zero, infinity and NaN: t_inv.
__device__ __forceinline__ double pivot_inv(double a) {
    const int e = ((__double2hiint(a) & 0x7fffffff) >> 20) - 1023;
    if (e < -1000 || e > 1000) return t_inv(a);
    const double s = pow2(-e), r = rcp_unit(fabs(a) * s) * s;
    return a < 0.0 ? -r : r;
}
__device__ __forceinline__ double2 pivot_inv(double2 a) {
    const int hx = __double2hiint(a.x) & 0x7fffffff, hy = __double2hiint(a.y) & 0x7fffffff;
    const int e = (max(hx, hy) >> 20) - 1023;
    if (e < -1000 || e > 1000) return t_inv(a);
    const double s = pow2(-e), x = a.x * s, y = a.y * s;
    const double r = rcp_unit(fma(x, x, y * y)) * s;
    return mk(x * r, -y * r);
}

// The same by a division, for the LU (its one chain has no other work beside it:
// with pivot_inv 12 two-sided RHS at k = 1024, l = 128 took the same time, Hermitian
// ones at k = 768 5.26 against 5.21 ms).
__device__ __forceinline__ double pivot_div(double a) { return 1.0 / a; }
__device__ __forceinline__ double2 pivot_div(double2 a) {
    const int hx = __double2hiint(a.x) & 0x7fffffff, hy = __double2hiint(a.y) & 0x7fffffff;
    const int e = (max(hx, hy) >> 20) - 1023;
    if (e < -1000 || e > 1000) return t_inv(a);
    const double s = pow2(-e), x = a.x * s, y = a.y * s;
    const double r = (1.0 / fma(x, x, y * y)) * s;
    return mk(x * r, -y * r);
}

// |x| as ordered bits: compares magnitudes without an FP64 comparison
__device__ __forceinline__ unsigned long long abs_bits(double x) {
    return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}

}  // namespace nk
