// Scalar recurrences of BiCGStab (van der Vorst) in FP64 or in double-FP32.
//
// The FP64 storage format computes its sums and scalars in FP64.  The low-precision formats use
// double-FP32 (48 bits, ddfloat.cuh) beyond the FP32 sum of a tile's 32 sites: GB300 issues two
// FP64 operations per clock and SM, so that the sums over tiles and the divisions of one iteration
// took 15.8 + 5.3 us for 12 columns of 16x24^3 in FP64 (k_fin of (t, s) and of (rh, v)), 6.6 + 3.9
// in double-FP32, and the vector updates no longer convert their scalars from FP64 in every thread
// (FP16 x, r, p update 98 -> 82 us).  The summands are good to 24 bits and the results are rounded
// to FP32 when used.
#pragma once

#include "ddfloat.cuh"

namespace ddp {

template <typename R>
struct ScalarOf {  // of a format that computes in R
    using type = double;
};
template <>
struct ScalarOf<float> {
    using type = dd;
};

__device__ __forceinline__ double nadd(double a, double b) { return a + b; }
__device__ __forceinline__ double nsub(double a, double b) { return a - b; }
__device__ __forceinline__ double nmul(double a, double b) { return a * b; }
__device__ __forceinline__ double ndiv(double a, double b) { return a / b; }
__device__ __forceinline__ bool nfinite(double a) { return isfinite(a); }
__device__ __forceinline__ bool npositive(double a) { return a > 0; }
__device__ __forceinline__ bool nzero(double a) { return a == 0; }
__device__ __forceinline__ dd nadd(dd a, dd b) { return dd_add(a, b); }
__device__ __forceinline__ dd nsub(dd a, dd b) { return dd_sub(a, b); }
__device__ __forceinline__ dd nmul(dd a, dd b) { return dd_mul(a, b); }
// a / b to about 2^-45: the FP32 quotient and that of the remainder
__device__ __forceinline__ dd ndiv(dd a, dd b) {
    const float q = a.hi / b.hi;
    const dd r = dd_sub(a, dd_mul(dd(q, 0.f), b));
    return dd_renorm(q, r.hi / b.hi);
}
__device__ __forceinline__ bool nfinite(dd a) { return isfinite(a.hi); }
__device__ __forceinline__ bool npositive(dd a) { return a.hi > 0.f; }
__device__ __forceinline__ bool nzero(dd a) { return a.hi == 0.f; }

// A summand joins a running sum (nsum_end: the low part of a double-FP32 sum is renormalised).
__device__ __forceinline__ void nsum(double &s, double v) { s += v; }
__device__ __forceinline__ void nsum_end(double &) {}
__device__ __forceinline__ void nsum(dd &s, float v) {
    const float t = __fadd_rn(s.hi, v), b = __fsub_rn(t, s.hi);
    s.lo = __fadd_rn(s.lo, __fadd_rn(__fsub_rn(s.hi, __fsub_rn(t, b)), __fsub_rn(v, b)));
    s.hi = t;
}
__device__ __forceinline__ void nsum_end(dd &s) { s = dd_renorm(s.hi, s.lo); }

__device__ __forceinline__ double nshfl_xor(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ dd nshfl_xor(dd a, int o) {
    return dd(__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o));
}
__device__ __forceinline__ double nshfl(double a, int l) { return __shfl_sync(0xffffffffu, a, l); }
__device__ __forceinline__ dd nshfl(dd a, int l) {
    return dd(__shfl_sync(0xffffffffu, a.hi, l), __shfl_sync(0xffffffffu, a.lo, l));
}
__device__ __forceinline__ void nset(double &a, double v) { a = v; }
__device__ __forceinline__ void nset(dd &a, double v) { a = dd_of(v); }

template <class T>
struct Cnum {
    T re, im;
};
template <class T>
__device__ __forceinline__ Cnum<T> cn_mul(Cnum<T> a, Cnum<T> b) {
    return {nsub(nmul(a.re, b.re), nmul(a.im, b.im)), nadd(nmul(a.re, b.im), nmul(a.im, b.re))};
}
__device__ __forceinline__ Cnum<double> cn_div(Cnum<double> a, Cnum<double> b) {
    const double d = b.re * b.re + b.im * b.im;
    return {(a.re * b.re + a.im * b.im) / d, (a.im * b.re - a.re * b.im) / d};
}
__device__ __forceinline__ Cnum<dd> cn_div(Cnum<dd> a, Cnum<dd> b) {
    // b scaled by a power of two, so that its square stays in range
    const int e = 127 - (int)((__float_as_uint(fmaxf(fabsf(b.re.hi), fabsf(b.im.hi))) >> 23) & 0xFF);
    const float f = __int_as_float((127 + max(-126, min(126, e))) << 23);
    b = {dd_scale2(b.re, f), dd_scale2(b.im, f)};
    const dd n = dd_add(dd_mul(b.re, b.re), dd_mul(b.im, b.im));
    const Cnum<dd> c = cn_mul(a, Cnum<dd>{b.re, dd_neg(b.im)});
    return {dd_scale2(ndiv(c.re, n), f), dd_scale2(ndiv(c.im, n), f)};
}
template <class T>
__device__ __forceinline__ bool cn_zero(Cnum<T> a) { return nzero(a.re) && nzero(a.im); }
template <class T>
__device__ __forceinline__ bool cn_finite(Cnum<T> a) { return nfinite(a.re) && nfinite(a.im); }

// alpha = rho / (rh, v); false: the recurrence has broken down.
template <class T>
__device__ __forceinline__ bool bicg_alpha(Cnum<T> rho, Cnum<T> hv, Cnum<T> &alpha) {
    if (cn_zero(hv) || !cn_finite(hv)) return false;
    alpha = cn_div(rho, hv);
    return true;
}

// omega and, before r is formed, the scalars of the next iteration, from the products
// w = (t, s), (rh, s), (rh, t), (t, t), (s, s) of the (t, s) stencil: with r = s - omega t,
//   rc = (rh, r) = (rh, s) - omega (rh, t),   rr = (r, r) = (s, s) - |(t, s)|^2 / (t, t).
// Returns 1 when the column has converged, 2 when the recurrence has broken down, 0 to go on.
template <class T>
__device__ __forceinline__ int bicg_omega(const T w[8], T target2, Cnum<T> &omega, Cnum<T> &rc) {
    const Cnum<T> ts = {w[0], w[1]}, hs = {w[2], w[3]}, ht = {w[4], w[5]};
    T zero;
    nset(zero, 0.0);
    omega = {zero, zero};
    T rr = w[7];
    if (npositive(w[6])) {
        omega = {ndiv(ts.re, w[6]), ndiv(ts.im, w[6])};
        rr = nsub(rr, nadd(nmul(ts.re, omega.re), nmul(ts.im, omega.im)));
    }
    const Cnum<T> m = cn_mul(omega, ht);
    rc = {nsub(hs.re, m.re), nsub(hs.im, m.im)};
    if (nfinite(rr) && !npositive(nsub(rr, target2))) return 1;
    return cn_zero(rc) || cn_zero(omega) || !cn_finite(rc) || !nfinite(rr) ? 2 : 0;
}

// beta = (rc / rho) (alpha / omega)
template <class T>
__device__ __forceinline__ Cnum<T> bicg_beta(Cnum<T> rc, Cnum<T> rho, Cnum<T> alpha, Cnum<T> omega) {
    return cn_div(cn_mul(rc, alpha), cn_mul(rho, omega));
}

}  // namespace ddp
