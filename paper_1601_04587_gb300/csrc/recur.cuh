// Scalar recurrences of BiCGStab (van der Vorst) in FP64, and the sums they start from.
//
// A tile's 32 sites are summed in the compute precision of the storage format; the sums over tiles
// and the recurrences are FP64, or more.  GB300 issues two FP64 operations per clock and SM, so the
// sums over tiles of FP32 values are formed on the FP32 pipe, in three floats: every addition is
// split exactly (Knuth's two-sum) and only the third float, about 2^-48 of the sum, is rounded, 2^-72
// where FP64 has 2^-53.  One conversion to FP64 at the end.  The recurrences are FP64 operations of
// one lane, with reciprocals in the place of divisions and both of an iteration's second half
// started from the sums; their results are stored in FP32 beside the FP64 scalars, so that the
// vector updates convert nothing.  k_fin of (t, s) and of (rh, v), 12 columns of 16x24^3: 15.8 + 5.3
// us with FP64 sums, one launch after another; chained (where a duration holds the wait for the
// kernel before) 13.8 + 9.8 so, 11.6 + 9.0 with sums and scalars of 48 bits, which is less than the
// reductions are to have.  The whole 8^4 propagator 2.49 / 2.56 ms with 48 bits / so, 16x24^3 in FP16
// the same to 0.2%; the columns come out bit for bit alike in most solves.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#define DDP_HD __host__ __device__ __forceinline__

namespace ddp {

struct Sum3 {
    float hi, mid, lo;
};

template <typename R>
struct SumOf {  // the sum of values of type R
    using type = double;
};
template <>
struct SumOf<float> {
    using type = Sum3;
};

// s + e = a + b exactly, s = a + b rounded (sums only: nothing to contract)
DDP_HD void two_sum(float a, float b, float &s, float &e) {
    s = a + b;
    const float t = s - a;
    e = (a - (s - t)) + (b - t);
}

DDP_HD void sum_zero(double &s) { s = 0.0; }
DDP_HD void sum_zero(Sum3 &s) { s = {0.f, 0.f, 0.f}; }
// s += v
DDP_HD void sum_add(double &s, double v) { s += v; }
DDP_HD void sum_add(Sum3 &s, float v) {
    float h, m, e;
    two_sum(s.hi, v, h, e);
    s.hi = h;
    two_sum(s.mid, e, m, e);
    s.mid = m;
    s.lo += e;
}
DDP_HD double sum_join(double a, double b) { return a + b; }
DDP_HD Sum3 sum_join(const Sum3 &a, const Sum3 &b) {
    Sum3 s;
    float e, f, g, m;
    two_sum(a.hi, b.hi, s.hi, e);
    two_sum(a.mid, b.mid, m, f);
    two_sum(m, e, s.mid, g);
    s.lo = (a.lo + b.lo) + (f + g);
    return s;
}
// Every FP64 instruction of a warp, conversions and comparisons among them, takes 16 clocks of the
// SM's FP64 pipe, whatever the number of active lanes: what integers can do, they do here.
// A float as a double.
DDP_HD double wide(float w) {
#ifdef __CUDA_ARCH__
    const unsigned u = __float_as_uint(w), e = (u >> 23) & 0xFF;
    if (e - 1u < 254u) return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7FFFFFFFu) >> 3) + 0x38000000u)), (int)(u << 29));
    return (u << 1) == 0 ? 0.0 : (double)w;
#else
    return (double)w;
#endif
}
// The bits of a double, and three questions to them.
DDP_HD unsigned long long bits_of(double v) {
#ifdef __CUDA_ARCH__
    return (unsigned long long)__double_as_longlong(v);
#else
    unsigned long long b;
    memcpy(&b, &v, sizeof(b));
    return b;
#endif
}
DDP_HD bool is_zero(double v) { return (bits_of(v) << 1) == 0; }
DDP_HD bool is_finite(double v) { return ((bits_of(v) >> 52) & 0x7FF) != 0x7FF; }
DDP_HD bool is_positive(double v) { return bits_of(v) - 1 < 0x7FF0000000000000ull; }  // infinity among them
DDP_HD double sum_value(double s) { return s; }
DDP_HD double sum_value(const Sum3 &s) {
    // a sum that is not finite has no parts
    return isfinite(s.hi) ? wide(s.hi) + (wide(s.mid) + wide(s.lo)) : (double)s.hi;
}
__device__ __forceinline__ double sum_shfl_xor(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ Sum3 sum_shfl_xor(const Sum3 &a, int o) {
    return {__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.mid, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
}

using Cnum = double2;
DDP_HD Cnum cn(double re, double im) { return make_double2(re, im); }
DDP_HD Cnum cn_mul(Cnum a, Cnum b) { return cn(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
DDP_HD Cnum cn_mulc(Cnum a, Cnum b) { return cn(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y); }  // a conj(b)
DDP_HD Cnum cn_scale(Cnum a, double r) { return cn(a.x * r, a.y * r); }
DDP_HD double cn_norm(Cnum a) { return a.x * a.x + a.y * a.y; }
DDP_HD bool cn_zero(Cnum a) { return is_zero(a.x) && is_zero(a.y); }
DDP_HD bool cn_finite(Cnum a) { return is_finite(a.x) && is_finite(a.y); }

// alpha = rho / (rh, v), and inv = 1 / (rh, v) for bicg_omega; false: the recurrence has broken down.
DDP_HD bool bicg_alpha(Cnum rho, Cnum hv, Cnum &alpha, Cnum &inv) {
    if (cn_zero(hv) || !cn_finite(hv)) return false;
    const double r = 1.0 / cn_norm(hv);
    inv = cn(hv.x * r, -hv.y * r);
    alpha = cn_mul(rho, inv);
    return true;
}

// omega and, before r is formed, the scalars of the next iteration, from the products
// w = (t, s), (rh, s), (rh, t), (t, t), (s, s) of the (t, s) stencil: with r = s - omega t,
//   rc = (rh, r) = (rh, s) - omega (rh, t),   rr = (r, r) = (s, s) - |(t, s)|^2 / (t, t),
//   beta = (rc / rho) (alpha / omega) = rc inv / omega,   1 / omega = (t, t) conj((t, s)) / |(t, s)|^2,
// so that both reciprocals start from the sums at once.
// The errors of rc and rr are those of the products, 2^-24 of |rh| |s| and (s, s) in the
// low-precision formats, where sums over r itself would have 2^-24 of |rh| |r| and (r, r): omega
// minimises |r|, so |r| < |s|, and what is lost is the factor by which this half step shrinks the
// residual, once and not over the iterations.  (rh, s) is zero but for rounding (alpha makes it so),
// and rr only ends the inner loop: the FP64 true residual of the outer cycle decides convergence.
// Returns 1 when the column has converged, 2 when the recurrence has broken down, 0 to go on.
DDP_HD int bicg_omega(const double w[8], double target2, Cnum inv, Cnum &omega, Cnum &rc, Cnum &beta) {
    const Cnum ts = cn(w[0], w[1]);
    const double tt = w[6], n = cn_norm(ts);
    const Cnum g = cn_scale(cn_mulc(inv, ts), tt * (1.0 / n));
    omega = cn(0.0, 0.0);
    double rr = w[7];
    if (is_positive(tt)) {
        const double r = 1.0 / tt;
        omega = cn_scale(ts, r);
        rr -= n * r;
    }
    const Cnum m = cn_mul(omega, cn(w[4], w[5]));
    rc = cn(w[2] - m.x, w[3] - m.y);
    beta = cn_mul(rc, g);
    if (is_finite(rr) && rr <= target2) return 1;
    return cn_zero(rc) || cn_zero(omega) || !cn_finite(rc) || !is_finite(rr) ? 2 : 0;
}

}  // namespace ddp
