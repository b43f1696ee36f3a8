// The hopping term at FP64 accuracy on the integer pipe.
//
// GB300 issues 2 FP64 multiply-adds per clock and SM but 64 widening 32 x 32 + 64 bit
// integer multiply-adds (measured: 2.0 and 64.7), and the hopping term in FP64 arithmetic
// ran at 0.9 of the FP64 pipe (2.10 ms per launch of 1.33 M site-columns).  Here a spinor is
// held in block fixed point, one exponent per site-column, and the SU(3) products are sums of
// integer products:
//
//   spinor component  v = F 2^(E - 56),  |v| < 2^E at every component of the site-column,
//                     F = F1 2^28 + F0,  F0 in [-2^27, 2^27),  |F1| <= 2^28
//   link entry        u = U 2^-57,       U = U1 2^28 + U0,     U0 in [-2^27, 2^27),  |U1| <= 2^29
//   u v               = [U1 F1 + (U1 F0 + U0 F1) 2^-28 + U0 F0 2^-56] 2^(E - 57)
//
// Three multiply-adds per real product, exact in 64 bits over the six products of an output
// component (|F| doubles in the spin projection: sums below 2^61); U0 F0, of random sign and
// below 2^-58 of the largest term, is left out.  A hop's result, w in units of 2^(E - 57), is
// shifted to the largest exponent of the eight neighbours and added; |sum| < 2^62.4.  Every step
// is exact but the shifts, which round to nearest: half a unit each, about 2^-57 of the largest
// component of the neighbours in all, where a chain of FP64 multiply-adds makes 2^-53 of each
// partial sum.  Against quad precision (relative, a 5x5x4x4 box, neighbouring time slices alike
// or a factor e^3 apart): one application 0.75e-16, FP64 arithmetic 1.5e-16; eighth power
// 1.6e-16, FP64 arithmetic 2.2e-16.  These are errors against the norm: a component that is smaller
// than the largest of its site-column and of the eight neighbours by a factor f keeps 57 - log2(f)
// bits, and none from f = 2^57 on.  With links that mix colours and spins every output component
// holds products of the largest one, whose rounding in FP64 arithmetic is 2^-53; only where such
// products vanish (links with zeros) would FP64 arithmetic keep more of the small ones.
//
// A site-column that holds a NaN or an infinity keeps its raw doubles under the exponent
// FX_RAW, and an output with such a neighbour is evaluated in FP64 arithmetic (fx_slow), so that
// non-finite values spread exactly as in plain arithmetic.
#pragma once

#include "ddp_device.cuh"

namespace ddp {

// Storage: 12 chunks of int4 (re F1, re F0, im F1, im F0), one complex component each, chunk-major
// like the other formats; the exponents are in FieldView::scale, as 32-bit integers.
struct PFX {
    using chunk = int4;
    static constexpr int NCH = 12;
    static constexpr bool SCALED = true;
};

constexpr int FX_BITS = 56;          // |F| <= 2^FX_BITS
constexpr int FX_LIMB = 28;
constexpr int FX_LINK = 57;          // units of a link entry: 2^-FX_LINK
constexpr int FX_ZERO = -(1 << 16);  // exponent of a site-column of zeros
constexpr int FX_RAW = 1 << 16;      // the chunks hold doubles (some of them not finite)

__device__ __forceinline__ int *fx_exponents(const FieldView &f) { return reinterpret_cast<int *>(f.scale); }

// N = N1 2^28 + N0, N0 in [-2^27, 2^27).
__device__ __forceinline__ void fx_split(long long n, int &n1, int &n0) {
    n1 = (int)((n + (1ll << (FX_LIMB - 1))) >> FX_LIMB);
    n0 = ((int)n << (32 - FX_LIMB)) >> (32 - FX_LIMB);
}
__device__ __forceinline__ long long fx_join(int n1, int n0) { return (long long)n1 * (1 << FX_LIMB) + n0; }

// round(v 2^(k + 1075 - max(1, e))) for a finite v with biased exponent e, i.e. its significand
// shifted left by k (right for k < 0); |result| < 2^63 by the caller's choice of k.
__device__ __forceinline__ long long fx_shifted(double v, int k) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const unsigned long long m = (b & ((1ull << 52) - 1)) | ((b << 1) >> 53 ? 1ull << 52 : 0ull);
    unsigned long long n;
    if (k >= 0)
        n = m << k;
    else if (k > -60)
        n = (m + (1ull << (-k - 1))) >> -k;
    else
        n = 0;
    return (long long)b < 0 ? -(long long)n : (long long)n;
}
__device__ __forceinline__ int fx_biased(double v) { return (__double2hiint(v) >> 20) & 0x7FF; }

// A link entry (|u| < 2) in units of 2^-57.
__device__ __forceinline__ long long fx_link(double u) {
    return fx_shifted(u, max(1, fx_biased(u)) - 1075 + FX_LINK);
}

// The double nearest a 2^e.
__device__ __forceinline__ double fx_value(long long a, int e) {
    if (a == 0) return 0.0;
    const unsigned long long m = a < 0 ? 0ull - (unsigned long long)a : (unsigned long long)a;
    const int lz = __clzll((long long)m);
    const int be = 63 - lz + e + 1023;   // biased exponent
    if (be < 1 || be > 2045) return ldexp((double)a, e);
    const unsigned long long t = m << lz;
    const unsigned long long s = (t >> 11) + ((t >> 10) & 1);  // 53 bits, or 2^53: the carry moves on
    const unsigned long long r = ((unsigned long long)(be - 1) << 52) + s;
    return __longlong_as_double((long long)(r | ((unsigned long long)a & (1ull << 63))));
}

// The site-column v in block fixed point.
__device__ __forceinline__ void fx_store_doubles(const FieldView &f, int64_t i, const double v[24]) {
    int top = 0;  // largest biased exponent, 0 if every component is zero
    bool any = false;
#pragma unroll
    for (int j = 0; j < 24; j++) {
        top = max(top, fx_biased(v[j]));
        any = any || ((__double_as_longlong(v[j]) << 1) != 0);
    }
    int4 *b = reinterpret_cast<int4 *>(f.p);
    if (top == 0x7FF) {
        fx_exponents(f)[i] = FX_RAW;
#pragma unroll
        for (int j = 0; j < 12; j++)
            b[j * f.stride + i] = make_int4(__double2loint(v[2 * j]), __double2hiint(v[2 * j]),
                                            __double2loint(v[2 * j + 1]), __double2hiint(v[2 * j + 1]));
        return;
    }
    top = max(top, 1);
    fx_exponents(f)[i] = any ? top - 1022 : FX_ZERO;
#pragma unroll
    for (int j = 0; j < 12; j++) {
        int4 c;
        fx_split(fx_shifted(v[2 * j], FX_BITS - 53 - (top - max(1, fx_biased(v[2 * j])))), c.x, c.y);
        fx_split(fx_shifted(v[2 * j + 1], FX_BITS - 53 - (top - max(1, fx_biased(v[2 * j + 1])))), c.z, c.w);
        b[j * f.stride + i] = c;
    }
}

// A site-column as doubles.
__device__ __forceinline__ void fx_load_doubles(const FieldView &f, int64_t i, double v[24]) {
    const int4 *b = reinterpret_cast<const int4 *>(f.p);
    const int E = fx_exponents(f)[i];
#pragma unroll
    for (int j = 0; j < 12; j++) {
        const int4 c = b[j * f.stride + i];
        if (E == FX_RAW) {
            v[2 * j] = __hiloint2double(c.y, c.x);
            v[2 * j + 1] = __hiloint2double(c.w, c.z);
        } else {
            v[2 * j] = fx_value(fx_join(c.x, c.y), E - FX_BITS);
            v[2 * j + 1] = fx_value(fx_join(c.z, c.w), E - FX_BITS);
        }
    }
}

// The sums acc 2^e of an output site-column, normalised to block fixed point.
__device__ __forceinline__ void fx_store_sums(const FieldView &f, int64_t i, const long long acc[24], int e) {
    unsigned long long any = 0;
#pragma unroll
    for (int j = 0; j < 24; j++) any |= (unsigned long long)(acc[j] ^ (acc[j] >> 63));
    // |acc| <= 2^len at every component
    const int len = any ? 64 - __clzll((long long)any) : 0;
    int4 *b = reinterpret_cast<int4 *>(f.p);
    bool zero = true;
#pragma unroll
    for (int j = 0; j < 24; j++) zero = zero && acc[j] == 0;
    fx_exponents(f)[i] = zero ? FX_ZERO : e + len;
    const int s = len - FX_BITS;
    const long long half = s > 0 ? 1ll << (s - 1) : 0;
#pragma unroll
    for (int j = 0; j < 12; j++) {
        int4 c;
        fx_split(s > 0 ? (acc[2 * j] + half) >> s : acc[2 * j] << -s, c.x, c.y);
        fx_split(s > 0 ? (acc[2 * j + 1] + half) >> s : acc[2 * j + 1] << -s, c.z, c.w);
        b[j * f.stride + i] = c;
    }
}

// One half-spinor component in two limbs.
struct FxC {
    int r1, r0, i1, i0;
};
__device__ __forceinline__ FxC fx_add(const int4 &a, const int4 &b) {
    return {a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w};
}
__device__ __forceinline__ FxC fx_sub(const int4 &a, const int4 &b) {
    return {a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w};
}
__device__ __forceinline__ FxC fx_add_i(const int4 &a, const int4 &b) {  // a + i b
    return {a.x - b.z, a.y - b.w, a.z + b.x, a.w + b.y};
}
__device__ __forceinline__ FxC fx_sub_i(const int4 &a, const int4 &b) {  // a - i b
    return {a.x + b.z, a.y + b.w, a.z - b.x, a.w - b.y};
}

// acc += [w; lower(w)] 2^-sh, w = u h, h the spin projection of hop D (as project() and
// accumulate() have it).  acc component 3 s + a, re and im.
template <int D>
__device__ __forceinline__ void fx_hop_step(const int4 v[12], const int4 *u, long long acc[24], int sh) {
    constexpr int MU = D >> 1;
    constexpr bool FWD = !(D & 1);
    constexpr long long FX_HALF = 1ll << (FX_LIMB - 1);
    const long long half = (1ll << sh) >> 1;
    FxC h[2][3];
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const int4 &p0 = v[a], &p1 = v[3 + a], &p2 = v[6 + a], &p3 = v[9 + a];
        if (MU == 0) {
            h[0][a] = FWD ? fx_sub(p0, p2) : fx_add(p0, p2);
            h[1][a] = FWD ? fx_sub(p1, p3) : fx_add(p1, p3);
        } else if (MU == 1) {
            h[0][a] = FWD ? fx_add_i(p0, p3) : fx_sub_i(p0, p3);
            h[1][a] = FWD ? fx_add_i(p1, p2) : fx_sub_i(p1, p2);
        } else if (MU == 2) {
            h[0][a] = FWD ? fx_add(p0, p3) : fx_sub(p0, p3);
            h[1][a] = FWD ? fx_sub(p1, p2) : fx_add(p1, p2);
        } else {
            h[0][a] = FWD ? fx_add_i(p0, p2) : fx_sub_i(p0, p2);
            h[1][a] = FWD ? fx_sub_i(p1, p3) : fx_add_i(p1, p3);
        }
    }
#pragma unroll
    for (int a = 0; a < 3; a++) {
        // both shifts round to nearest: the halves are the sums' initial values
        long long hr[2] = {half, half}, hi[2] = {half, half};
        long long mr[2] = {FX_HALF, FX_HALF}, mi[2] = {FX_HALF, FX_HALF};
#pragma unroll
        for (int b = 0; b < 3; b++) {
            const int4 c = u[3 * a + b];
            const int n1 = -c.z, n0 = -c.w;
#pragma unroll
            for (int s = 0; s < 2; s++) {
                const FxC &x = h[s][b];
                hr[s] += (long long)c.x * x.r1;
                hr[s] += (long long)n1 * x.i1;
                mr[s] += (long long)c.x * x.r0;
                mr[s] += (long long)c.y * x.r1;
                mr[s] += (long long)n1 * x.i0;
                mr[s] += (long long)n0 * x.i1;
                hi[s] += (long long)c.x * x.i1;
                hi[s] += (long long)c.z * x.r1;
                mi[s] += (long long)c.x * x.i0;
                mi[s] += (long long)c.y * x.i1;
                mi[s] += (long long)c.z * x.r0;
                mi[s] += (long long)c.w * x.r1;
            }
        }
        long long wr[2], wi[2];
#pragma unroll
        for (int s = 0; s < 2; s++) {
            wr[s] = (hr[s] + (mr[s] >> FX_LIMB)) >> sh;
            wi[s] = (hi[s] + (mi[s] >> FX_LIMB)) >> sh;
        }
#define FX_RE(s) acc[2 * (3 * (s) + a)]
#define FX_IM(s) acc[2 * (3 * (s) + a) + 1]
        FX_RE(0) += wr[0];
        FX_IM(0) += wi[0];
        FX_RE(1) += wr[1];
        FX_IM(1) += wi[1];
        if (MU == 0) {  // -+ w
            FX_RE(2) += FWD ? -wr[0] : wr[0];
            FX_IM(2) += FWD ? -wi[0] : wi[0];
            FX_RE(3) += FWD ? -wr[1] : wr[1];
            FX_IM(3) += FWD ? -wi[1] : wi[1];
        } else if (MU == 1) {  // -+ i (w1, w0)
            FX_RE(2) += FWD ? wi[1] : -wi[1];
            FX_IM(2) += FWD ? -wr[1] : wr[1];
            FX_RE(3) += FWD ? wi[0] : -wi[0];
            FX_IM(3) += FWD ? -wr[0] : wr[0];
        } else if (MU == 2) {  // -+ w1, +- w0
            FX_RE(2) += FWD ? -wr[1] : wr[1];
            FX_IM(2) += FWD ? -wi[1] : wi[1];
            FX_RE(3) += FWD ? wr[0] : -wr[0];
            FX_IM(3) += FWD ? wi[0] : -wi[0];
        } else {  // -+ i w0, +- i w1
            FX_RE(2) += FWD ? wi[0] : -wi[0];
            FX_IM(2) += FWD ? -wr[0] : wr[0];
            FX_RE(3) += FWD ? -wi[1] : wi[1];
            FX_IM(3) += FWD ? wr[1] : -wr[1];
        }
#undef FX_RE
#undef FX_IM
    }
}

// The hopping sum of one output in FP64 arithmetic, for outputs with a non-finite neighbour.
// nb[d * TS], u[(d * TS) * 9]: neighbour and link of hop d of the site.
template <int TS>
__device__ __noinline__ void fx_slow(const FieldView &in, int64_t cb, const int *nb, const int4 *u, double out[24]) {
    cx<double> acc[4][3];
    for (int s = 0; s < 4; s++)
        for (int c = 0; c < 3; c++) acc[s][c] = mk(0.0, 0.0);
    for (int d = 0; d < 8; d++) {
        const int k = nb[d * TS];
        if (k < 0) continue;
        double v[24];
        fx_load_doubles(in, cb + k, v);
        cx<double> l[3][3];
        for (int j = 0; j < 9; j++) {
            const int4 c = u[d * TS * 9 + j];
            l[j / 3][j % 3] = mk(fx_value(fx_join(c.x, c.y), -FX_LINK), fx_value(fx_join(c.z, c.w), -FX_LINK));
        }
        switch (d) {
            case 0: hop_step<0>(v, l, acc, 1.0); break;
            case 1: hop_step<1>(v, l, acc, 1.0); break;
            case 2: hop_step<2>(v, l, acc, 1.0); break;
            case 3: hop_step<3>(v, l, acc, 1.0); break;
            case 4: hop_step<4>(v, l, acc, 1.0); break;
            case 5: hop_step<5>(v, l, acc, 1.0); break;
            case 6: hop_step<6>(v, l, acc, 1.0); break;
            default: hop_step<7>(v, l, acc, 1.0); break;
        }
    }
    for (int j = 0; j < 12; j++) {
        out[2 * j] = acc[j / 3][j % 3].re;
        out[2 * j + 1] = acc[j / 3][j % 3].im;
    }
}

}  // namespace ddp
