// Device-side building blocks of libddp: complex arithmetic, storage formats of
// spinor and link fields, the batch work table and the Dirichlet-masked
// even-odd hopping term of the Wilson-Dirac operator (App. A, Sec. 2).
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>
#include <stdint.h>

namespace ddp {

// ---------------------------------------------------------------- complex

template <typename T>
struct cx {
    T re, im;
};

template <typename T>
__device__ __forceinline__ cx<T> mk(T r, T i) {
    cx<T> c;
    c.re = r;
    c.im = i;
    return c;
}
template <typename T>
__device__ __forceinline__ cx<T> operator+(cx<T> a, cx<T> b) { return mk(a.re + b.re, a.im + b.im); }
template <typename T>
__device__ __forceinline__ cx<T> operator-(cx<T> a, cx<T> b) { return mk(a.re - b.re, a.im - b.im); }
template <typename T>
__device__ __forceinline__ cx<T> operator-(cx<T> a) { return mk(-a.re, -a.im); }
template <typename T>
__device__ __forceinline__ cx<T> operator*(cx<T> a, cx<T> b) {
    return mk(a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re);
}
template <typename T>
__device__ __forceinline__ cx<T> operator*(T s, cx<T> a) { return mk(s * a.re, s * a.im); }
// i * a and -i * a
template <typename T>
__device__ __forceinline__ cx<T> mul_i(cx<T> a) { return mk(-a.im, a.re); }
template <typename T>
__device__ __forceinline__ cx<T> mul_mi(cx<T> a) { return mk(a.im, -a.re); }
template <typename T>
__device__ __forceinline__ cx<T> conj(cx<T> a) { return mk(a.re, -a.im); }
// conj(a) * b
template <typename T>
__device__ __forceinline__ cx<T> cmul(cx<T> a, cx<T> b) {
    return mk(a.re * b.re + a.im * b.im, a.re * b.im - a.im * b.re);
}

// ------------------------------------------------------- storage formats
//
// A spinor field holds one parity of ncol columns of several domains.  Site
// component (spin s, colour a) is complex number 3 s + a, i.e. reals
// 2(3s+a), 2(3s+a)+1 of a 24-real site vector.  The field is chunk-major:
// chunk j of site-column i lives at base[j * stride + i], so that a warp
// reading 32 consecutive site-columns issues fully coalesced 16-byte loads.
//
//   FP64 : 12 chunks of double2  (one complex each)
//   FP32 :  6 chunks of float4   (two complex each)
//   FP16 :  3 chunks of 8 halves (uint4) + one float scale per site-column;
//           stored values are v / max|v| so the site's largest component is
//           exactly representable and small sites keep 11 significant bits.
//   BF16 :  3 chunks of 8 bfloat16 (uint4), no scale (FP32 exponent range).
//
// Links: FP64 keeps all 9 complex entries (9 double2 chunks per link); the
// low-precision copies keep rows 0 and 1 (6 complex) and rebuild row 2 as
// the conjugated cross product, exact for SU(3).
//   FP32 : 3 float4 chunks; FP16 / BF16 : 3 uint2 chunks (4 halves each).
// Link field layout [mu][chunk][V], sites in the global even-odd order
// parity * V/2 + (lex >> 1).

struct PF64 {
    using real = double;
    using chunk = double2;
    static constexpr int NCH = 12;
    static constexpr bool SCALED = false;
    static constexpr int LCH = 9;
    static constexpr bool IS64 = true;
};
struct PF32 {
    using real = float;
    using chunk = float4;
    static constexpr int NCH = 6;
    static constexpr bool SCALED = false;
    static constexpr int LCH = 3;
    static constexpr bool IS64 = false;
};
struct PF16 {
    using real = float;
    using chunk = uint4;
    static constexpr int NCH = 3;
    static constexpr bool SCALED = true;
    static constexpr int LCH = 3;
    static constexpr bool IS64 = false;
};
struct PBF16 {
    using real = float;
    using chunk = uint4;
    static constexpr int NCH = 3;
    static constexpr bool SCALED = false;
    static constexpr int LCH = 3;
    static constexpr bool IS64 = false;
};

struct FieldView {
    void *p;        // chunk array
    float *scale;   // per-site-column scale (FP16 only)
    int64_t stride; // chunks between consecutive chunk rows
};

__device__ __forceinline__ float2 h2f(unsigned int u) {
    __half2 h = *reinterpret_cast<__half2 *>(&u);
    return __half22float2(h);
}
__device__ __forceinline__ unsigned int f2h(float a, float b) {
    __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<unsigned int *>(&h);
}
__device__ __forceinline__ float2 b2f(unsigned int u) {
    __nv_bfloat162 h = *reinterpret_cast<__nv_bfloat162 *>(&u);
    return __bfloat1622float2(h);
}
__device__ __forceinline__ unsigned int f2b(float a, float b) {
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<unsigned int *>(&h);
}

// A load of data that kernels write: spinor fields, their scales, partial sums.  Never through the
// read-only path (__ldg): that one is for memory that does not change while the reading kernel is
// resident, and the kernels of an iteration are resident before their predecessor has ended (see
// chain_wait).  A plain load is ordered behind the wait, for the compiler and in the caches.  Links,
// work tables and clover matrices, which no kernel of a solve writes, keep __ldg.
template <class C>
__device__ __forceinline__ C ld_field(const C *p) {
    return *p;
}
// The same where the loads are to be issued in the order they are written in.
__device__ __forceinline__ float4 ld_field_here(const float4 *p) {
    float4 v;
    asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(__cvta_generic_to_global(p)));
    return v;
}
__device__ __forceinline__ uint4 ld_field_here(const uint4 *p) {
    uint4 v;
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(__cvta_generic_to_global(p)));
    return v;
}

template <class P>
__device__ __forceinline__ void load_spinor(const FieldView &f, int64_t i, typename P::real v[24]);

template <>
__device__ __forceinline__ void load_spinor<PF64>(const FieldView &f, int64_t i, double v[24]) {
    const double2 *b = reinterpret_cast<const double2 *>(f.p);
#pragma unroll
    for (int j = 0; j < 12; j++) {
        double2 c = ld_field(b + j * f.stride + i);
        v[2 * j] = c.x;
        v[2 * j + 1] = c.y;
    }
}
template <>
__device__ __forceinline__ void load_spinor<PF32>(const FieldView &f, int64_t i, float v[24]) {
    const float4 *b = reinterpret_cast<const float4 *>(f.p);
#pragma unroll
    for (int j = 0; j < 6; j++) {
        float4 c = ld_field(b + j * f.stride + i);
        v[4 * j] = c.x;
        v[4 * j + 1] = c.y;
        v[4 * j + 2] = c.z;
        v[4 * j + 3] = c.w;
    }
}
template <>
__device__ __forceinline__ void load_spinor<PF16>(const FieldView &f, int64_t i, float v[24]) {
    const uint4 *b = reinterpret_cast<const uint4 *>(f.p);
    float s = ld_field(f.scale + i);
#pragma unroll
    for (int j = 0; j < 3; j++) {
        uint4 c = ld_field(b + j * f.stride + i);
        float2 a0 = h2f(c.x), a1 = h2f(c.y), a2 = h2f(c.z), a3 = h2f(c.w);
        v[8 * j + 0] = s * a0.x;
        v[8 * j + 1] = s * a0.y;
        v[8 * j + 2] = s * a1.x;
        v[8 * j + 3] = s * a1.y;
        v[8 * j + 4] = s * a2.x;
        v[8 * j + 5] = s * a2.y;
        v[8 * j + 6] = s * a3.x;
        v[8 * j + 7] = s * a3.y;
    }
}
template <>
__device__ __forceinline__ void load_spinor<PBF16>(const FieldView &f, int64_t i, float v[24]) {
    const uint4 *b = reinterpret_cast<const uint4 *>(f.p);
#pragma unroll
    for (int j = 0; j < 3; j++) {
        uint4 c = ld_field(b + j * f.stride + i);
        float2 a0 = b2f(c.x), a1 = b2f(c.y), a2 = b2f(c.z), a3 = b2f(c.w);
        v[8 * j + 0] = a0.x;
        v[8 * j + 1] = a0.y;
        v[8 * j + 2] = a1.x;
        v[8 * j + 3] = a1.y;
        v[8 * j + 4] = a2.x;
        v[8 * j + 5] = a2.y;
        v[8 * j + 6] = a3.x;
        v[8 * j + 7] = a3.y;
    }
}

// Spinor as stored, as (re, im) pairs: FP16 values without their site-column
// scale, which is returned in *s (1 for the other formats).
// off: the byte offsets of the storage chunks, kernel parameters, so that no strides are held in
// registers.
// IN_ORDER: see ld_field_here.
template <class P, bool IN_ORDER>
__device__ __forceinline__ void load_pairs(const FieldView &f, const int64_t *off, int64_t i, float2 v[12], float *s) {
    using C = typename P::chunk;
    const char *b = reinterpret_cast<const char *>(f.p) + i * (int64_t)sizeof(C);
    *s = P::SCALED ? ld_field(f.scale + i) : 1.f;
#pragma unroll
    for (int j = 0; j < P::NCH; j++) {
        const C *q = reinterpret_cast<const C *>(b + off[j]);
        const C c = IN_ORDER ? ld_field_here(q) : ld_field(q);
        if constexpr (P::NCH == 6) {
            v[2 * j] = make_float2(c.x, c.y);
            v[2 * j + 1] = make_float2(c.z, c.w);
        } else {
            v[4 * j] = P::SCALED ? h2f(c.x) : b2f(c.x);
            v[4 * j + 1] = P::SCALED ? h2f(c.y) : b2f(c.y);
            v[4 * j + 2] = P::SCALED ? h2f(c.z) : b2f(c.z);
            v[4 * j + 3] = P::SCALED ? h2f(c.w) : b2f(c.w);
        }
    }
}

template <class P>
__device__ __forceinline__ void store_spinor(const FieldView &f, int64_t i, const typename P::real v[24]);

template <>
__device__ __forceinline__ void store_spinor<PF64>(const FieldView &f, int64_t i, const double v[24]) {
    double2 *b = reinterpret_cast<double2 *>(f.p);
#pragma unroll
    for (int j = 0; j < 12; j++) b[j * f.stride + i] = make_double2(v[2 * j], v[2 * j + 1]);
}
template <>
__device__ __forceinline__ void store_spinor<PF32>(const FieldView &f, int64_t i, const float v[24]) {
    float4 *b = reinterpret_cast<float4 *>(f.p);
#pragma unroll
    for (int j = 0; j < 6; j++) b[j * f.stride + i] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
}
template <>
__device__ __forceinline__ void store_spinor<PF16>(const FieldView &f, int64_t i, const float v[24]) {
    float m = 0.f;
#pragma unroll
    for (int j = 0; j < 24; j++) m = fmaxf(m, fabsf(v[j]));
    float inv = (m > 0.f) ? 1.0f / m : 0.f;
    f.scale[i] = m;
    uint4 *b = reinterpret_cast<uint4 *>(f.p);
#pragma unroll
    for (int j = 0; j < 3; j++) {
        uint4 c;
        c.x = f2h(v[8 * j + 0] * inv, v[8 * j + 1] * inv);
        c.y = f2h(v[8 * j + 2] * inv, v[8 * j + 3] * inv);
        c.z = f2h(v[8 * j + 4] * inv, v[8 * j + 5] * inv);
        c.w = f2h(v[8 * j + 6] * inv, v[8 * j + 7] * inv);
        b[j * f.stride + i] = c;
    }
}
template <>
__device__ __forceinline__ void store_spinor<PBF16>(const FieldView &f, int64_t i, const float v[24]) {
    uint4 *b = reinterpret_cast<uint4 *>(f.p);
#pragma unroll
    for (int j = 0; j < 3; j++) {
        uint4 c;
        c.x = f2b(v[8 * j + 0], v[8 * j + 1]);
        c.y = f2b(v[8 * j + 2], v[8 * j + 3]);
        c.z = f2b(v[8 * j + 4], v[8 * j + 5]);
        c.w = f2b(v[8 * j + 6], v[8 * j + 7]);
        b[j * f.stride + i] = c;
    }
}

// -------------------------------------------------------------- links

template <typename T>
__device__ __forceinline__ void reconstruct_row2(cx<T> u[3][3]) {
    // row2 = conj(row0 x row1), exact for SU(3)
    u[2][0] = conj(u[0][1] * u[1][2] - u[0][2] * u[1][1]);
    u[2][1] = conj(u[0][2] * u[1][0] - u[0][0] * u[1][2]);
    u[2][2] = conj(u[0][0] * u[1][1] - u[0][1] * u[1][0]);
}

template <class P>
__device__ __forceinline__ void load_link(const void *L, int64_t V, int mu, int64_t g, cx<typename P::real> u[3][3]);

template <>
__device__ __forceinline__ void load_link<PF64>(const void *L, int64_t V, int mu, int64_t g, cx<double> u[3][3]) {
    const double2 *b = reinterpret_cast<const double2 *>(L) + (int64_t)mu * 9 * V + g;
#pragma unroll
    for (int j = 0; j < 9; j++) {
        double2 c = __ldg(b + j * V);
        u[j / 3][j % 3] = mk(c.x, c.y);
    }
}
template <>
__device__ __forceinline__ void load_link<PF32>(const void *L, int64_t V, int mu, int64_t g, cx<float> u[3][3]) {
    const float4 *b = reinterpret_cast<const float4 *>(L) + (int64_t)mu * 3 * V + g;
    float4 c0 = __ldg(b), c1 = __ldg(b + V), c2 = __ldg(b + 2 * V);
    u[0][0] = mk(c0.x, c0.y);
    u[0][1] = mk(c0.z, c0.w);
    u[0][2] = mk(c1.x, c1.y);
    u[1][0] = mk(c1.z, c1.w);
    u[1][1] = mk(c2.x, c2.y);
    u[1][2] = mk(c2.z, c2.w);
    reconstruct_row2(u);
}
template <>
__device__ __forceinline__ void load_link<PF16>(const void *L, int64_t V, int mu, int64_t g, cx<float> u[3][3]) {
    const uint2 *b = reinterpret_cast<const uint2 *>(L) + (int64_t)mu * 3 * V + g;
    uint2 c0 = __ldg(b), c1 = __ldg(b + V), c2 = __ldg(b + 2 * V);
    float2 a;
    a = h2f(c0.x); u[0][0] = mk(a.x, a.y);
    a = h2f(c0.y); u[0][1] = mk(a.x, a.y);
    a = h2f(c1.x); u[0][2] = mk(a.x, a.y);
    a = h2f(c1.y); u[1][0] = mk(a.x, a.y);
    a = h2f(c2.x); u[1][1] = mk(a.x, a.y);
    a = h2f(c2.y); u[1][2] = mk(a.x, a.y);
    reconstruct_row2(u);
}
template <>
__device__ __forceinline__ void load_link<PBF16>(const void *L, int64_t V, int mu, int64_t g, cx<float> u[3][3]) {
    const uint2 *b = reinterpret_cast<const uint2 *>(L) + (int64_t)mu * 3 * V + g;
    uint2 c0 = __ldg(b), c1 = __ldg(b + V), c2 = __ldg(b + 2 * V);
    float2 a;
    a = b2f(c0.x); u[0][0] = mk(a.x, a.y);
    a = b2f(c0.y); u[0][1] = mk(a.x, a.y);
    a = b2f(c1.x); u[0][2] = mk(a.x, a.y);
    a = b2f(c1.y); u[1][0] = mk(a.x, a.y);
    a = b2f(c2.x); u[1][1] = mk(a.x, a.y);
    a = b2f(c2.y); u[1][2] = mk(a.x, a.y);
    reconstruct_row2(u);
}

// ------------------------------------------------------ batch work table
//
// One Item per (domain, request) of a launch.  All spinor fields of a launch
// are concatenations of the items' column segments: column c of item it
// occupies site-columns [fbase + c*nh, fbase + (c+1)*nh) of each parity field.
// Hop-style kernels use blocks of TS sites x CG columns; item it owns blocks
// [blk0, blk0 + ntiles*ncg).  Reduction partials of (column c, tile t) live at
// pbase + c*ntiles + t.

// n / d for 0 <= n < 2^31 by a multiplication: q = n m >> s with m = floor(2^s / d) + 1,
// s = 31 + ceil(log2 d).
struct FastDiv {
    unsigned m;
    int s;
};
inline FastDiv fast_div(int d) {
    int l = 0;
    while ((1ll << l) < d) l++;
    FastDiv f;
    f.s = 31 + l;
    f.m = (unsigned)((1ull << f.s) / (unsigned)d + 1);
    return f;
}
__device__ __forceinline__ int fdiv(int n, const FastDiv &f) {
    return (int)(((unsigned long long)(unsigned)n * f.m) >> f.s);
}

struct __align__(16) Item {
    int o[4];        // origin (global coordinates, reduced mod L)
    int e[4];        // extent
    int L[4];        // lattice
    int rmask;       // bit mu set: direction mu restricted (Dirichlet faces)
    int bc;          // time boundary: 0 periodic, 1 antiperiodic, 2 open
    int par_o;       // (o0+o1+o2+o3) & 1
    int nh;          // sites per parity = n/2
    int ntiles;      // ceil(nh / TS)
    int ncol;
    int ncg;         // ceil(ncol / CG)
    int blk0;
    int solve0;      // first solve (column) index
    // small domains (small.cuh): first cluster in the launch of their cluster size; blocks of a
    // cluster along each direction, and the extents of a block's sub-box (the last one even)
    int sblk0, sc[4], sb[4];
    int64_t fbase;
    int64_t pbase;
    double kappa;
    const void *links;    // links of the launch's storage precision
    const void *links64;  // FP64 links
    int64_t gV;           // lattice volume (link field row length)
    FastDiv by_hx, by_e2, by_e1, by_nt;  // division by e[3] / 2, e[2], e[1] and ntiles
    // clover term (clover.cuh), NULL without it: T and T^-1 in the launch's arithmetic
    // (FP64 packed for the FP64 path, FP32 packed otherwise) and T in FP64
    const void *clov;
    const void *clovinv;
    const void *clov64;
};

constexpr int INLINE_ITEMS = 4;  // a series of nested domains fits

struct Launch {
    const Item *items;
    int nitems;
    int TS, CG;          // sites per tile (multiple of 32), columns per block
    Item inl[INLINE_ITEMS];  // the items themselves where they are so few 
};

// Locate the item owning block b (items sorted by blk0).
__device__ __forceinline__ int find_item(const Item *items, int nitems, int b) {
    int lo = 0, hi = nitems - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (items[mid].blk0 <= b)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// Domain-local coordinates of the even-odd index h of parity p (requires e3 even):
// the local lexicographic index l = ((k0 e1 + k1) e2 + k2) e3 + k3 satisfies h = l >> 1.
__device__ __forceinline__ void decode_site(const Item &it, int h, int p, int k[4]) {
    const int row = fdiv(h, it.by_hx);
    const int j = h - row * (it.e[3] >> 1);
    const int r1 = fdiv(row, it.by_e2);
    k[2] = row - r1 * it.e[2];
    k[0] = fdiv(r1, it.by_e1);
    k[1] = r1 - k[0] * it.e[1];
    k[3] = 2 * j + ((p + it.par_o + k[0] + k[1] + k[2]) & 1);
}

__device__ __forceinline__ int local_lex(const Item &it, const int k[4]) {
    return ((k[0] * it.e[1] + k[1]) * it.e[2] + k[2]) * it.e[3] + k[3];
}

__device__ __forceinline__ int64_t global_lex(const Item &it, const int x[4]) {
    return (((int64_t)x[0] * it.L[1] + x[1]) * it.L[2] + x[2]) * it.L[3] + x[3];
}

// Link-field row of global site x with parity p.
__device__ __forceinline__ int64_t link_row(const Item &it, const int x[4], int p) {
    return (p ? (it.gV >> 1) : 0) + (global_lex(it, x) >> 1);
}

// ------------------------------------------------------------ hopping
//
// acc(y) = sum_mu [ f+ (1 - g_mu) U_mu(y) psi(y+mu) + f- (1 + g_mu) U_mu(y-mu)^+ psi(y-mu) ]
// restricted to the item's box: f = 0 for hops leaving a restricted direction
// or crossing an open time boundary, -1 across an antiperiodic one.  The spin
// projectors (1 -/+ g_mu) have rank 2 in the chiral basis
// g_mu = [[0, A_mu], [A_mu^+, 0]]: (1 - g)psi = [h; -A^+ h] with h = psi_up - A psi_dn
// and (1 + g)psi = [h; A^+ h] with h = psi_up + A psi_dn, so only the two
// rows of h are multiplied by the link.

// w = u h, one multiply-add chain per real component.
template <typename R>
__device__ __forceinline__ void su3_mul_half(const cx<R> u[3][3], const cx<R> h[2][3], cx<R> w[2][3]) {
#pragma unroll
    for (int s = 0; s < 2; s++)
#pragma unroll
        for (int a = 0; a < 3; a++) {
            R re = u[a][0].re * h[s][0].re;
            R im = u[a][0].re * h[s][0].im;
            re = fma(-u[a][0].im, h[s][0].im, re);
            im = fma(u[a][0].im, h[s][0].re, im);
#pragma unroll
            for (int b = 1; b < 3; b++) {
                re = fma(u[a][b].re, h[s][b].re, re);
                im = fma(u[a][b].re, h[s][b].im, im);
                re = fma(-u[a][b].im, h[s][b].im, re);
                im = fma(u[a][b].im, h[s][b].re, im);
            }
            w[s][a] = mk(re, im);
        }
}

// Spin projection of direction MU, FWD = forward hop (1 - g_mu), else (1 + g_mu).
template <int MU, bool FWD, typename R>
__device__ __forceinline__ void project(const R v[24], cx<R> h[2][3]) {
#pragma unroll
    for (int a = 0; a < 3; a++) {
        cx<R> p0 = mk(v[2 * a], v[2 * a + 1]);
        cx<R> p1 = mk(v[6 + 2 * a], v[6 + 2 * a + 1]);
        cx<R> p2 = mk(v[12 + 2 * a], v[12 + 2 * a + 1]);
        cx<R> p3 = mk(v[18 + 2 * a], v[18 + 2 * a + 1]);
        if (MU == 0) {
            h[0][a] = FWD ? p0 - p2 : p0 + p2;
            h[1][a] = FWD ? p1 - p3 : p1 + p3;
        } else if (MU == 1) {
            h[0][a] = FWD ? p0 + mul_i(p3) : p0 - mul_i(p3);
            h[1][a] = FWD ? p1 + mul_i(p2) : p1 - mul_i(p2);
        } else if (MU == 2) {
            h[0][a] = FWD ? p0 + p3 : p0 - p3;
            h[1][a] = FWD ? p1 - p2 : p1 + p2;
        } else {
            h[0][a] = FWD ? p0 + mul_i(p2) : p0 - mul_i(p2);
            h[1][a] = FWD ? p1 - mul_i(p3) : p1 + mul_i(p3);
        }
    }
}

// acc += f * [w; lower(w)] for direction MU and hop sense FWD, each real
// component one multiply-add (f is 1 for unscaled storage, the site-column
// scale for FP16).
template <typename R>
__device__ __forceinline__ void cfma(cx<R> &acc, R f, cx<R> w) {
    acc.re = fma(f, w.re, acc.re);
    acc.im = fma(f, w.im, acc.im);
}
template <int MU, bool FWD, typename R>
__device__ __forceinline__ void accumulate(cx<R> acc[4][3], const cx<R> w[2][3], R f) {
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const cx<R> w0 = w[0][a], w1 = w[1][a];
        cfma(acc[0][a], f, w0);
        cfma(acc[1][a], f, w1);
        if (MU == 0) {
            cfma(acc[2][a], FWD ? -f : f, w0);
            cfma(acc[3][a], FWD ? -f : f, w1);
        } else if (MU == 1) {
            cfma(acc[2][a], f, FWD ? mul_mi(w1) : mul_i(w1));
            cfma(acc[3][a], f, FWD ? mul_mi(w0) : mul_i(w0));
        } else if (MU == 2) {
            cfma(acc[2][a], FWD ? -f : f, w1);
            cfma(acc[3][a], FWD ? f : -f, w0);
        } else {
            cfma(acc[2][a], f, FWD ? mul_mi(w0) : mul_i(w0));
            cfma(acc[3][a], f, FWD ? mul_i(w1) : mul_mi(w1));
        }
    }
}

// The neighbour of local coordinates k (replaced by the neighbour's) in hop d = 2 mu + (backward ?
// 1 : 0) from parity p: false when the hop is dropped; the row of the link it is transported with,
// U_mu(x) forward and U_mu(x - mu)^+ backward, and whether the hop changes sign (across an
// antiperiodic time boundary).
__device__ __forceinline__ bool hop_neighbour(const Item &it, int k[4], int p, int d, int64_t &row, bool &neg) {
    int x[4];
#pragma unroll
    for (int m = 0; m < 4; m++) {
        int t = it.o[m] + k[m];
        x[m] = (t >= it.L[m]) ? t - it.L[m] : t;
    }
    const int mu = d >> 1;
    const bool fwd = !(d & 1);
    bool ok = true;
    const bool restricted = (it.rmask >> mu) & 1;
    if (fwd) {
        k[mu] += 1;
        if (restricted)
            ok = k[mu] < it.e[mu];
        else if (k[mu] == it.e[mu])
            k[mu] = 0;
    } else {
        k[mu] -= 1;
        if (restricted)
            ok = k[mu] >= 0;
        else if (k[mu] < 0)
            k[mu] = it.e[mu] - 1;
    }
    neg = false;
    if (mu == 0 && x[0] == (fwd ? it.L[0] - 1 : 0)) {
        neg = it.bc == 1;
        if (it.bc == 2) ok = false;
    }
    if (!ok) return false;
    if (fwd) {
        row = link_row(it, x, p);
    } else {
        x[mu] = (x[mu] == 0) ? it.L[mu] - 1 : x[mu] - 1;
        row = link_row(it, x, p ^ 1);
    }
    return true;
}

// The same from even-odd site h: the neighbour's even-odd index, -1 when the hop is dropped.
__device__ __forceinline__ int hop_geometry(const Item &it, int h, int p, int d, int64_t &row, bool &neg) {
    int k[4];
    decode_site(it, h, p, k);
    return hop_neighbour(it, k, p, d, row, neg) ? local_lex(it, k) >> 1 : -1;
}

// The neighbour's index of a hop and its link in storage format P, oriented and
// multiplied by the boundary sign of the hop.
template <class P>
__device__ __forceinline__ int stage_hop(const Item &it, int h, int p, int d, cx<typename P::real> u[3][3]) {
    using R = typename P::real;
    int64_t row = 0;
    bool neg;
    const int nb = hop_geometry(it, h, p, d, row, neg);
    if (nb < 0) return -1;
    const R f = neg ? R(-1) : R(1);
    if (!(d & 1)) {
        load_link<P>(it.links, it.gV, d >> 1, row, u);
#pragma unroll
        for (int i = 0; i < 3; i++)
#pragma unroll
            for (int j = 0; j < 3; j++) u[i][j] = f * u[i][j];
    } else {
        cx<R> v[3][3];
        load_link<P>(it.links, it.gV, d >> 1, row, v);
#pragma unroll
        for (int i = 0; i < 3; i++)
#pragma unroll
            for (int j = 0; j < 3; j++) u[i][j] = f * conj(v[j][i]);
    }
    return nb;
}

// acc += f (1 -/+ g_mu) u psi for hop D (compile-time), link u already
// oriented, in plain arithmetic (the boundary source and the non-finite cases).
template <int D, typename R>
__device__ __forceinline__ void hop_step(const R v[24], const cx<R> u[3][3], cx<R> acc[4][3], R f) {
    constexpr int MU = D >> 1;
    constexpr bool FWD = !(D & 1);
    cx<R> h[2][3], w[2][3];
    project<MU, FWD>(v, h);
    su3_mul_half(u, h, w);
    accumulate<MU, FWD>(acc, w, f);
}

// ------------------------------------------------ packed FP32 hopping step
//
// The low-precision stencils compute on (re, im) pairs with GB300's two-lane FP32
// instructions (one issue slot for two multiply-adds).  u h = A + i B with the pairs
// A = sum re(u) * h and B = sum im(u) * h, so that only the link's parts are duplicated, never a
// spinor operand swapped: 72 FP instructions and 24 moves per hop, where the scalar form issues
// 132.  (Links staged as (re, re, im, im) need no moves but twice the shared-memory reads, which
// cost more: 0.36 against 0.28 ms for the plain FP32 stencil on 48x24^3, 12 columns.  Scalar
// arithmetic: 0.305 ms; with the division-free set-up and the items as parameters, 0.264.)

__device__ __forceinline__ float2 f2(float x, float y) { return make_float2(x, y); }
__device__ __forceinline__ float2 f2_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 f2_sub(float2 a, float2 b) { return __ffma2_rn(b, f2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 f2_add_i(float2 a, float2 b) { return f2(a.x - b.y, a.y + b.x); }  // a + i b
__device__ __forceinline__ float2 f2_sub_i(float2 a, float2 b) { return f2(a.x + b.y, a.y - b.x); }

template <int MU, bool FWD>
__device__ __forceinline__ void f2_project(const float2 v[12], float2 h[2][3]) {
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const float2 p0 = v[a], p1 = v[3 + a], p2 = v[6 + a], p3 = v[9 + a];
        if (MU == 0) {
            h[0][a] = FWD ? f2_sub(p0, p2) : f2_add(p0, p2);
            h[1][a] = FWD ? f2_sub(p1, p3) : f2_add(p1, p3);
        } else if (MU == 1) {
            h[0][a] = FWD ? f2_add_i(p0, p3) : f2_sub_i(p0, p3);
            h[1][a] = FWD ? f2_add_i(p1, p2) : f2_sub_i(p1, p2);
        } else if (MU == 2) {
            h[0][a] = FWD ? f2_add(p0, p3) : f2_sub(p0, p3);
            h[1][a] = FWD ? f2_sub(p1, p2) : f2_add(p1, p2);
        } else {
            h[0][a] = FWD ? f2_add_i(p0, p2) : f2_sub_i(p0, p2);
            h[1][a] = FWD ? f2_sub_i(p1, p3) : f2_add_i(p1, p3);
        }
    }
}

// acc += f w, acc -= f w, acc += i f w, acc -= i f w (SCALED: f != 1)
template <bool SCALED>
__device__ __forceinline__ void f2_acc(float2 &acc, float2 w, float f) {
    acc = SCALED ? __ffma2_rn(f2(f, f), w, acc) : __fadd2_rn(acc, w);
}
template <bool SCALED>
__device__ __forceinline__ void f2_acc_neg(float2 &acc, float2 w, float f) {
    acc = __ffma2_rn(SCALED ? f2(-f, -f) : f2(-1.f, -1.f), w, acc);
}
template <bool SCALED>
__device__ __forceinline__ void f2_acc_i(float2 &acc, float2 w, float f) {
    acc.x = SCALED ? fmaf(-f, w.y, acc.x) : acc.x - w.y;
    acc.y = SCALED ? fmaf(f, w.x, acc.y) : acc.y + w.x;
}
template <bool SCALED>
__device__ __forceinline__ void f2_acc_mi(float2 &acc, float2 w, float f) {
    acc.x = SCALED ? fmaf(f, w.y, acc.x) : acc.x + w.y;
    acc.y = SCALED ? fmaf(-f, w.x, acc.y) : acc.y - w.x;
}

// acc += f (1 -/+ g_mu) u psi for hop D; u: 9 staged entries.
template <int D, bool SCALED>
__device__ __forceinline__ void f2_hop_step(const float2 v[12], const float2 *u, float2 acc[4][3], float f) {
    constexpr int MU = D >> 1;
    constexpr bool FWD = !(D & 1);
    float2 h[2][3];
    f2_project<MU, FWD>(v, h);
#pragma unroll
    for (int a = 0; a < 3; a++) {
        float2 A[2], B[2];
#pragma unroll
        for (int b = 0; b < 3; b++) {
            const float2 c = u[3 * a + b];
#pragma unroll
            for (int s = 0; s < 2; s++) {
                A[s] = b ? __ffma2_rn(f2(c.x, c.x), h[s][b], A[s]) : __fmul2_rn(f2(c.x, c.x), h[s][b]);
                B[s] = b ? __ffma2_rn(f2(c.y, c.y), h[s][b], B[s]) : __fmul2_rn(f2(c.y, c.y), h[s][b]);
            }
        }
        const float2 w0 = f2_add_i(A[0], B[0]), w1 = f2_add_i(A[1], B[1]);
        f2_acc<SCALED>(acc[0][a], w0, f);
        f2_acc<SCALED>(acc[1][a], w1, f);
        if (MU == 0) {
            if (FWD) { f2_acc_neg<SCALED>(acc[2][a], w0, f); f2_acc_neg<SCALED>(acc[3][a], w1, f); }
            else { f2_acc<SCALED>(acc[2][a], w0, f); f2_acc<SCALED>(acc[3][a], w1, f); }
        } else if (MU == 1) {
            if (FWD) { f2_acc_mi<SCALED>(acc[2][a], w1, f); f2_acc_mi<SCALED>(acc[3][a], w0, f); }
            else { f2_acc_i<SCALED>(acc[2][a], w1, f); f2_acc_i<SCALED>(acc[3][a], w0, f); }
        } else if (MU == 2) {
            if (FWD) { f2_acc_neg<SCALED>(acc[2][a], w1, f); f2_acc<SCALED>(acc[3][a], w0, f); }
            else { f2_acc<SCALED>(acc[2][a], w1, f); f2_acc_neg<SCALED>(acc[3][a], w0, f); }
        } else {
            if (FWD) { f2_acc_mi<SCALED>(acc[2][a], w0, f); f2_acc_i<SCALED>(acc[3][a], w1, f); }
            else { f2_acc_i<SCALED>(acc[2][a], w0, f); f2_acc_mi<SCALED>(acc[3][a], w1, f); }
        }
    }
}

// --------------------------------------------------------- reductions

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

}  // namespace ddp
