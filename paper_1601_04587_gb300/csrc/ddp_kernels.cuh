// Kernels of the domain solver: the masked even-odd hopping term with fused
// epilogues and dot products, BiCGStab vector updates, per-solve scalar
// updates, FP64 defect-correction steps and layout conversions.
#pragma once

#include <type_traits>

#include "ddp_device.cuh"
#include "clover.cuh"
#include "fx64.cuh"
#include "recur.cuh"

namespace ddp {

// ------------------------------------------------------------ solver state

// Per solve (one column of one request).
struct SolveState {
    double2 rho, alpha, omega, beta, inv;   // the inner recurrence (recur.cuh)
    float2 alpha32, omega32, beta32;         // the same rounded, for the vector updates in FP32
    double target2;  // inner stopping threshold on |r|^2
    double bnorm2;   // |eta|^2 (FP64)
    double rr64;     // |eta - D_Gamma x|^2 of the current outer cycle (FP64)
    double sigma;    // about |r64| of the current cycle (0: nothing to do)
    double scale;    // 2 kappa / sigma, a power of two
    double delta;    // inner relative tolerance of the cycle
    double tol;      // requested relative tolerance
    double floor_delta;  // smallest useful inner tolerance of the storage format
    int active;      // inner iteration: 1 running, 2 its last update of x and r pending, 0 done
    int iters;       // inner iterations of the current cycle
    int total_iters; // inner iterations over all cycles
    int status;      // inner: 0 running, 1 converged, 2 breakdown, 3 iteration cap, 4 skipped
    int outer_done;  // 1 once |eta - D x| <= tol |eta|
    int item, col;
    int maxit;       // inner iteration cap per cycle
    // from the column's item, so that the scalar kernels reach the partials in one step
    int ntiles;
    int64_t pbase;   // first partial slot of the column
    double kappa;
};

__device__ __forceinline__ void set_scalar(double2 &v, float2 &v32, Cnum c) {
    v = c;
    v32 = make_float2((float)c.x, (float)c.y);
}
// A scalar of the recurrence in the compute precision.
__device__ __forceinline__ double2 scalar_value(const double2 &v, const float2 &, double) { return v; }
__device__ __forceinline__ float2 scalar_value(const double2 &, const float2 &v32, float) { return v32; }

struct LoopCtl {
    unsigned long long arrived;  // this iteration: columns decided (low half), columns going on (high half)
    int iter;
    int maxit;
    int pad;  // host-polled loop: 1 while the loop continues
};

// Reduction partials: NV sums per (item, column, tile) at d[slot * NV + k], NV = dot_sums(DOT), in
// the precision they were formed in (FP32 or FP64).
struct Partials {
    void *d;
};
constexpr int PART_MAX = 8;  // largest NV

// Epilogues of the hopping kernel (acc = the hopping sum, v1, v2 operands at the
// output site; T / T^-1 the clover matrices of the output site, identity without
// the clover term):
//   PLAIN  T^-1 acc                 MHAT  v1 - kappa^2 T^-1 acc
//   AXPY_K v1 + kappa T^-1 acc      RHS   T^-1 (v1 + kappa acc)
//   DIRAC  T v1 / (2 kappa) - acc/2 RESID v2 - T v1 / (2 kappa) + acc/2
enum Epi { EPI_PLAIN = 0, EPI_MHAT = 1, EPI_AXPY_K = 2, EPI_DIRAC = 3, EPI_RESID = 4, EPI_RHS = 5 };
// Dot products of the epilogue (o the output, v1 its operand):
//   RHAT (rh, o)     NORM (o, o)     TS (o, v1), (rh, v1), (rh, o), (o, o), (v1, v1)
enum Dot { DOT_NONE = 0, DOT_RHAT = 1, DOT_TS = 2, DOT_NORM = 3 };
__host__ __device__ constexpr int dot_sums(int dot) {
    return dot == DOT_RHAT ? 2 : dot == DOT_TS ? PART_MAX : dot == DOT_NORM ? 1 : 0;
}

struct HopArgs {
    Launch L;
    int p;          // parity of the output sites
    FieldView in;   // opposite-parity input
    FieldView out;  // output (parity p)
    FieldView v1;   // same-parity operand of the epilogue
    FieldView v2;   // second same-parity operand (EPI_RESID: eta)
    FieldView rh;   // shadow residual for DOT_RHAT and DOT_TS
    Partials part;
    const SolveState *st;  // skip 1: leave columns whose inner solve is not active untouched;
    int skip;              // skip 2: leave columns whose outer solve has converged untouched
    int64_t off[6];        // byte offsets of the storage chunks of in (set by launch_hop)
};

// Whether a kernel with the given skip mode leaves the column alone.
__device__ __forceinline__ bool skipped(const SolveState &S, int skip) {
    return (skip == 1) ? S.active != 1 : (skip == 2) && S.outer_done;
}

// The kernels of an iteration are launched as programmatic dependents of one another: a kernel may
// start while its predecessor runs, does what depends on the work table and the links alone, waits
// in chain_wait until the predecessor has completed with its writes visible, and lets its own
// successor start (chain_next, always after chain_wait: when a kernel starts, all but its direct
// predecessor are complete).  Every block of a chained kernel waits before it ends, so that a
// completed kernel implies that all before it are complete.  Without the launch attribute both do
// nothing.  What kernels write is read with plain loads throughout (ld_field).  What it hides is
// each kernel's start, its item and, in the stencils, the staging of the first wave's links behind
// the tail of the kernel before: 8 kernels an iteration, 12 columns FP32, 8^4 block 2.84 -> 2.47 ms,
// 4x32^3 slab 34.5 -> 33.6, 16x24^3 FP16 48.1 -> 46.2.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Tiles are exactly HOP_TS = 32 sites (one warp per column of a tile); a
// block holds at most HOP_MAX_CG = 12 columns.  The kernels use the tile size
// as a compile-time constant.
// Storage of the BiCGStab shadow residual rh: any fixed vector serves as rh, so with
// FP32 storage it is kept as a BF16 copy of r_0 (same exponent range, half the bytes
// of the two reads per iteration); the other formats keep their own.
template <class P>
struct ShadowOf {
    using type = P;
};
template <>
struct ShadowOf<PF32> {
    using type = PBF16;
};

constexpr int HOP_TS = 32;
constexpr int HOP_MAX_CG = 12;

// Map a block/thread of a tile-structured launch to (item, column, site).
struct TileCoord {
    int col, h, tile;
    bool valid;
    int64_t cb;  // column base in the fields
};

__device__ __forceinline__ TileCoord tile_coord(const Item &it, const Launch &L, int blk) {
    TileCoord t;
    int lb = blk - it.blk0;
    const int cg = fdiv(lb, it.by_nt);
    t.tile = lb - cg * it.ntiles;
    int cl = threadIdx.x / HOP_TS;
    int sl = threadIdx.x - cl * HOP_TS;
    t.col = cg * L.CG + cl;
    t.h = t.tile * HOP_TS + sl;
    t.valid = (t.col < it.ncol) && (t.h < it.nh) && (cl < L.CG);
    t.cb = it.fbase + (int64_t)t.col * it.nh;
    return t;
}
__device__ __forceinline__ TileCoord tile_coord(const Item &it, const Launch &L) {
    return tile_coord(it, L, (int)blockIdx.x);
}

// Sums of NV values over the 32 sites of a tile, which are one warp of one column.  Each
// thread's products and the warp's sums are formed in the compute precision R (FP32 for the
// low-precision formats: FP64 arithmetic is a small fraction of GB300's FP32 rate); the sums over
// tiles, in the scalar kernels, have at least the precision of FP64 (recur.cuh).  Fixed order:
// results do not depend on the batch around them.  The lanes split the values as the distance halves
// (9 shuffles for 8 values, not 40): value k ends in lanes k * 32 / NV and following.
template <int NV, typename R>
__device__ __forceinline__ void warp_partials(const Item &it, const TileCoord &tc, R v[NV], Partials part) {
    const int lane = threadIdx.x & 31;
    int off = 16;
#pragma unroll
    for (int n = NV; n > 1; n >>= 1, off >>= 1) {
        const bool up = lane & off;
#pragma unroll
        for (int i = 0; i < n / 2; i++) {
            const R keep = up ? v[i + n / 2] : v[i], send = up ? v[i] : v[i + n / 2];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
#pragma unroll
    for (; off > 0; off >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
    if (tc.col < it.ncol && (lane & (32 / NV - 1)) == 0)
        reinterpret_cast<R *>(part.d)[(it.pbase + (int64_t)tc.col * it.ntiles + tc.tile) * NV + lane / (32 / NV)] = v[0];
}

// The block's item, copied by words by one warp: from the kernel parameters where the launch
// carries its items there (Launch::inl), so that a block does not begin with a wait for memory.
// Every block starts with this, so it counts: plain FP32 stencil on 48x24^3, 12 columns, 0.287 ms
// with a copy by one thread, 0.267 from global memory, 0.264 from the
// parameters.
__device__ __forceinline__ void load_item(const Launch &L, Item &dst, int blk) {
    static_assert(sizeof(Item) % 16 == 0, "copied by 16 bytes");
    constexpr int N = sizeof(Item) / 16;
    if (threadIdx.x < 32) {
        if (L.nitems <= INLINE_ITEMS) {
            int i = 0;
#pragma unroll
            for (int k = 1; k < INLINE_ITEMS; k++) i += (k < L.nitems && L.inl[k].blk0 <= blk) ? 1 : 0;
            if (threadIdx.x < N)
                reinterpret_cast<int4 *>(&dst)[threadIdx.x] = reinterpret_cast<const int4 *>(L.inl + i)[threadIdx.x];
        } else {
            const int4 *src = reinterpret_cast<const int4 *>(L.items + find_item(L.items, L.nitems, blk));
            if (threadIdx.x < N) reinterpret_cast<int4 *>(&dst)[threadIdx.x] = __ldg(src + threadIdx.x);
        }
    }
    __syncthreads();
}
__device__ __forceinline__ void load_item(const Launch &L, Item &dst) { load_item(L, dst, (int)blockIdx.x); }

// ------------------------------------------------------------ hopping kernel

// The (re, im) pairs of a storage chunk, and a chunk of an unscaled format from them.
template <class P>
__device__ __forceinline__ void chunk_pairs(const typename P::chunk &c, float2 *v) {
    if constexpr (std::is_same<P, PF32>::value) {
        v[0] = f2(c.x, c.y);
        v[1] = f2(c.z, c.w);
    } else {
        v[0] = P::SCALED ? h2f(c.x) : b2f(c.x);
        v[1] = P::SCALED ? h2f(c.y) : b2f(c.y);
        v[2] = P::SCALED ? h2f(c.z) : b2f(c.z);
        v[3] = P::SCALED ? h2f(c.w) : b2f(c.w);
    }
}
template <class P>
__device__ __forceinline__ typename P::chunk pairs_chunk(const float2 *v) {
    if constexpr (std::is_same<P, PF32>::value)
        return make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
    else
        return make_uint4(f2b(v[0].x, v[0].y), f2b(v[1].x, v[1].y), f2b(v[2].x, v[2].y), f2b(v[3].x, v[3].y));
}

// ------------------------------------------------------------ hopping kernel

// Tiles of TS sites: the links (oriented, boundary sign folded in, row 2
// rebuilt) and neighbour indices of the tile's 8 TS hops are staged in shared
// memory once and shared by the CG column-threads of every site.
// Epilogue of the hopping kernels: out = combination of acc and same-parity
// operands, stored in the storage format, plus the requested dot products.
template <class P, int EPI, int DOT, bool CLOV>
__device__ __forceinline__ void hop_store_epilogue(const HopArgs &a, const Item &it, const TileCoord &tc,
                                                   const cx<typename P::real> acc[4][3],
                                                   typename P::real sums[PART_MAX]) {
    using R = typename P::real;
    R o[24];
    int64_t i = tc.cb + tc.h;
    const R kap = (R)it.kappa;
    // clover matrices of the output site (T^-1 on the hopping sum, T on v1)
    const bool clov = CLOV && it.clovinv;
    int64_t row = 0;
    if (clov) row = site_row(it, tc.h, a.p);
    R h[24];
#pragma unroll
    for (int s = 0; s < 4; s++)
#pragma unroll
        for (int c = 0; c < 3; c++) {
            h[2 * (3 * s + c)] = acc[s][c].re;
            h[2 * (3 * s + c) + 1] = acc[s][c].im;
        }
    if (clov && (EPI == EPI_PLAIN || EPI == EPI_MHAT || EPI == EPI_AXPY_K)) clover_apply<R>(it.clovinv, it.gV, row, h);
    if (EPI == EPI_PLAIN) {
#pragma unroll
        for (int j = 0; j < 24; j++) o[j] = h[j];
    } else {
        R w[24];
        load_spinor<P>(a.v1, i, w);
        if (clov && (EPI == EPI_DIRAC || EPI == EPI_RESID))
            clover_apply<R>(EPI == EPI_RESID ? it.clov64 : it.clov, it.gV, row, w);
        R cw, ca;
        if (EPI == EPI_MHAT) {
            cw = R(1);
            ca = -kap * kap;
        } else if (EPI == EPI_AXPY_K || EPI == EPI_RHS) {
            cw = R(1);
            ca = kap;
        } else if (EPI == EPI_DIRAC) {
            cw = R(1) / (R(2) * kap);
            ca = R(-0.5);
        } else {  // EPI_RESID: eta - T x/(2 kappa) + acc/2
            cw = -R(1) / (R(2) * kap);
            ca = R(0.5);
        }
        if (EPI == EPI_RESID) {
            // two multiply-adds a component (the FP64 pipe is this kernel's scarce unit)
            R e[24];
            load_spinor<P>(a.v2, i, e);
#pragma unroll
            for (int j = 0; j < 24; j++) o[j] = fma(ca, h[j], fma(cw, w[j], e[j]));
        } else {
#pragma unroll
            for (int j = 0; j < 24; j++) o[j] = cw * w[j] + ca * h[j];
        }
        if (clov && EPI == EPI_RHS) clover_apply<R>(it.clovinv, it.gV, row, o);
    }
    if (DOT == DOT_RHAT) {
        R r[24];
        load_spinor<typename ShadowOf<P>::type>(a.rh, i, r);
#pragma unroll
        for (int j = 0; j < 12; j++) {
            sums[0] += r[2 * j] * o[2 * j] + r[2 * j + 1] * o[2 * j + 1];
            sums[1] += r[2 * j] * o[2 * j + 1] - r[2 * j + 1] * o[2 * j];
        }
    }
    if (DOT == DOT_TS) {
        // t = out, s = v1 (loaded again: its registers were reused)
        R q[24];
        load_spinor<P>(a.v1, i, q);
#pragma unroll
        for (int j = 0; j < 12; j++) {
            sums[0] += o[2 * j] * q[2 * j] + o[2 * j + 1] * q[2 * j + 1];  // (t, s)
            sums[1] += o[2 * j] * q[2 * j + 1] - o[2 * j + 1] * q[2 * j];
            sums[7] += q[2 * j] * q[2 * j] + q[2 * j + 1] * q[2 * j + 1];  // (s, s)
        }
        R r[24];
        load_spinor<typename ShadowOf<P>::type>(a.rh, i, r);
#pragma unroll
        for (int j = 0; j < 12; j++) {
            sums[2] += r[2 * j] * q[2 * j] + r[2 * j + 1] * q[2 * j + 1];  // (rh, s)
            sums[3] += r[2 * j] * q[2 * j + 1] - r[2 * j + 1] * q[2 * j];
            sums[4] += r[2 * j] * o[2 * j] + r[2 * j + 1] * o[2 * j + 1];  // (rh, t)
            sums[5] += r[2 * j] * o[2 * j + 1] - r[2 * j + 1] * o[2 * j];
        }
    }
    if (DOT == DOT_TS || DOT == DOT_NORM) {
        R n = 0;
#pragma unroll
        for (int j = 0; j < 24; j++) n += o[j] * o[j];
        sums[DOT == DOT_TS ? 6 : 0] = n;
    }
    store_spinor<P>(a.out, i, o);  // last: no load moves above a store
}

// The FP32 stencil of the five products has no registers to spare: its loads stay where they are
// written, a few at a time.
template <class P, int DOT>
constexpr bool HOP_IN_ORDER = std::is_same<P, PF32>::value && DOT == DOT_TS;

// The same for the low-precision formats without a clover term, one storage chunk at a time (few
// registers live beside the sums) and in two-lane arithmetic.
template <class P, int EPI, int DOT>
__device__ __forceinline__ void hop_store_pairs(const HopArgs &a, float kap, int64_t i, float2 acc[12],
                                                float sums[PART_MAX]) {
    using SH = typename ShadowOf<P>::type;
    using C = typename P::chunk;
    constexpr int NC = 12 / P::NCH;  // complex components per chunk
    constexpr bool WITH_V1 = EPI != EPI_PLAIN, WITH_RH = DOT == DOT_RHAT || DOT == DOT_TS;
    const float cw = EPI == EPI_DIRAC ? 1.f / (2.f * kap) : 1.f;
    const float ca = EPI == EPI_DIRAC ? -0.5f : EPI == EPI_MHAT ? -kap * kap : kap;
    const float sw = (WITH_V1 && P::SCALED) ? ld_field(a.v1.scale + i) : 1.f;
    const float sr = (WITH_RH && SH::SCALED) ? ld_field(a.rh.scale + i) : 1.f;
    float2 oo = f2(0.f, 0.f), ww = oo, ow = oo, rw = oo, ro = oo;  // (x.re y.re, x.im y.im) sums
    float owi = 0.f, rwi = 0.f, roi = 0.f;                          // imaginary parts
    // The chunks of v1 and rh are requested AHEAD of their use: they are data that kernels write, so
    // no load of them moves above the stores in between.  All at once, but for the five products in
    // FP32, one chunk.  32x24^3, 12 columns, FP32, with the loads at their use / so: (rh, v) 0.242 /
    // 0.208 ms, (t, s) 0.258 / 0.217 (0.226 without HOP_IN_ORDER).
    constexpr bool HALF = std::is_same<P, PF32>::value;  // FP32 chunk j of rh: half j % 2 of BF16 chunk j / 2
    constexpr bool TIGHT = HOP_IN_ORDER<P, DOT>;
    constexpr int AHEAD = TIGHT ? 1 : P::NCH - 1;
    using CR = typename SH::chunk;
    C nw[P::NCH];
    CR nr[P::NCH];
    auto request = [&](int j) {
        const C *w = reinterpret_cast<const C *>(a.v1.p) + j * a.v1.stride + i;
        const CR *r = reinterpret_cast<const CR *>(a.rh.p) + (HALF ? j / 2 : j) * a.rh.stride + i;
        if (WITH_V1) nw[j] = TIGHT ? ld_field_here(w) : ld_field(w);
        if (WITH_RH && !(HALF && j % 2)) nr[j] = TIGHT ? ld_field_here(r) : ld_field(r);
    };
#pragma unroll
    for (int j = 0; j < AHEAD; j++) request(j);
#pragma unroll
    for (int j = 0; j < P::NCH; j++) {
        float2 w[NC], r[NC];
        if (j + AHEAD < P::NCH) request(j + AHEAD);
        if (WITH_V1) {
            chunk_pairs<P>(nw[j], w);
#pragma unroll
            for (int c = 0; c < NC; c++) {
                if (P::SCALED) w[c] = __fmul2_rn(f2(sw, sw), w[c]);
                acc[j * NC + c] = __ffma2_rn(f2(ca, ca), acc[j * NC + c], EPI == EPI_DIRAC ? __fmul2_rn(f2(cw, cw), w[c]) : w[c]);
            }
        }
        if (!P::SCALED) reinterpret_cast<C *>(a.out.p)[j * a.out.stride + i] = pairs_chunk<P>(acc + j * NC);
        if (WITH_RH) {
            if constexpr (HALF) {
                const CR &q = nr[j - j % 2];
                r[0] = b2f(j % 2 ? q.z : q.x);
                r[1] = b2f(j % 2 ? q.w : q.y);
            } else {
                chunk_pairs<SH>(nr[j], r);
                if (SH::SCALED)
#pragma unroll
                    for (int c = 0; c < NC; c++) r[c] = __fmul2_rn(f2(sr, sr), r[c]);
            }
        }
#pragma unroll
        for (int c = 0; c < NC; c++) {
            const float2 o = acc[j * NC + c];
            if (DOT == DOT_TS || DOT == DOT_NORM) oo = __ffma2_rn(o, o, oo);
            if (DOT == DOT_TS) {
                ww = __ffma2_rn(w[c], w[c], ww);
                ow = __ffma2_rn(o, w[c], ow);
                owi = fmaf(o.x, w[c].y, fmaf(-o.y, w[c].x, owi));
                rw = __ffma2_rn(r[c], w[c], rw);
                rwi = fmaf(r[c].x, w[c].y, fmaf(-r[c].y, w[c].x, rwi));
            }
            if (WITH_RH) {
                ro = __ffma2_rn(r[c], o, ro);
                roi = fmaf(r[c].x, o.y, fmaf(-r[c].y, o.x, roi));
            }
        }
    }
    if (P::SCALED) {
        float o[24];
#pragma unroll
        for (int c = 0; c < 12; c++) {
            o[2 * c] = acc[c].x;
            o[2 * c + 1] = acc[c].y;
        }
        store_spinor<P>(a.out, i, o);
    }
    if (DOT == DOT_NORM) sums[0] = oo.x + oo.y;
    if (DOT == DOT_RHAT) {
        sums[0] = ro.x + ro.y;
        sums[1] = roi;
    }
    if (DOT == DOT_TS) {
        sums[0] = ow.x + ow.y;  // (t, s) with t = out, s = v1
        sums[1] = owi;
        sums[2] = rw.x + rw.y;  // (rh, s)
        sums[3] = rwi;
        sums[4] = ro.x + ro.y;  // (rh, t)
        sums[5] = roi;
        sums[6] = oo.x + oo.y;  // (t, t)
        sums[7] = ww.x + ww.y;  // (s, s)
    }
}

// A staged link in shared memory: 9 entries.
__device__ __forceinline__ void put_link(float2 *q, const cx<float> u[3][3]) {
#pragma unroll
    for (int k = 0; k < 9; k++) q[k] = f2(u[k / 3][k % 3].re, u[k / 3][k % 3].im);
}

// Resident blocks per SM the register budget of the 32- and 16-bit stencils is fitted to
// (3: 56 registers a thread; 2: 80).
#ifndef DDP_HOP_MINB
#define DDP_HOP_MINB 3
#endif

constexpr unsigned HOP_EARLY = 3 * 152;  // three blocks on each SM
template <class P, int EPI, int DOT, bool CLOV = false>
__global__ void __launch_bounds__(384, DDP_HOP_MINB) k_hop(const __grid_constant__ HopArgs a) {
    constexpr int TS = HOP_TS;
    // oriented link of hop slot q at s_u[q * 9]; consecutive slots fall in distinct banks
    __shared__ __align__(16) Item it;
    __shared__ int s_nb[8 * TS];
    __shared__ float2 s_u[8 * TS * 9];
    load_item(a.L, it);
    const TileCoord tc0 = tile_coord(it, a.L);
    // the blocks of the first wave may start before the preceding kernel ends: they stage their
    // links first and wait then
    const bool early = blockIdx.x < HOP_EARLY;
    if (!early) chain_wait();
    if (a.skip) {
        // a block whose columns are all finished has nothing to stage or compute (the flags are set
        // by k_fin, which is complete: it never directly precedes a stencil; and within a loop a
        // flag only goes from 1 to 2 to 0, so a column that is seen finished stays so)
        const int col = tc0.col - (int)threadIdx.x / TS + (int)threadIdx.x;
        int live = 0;
        if ((int)threadIdx.x < a.L.CG && col < it.ncol) live = !skipped(a.st[it.solve0 + col], a.skip);
        if (!__syncthreads_or(live)) {
            chain_wait();
            return;
        }
    }
    if (std::is_same<P, PF32>::value && tc0.valid && !early) {
        // FP32 storage: the forward time-direction neighbour of this thread's site-column is
        // requested into L1 before the links are staged, so that its latency overlaps the
        // staging (with the backward one too, or with 16-bit storage, it gains less or nothing)
        const int v3h = it.nh / it.e[0];  // sites of one parity in a time slice
        int nbf = tc0.h + v3h;
        if (nbf >= it.nh) nbf -= it.nh;
        const float4 *base = reinterpret_cast<const float4 *>(a.in.p) + tc0.cb + nbf;
#pragma unroll
        for (int j = 0; j < P::NCH; j++) asm volatile("prefetch.global.L1 [%0];" ::"l"(base + j * a.in.stride));
    }
    for (int q = threadIdx.x; q < 8 * TS; q += blockDim.x) {
        const int d = q / TS, h = tc0.tile * TS + (q - d * TS);
        int nb = -1;
        cx<float> u[3][3];
        if (h < it.nh) nb = stage_hop<P>(it, h, a.p, d, u);
        s_nb[q] = nb;
        if (nb >= 0) put_link(s_u + q * 9, u);
    }
    chain_wait();
    chain_next();
    __syncthreads();
    const TileCoord tc = tile_coord(it, a.L);  // formed again: nothing of it was held in registers meanwhile
    const bool valid = tc.valid && !(a.skip && skipped(a.st[it.solve0 + tc.col], a.skip));
    float sums[PART_MAX] = {};
    if (valid) {
        float2 acc[4][3];
#pragma unroll
        for (int s2 = 0; s2 < 4; s2++)
#pragma unroll
            for (int c = 0; c < 3; c++) acc[s2][c] = f2(0.f, 0.f);
        const int sl = tc.h - tc.tile * TS;
#define DDP_HOP_STEP(D)                                                   \
        {                                                                 \
            const int nb = s_nb[(D) * TS + sl];                           \
            if (nb >= 0) {                                                \
                float2 v[12];                                             \
                float f;                                                  \
                load_pairs<P, HOP_IN_ORDER<P, DOT>>(a.in, a.off, tc.cb + nb, v, &f); \
                f2_hop_step<D, P::SCALED>(v, s_u + ((D) * TS + sl) * 9, acc, f); \
            }                                                             \
        }
        DDP_HOP_STEP(0)
        DDP_HOP_STEP(1)
        DDP_HOP_STEP(2)
        DDP_HOP_STEP(3)
        DDP_HOP_STEP(4)
        DDP_HOP_STEP(5)
        DDP_HOP_STEP(6)
        DDP_HOP_STEP(7)
#undef DDP_HOP_STEP
        if constexpr (CLOV) {
            cx<float> c4[4][3];
#pragma unroll
            for (int j = 0; j < 12; j++) c4[j / 3][j % 3] = mk(acc[j / 3][j % 3].x, acc[j / 3][j % 3].y);
            hop_store_epilogue<P, EPI, DOT, true>(a, it, tc, c4, sums);
        } else {
            hop_store_pairs<P, EPI, DOT>(a, (float)it.kappa, tc.cb + tc.h, &acc[0][0], sums);
        }
    }
    if (DOT != DOT_NONE) warp_partials<DOT != DOT_NONE ? dot_sums(DOT) : 1>(it, tc, sums, a.part);
}

// ------------------------------------------------------------ vector updates

// The reals of one storage chunk of an unscaled format, and back.
template <class P>
__device__ __forceinline__ void chunk_to_reals(const typename P::chunk &c, typename P::real *v);
template <>
__device__ __forceinline__ void chunk_to_reals<PF64>(const double2 &c, double *v) {
    v[0] = c.x;
    v[1] = c.y;
}
template <>
__device__ __forceinline__ void chunk_to_reals<PF32>(const float4 &c, float *v) {
    v[0] = c.x;
    v[1] = c.y;
    v[2] = c.z;
    v[3] = c.w;
}
template <>
__device__ __forceinline__ void chunk_to_reals<PBF16>(const uint4 &c, float *v) {
    const float2 a0 = b2f(c.x), a1 = b2f(c.y), a2 = b2f(c.z), a3 = b2f(c.w);
    v[0] = a0.x;
    v[1] = a0.y;
    v[2] = a1.x;
    v[3] = a1.y;
    v[4] = a2.x;
    v[5] = a2.y;
    v[6] = a3.x;
    v[7] = a3.y;
}
template <>
__device__ __forceinline__ void chunk_to_reals<PF16>(const uint4 &, float *) {}  // scaled: not chunk-local
template <class P>
__device__ __forceinline__ typename P::chunk reals_to_chunk(const typename P::real *v);
template <>
__device__ __forceinline__ double2 reals_to_chunk<PF64>(const double *v) {
    return make_double2(v[0], v[1]);
}
template <>
__device__ __forceinline__ float4 reals_to_chunk<PF32>(const float *v) {
    return make_float4(v[0], v[1], v[2], v[3]);
}
template <>
__device__ __forceinline__ uint4 reals_to_chunk<PBF16>(const float *v) {
    uint4 c;
    c.x = f2b(v[0], v[1]);
    c.y = f2b(v[2], v[3]);
    c.z = f2b(v[4], v[5]);
    c.w = f2b(v[6], v[7]);
    return c;
}
template <>
__device__ __forceinline__ uint4 reals_to_chunk<PF16>(const float *) {
    return make_uint4(0, 0, 0, 0);
}

enum BlasOp { OP_S_UPDATE = 1, OP_XRP_UPDATE = 2, OP_INIT = 3, OP_NORM = 4 };

struct BlasArgs {
    Launch L;
    FieldView x, r, rh, p, v, s, t;
    const SolveState *st;
    Partials part;
    int skip;
};

// One complex component: x += alpha p + omega s ; s <- r = s - omega t ; p <- r + beta (p - omega v).
template <typename R>
__device__ __forceinline__ void xrp_update(R x[2], R p[2], R s[2], const R t[2], const R v[2], R ar, R ai, R wr, R wi,
                                           R br, R bi) {
    x[0] += (ar * p[0] - ai * p[1]) + (wr * s[0] - wi * s[1]);
    x[1] += (ar * p[1] + ai * p[0]) + (wr * s[1] + wi * s[0]);
    s[0] -= wr * t[0] - wi * t[1];
    s[1] -= wr * t[1] + wi * t[0];
    const R qr = p[0] - (wr * v[0] - wi * v[1]), qi = p[1] - (wr * v[1] + wi * v[0]);
    p[0] = s[0] + (br * qr - bi * qi);
    p[1] = s[1] + (br * qi + bi * qr);
}

template <class P, int OP>
__global__ void __launch_bounds__(384) k_blas(const __grid_constant__ BlasArgs a) {
    using R = typename P::real;
    __shared__ __align__(16) Item it;
    load_item(a.L, it);
    TileCoord tc = tile_coord(it, a.L);
    chain_wait();
    chain_next();
    if (a.skip && tc.valid && !a.st[it.solve0 + tc.col].active) tc.valid = false;
    R nn[1] = {0};
    if (tc.valid) {
        int64_t i = tc.cb + tc.h;
        const SolveState &S = a.st[it.solve0 + tc.col];
        if (OP == OP_S_UPDATE) {  // s = r - alpha v
            R r[24], v[24];
            load_spinor<P>(a.r, i, r);
            load_spinor<P>(a.v, i, v);
            const auto al = scalar_value(S.alpha, S.alpha32, R(0));
            const R ar = al.x, ai = al.y;
#pragma unroll
            for (int j = 0; j < 12; j++) {
                r[2 * j] -= ar * v[2 * j] - ai * v[2 * j + 1];
                r[2 * j + 1] -= ar * v[2 * j + 1] + ai * v[2 * j];
            }
            store_spinor<P>(a.s, i, r);
        } else if (OP == OP_XRP_UPDATE && !P::SCALED) {
            // x += alpha p + omega s ; r = s - omega t ; p = r + beta (p - omega v), one pass (beta
            // is known beforehand, see FIN_OMEGA): 5 spinors read and 3 written, where the update
            // of x and r with its dot products and that of p took 6.5 and 4.  One storage chunk at
            // a time, the next one requested before this one is stored (x, p and r are written, so
            // no load moves above a store by itself): few registers and many loads in flight.
            using C = typename P::chunk;
            constexpr int NR = 24 / P::NCH;
            C *const fx = reinterpret_cast<C *>(a.x.p), *const fp = reinterpret_cast<C *>(a.p.p);
            C *const fr = reinterpret_cast<C *>(a.r.p);
            const C *const fs = reinterpret_cast<const C *>(a.s.p), *const ft = reinterpret_cast<const C *>(a.t.p);
            const C *const fv = reinterpret_cast<const C *>(a.v.p);
            const auto al = scalar_value(S.alpha, S.alpha32, R(0)), om = scalar_value(S.omega, S.omega32, R(0)),
                       be = scalar_value(S.beta, S.beta32, R(0));
            const R ar = al.x, ai = al.y, wr = om.x, wi = om.y, br = be.x, bi = be.y;
            C n[5];
            auto request = [&](int64_t o) {
                n[0] = ld_field(fx + o);
                n[1] = ld_field(fp + o);
                n[2] = ld_field(fs + o);
                n[3] = ld_field(ft + o);
                n[4] = ld_field(fv + o);
            };
            request(i);
#pragma unroll
            for (int j = 0; j < P::NCH; j++) {
                const int64_t o = j * a.x.stride + i;
                R x[NR], p[NR], s[NR], t[NR], v[NR];
                chunk_to_reals<P>(n[0], x);
                chunk_to_reals<P>(n[1], p);
                chunk_to_reals<P>(n[2], s);
                chunk_to_reals<P>(n[3], t);
                chunk_to_reals<P>(n[4], v);
                if (j + 1 < P::NCH) request(o + a.x.stride);
#pragma unroll
                for (int k = 0; k < NR / 2; k++)
                    xrp_update(x + 2 * k, p + 2 * k, s + 2 * k, t + 2 * k, v + 2 * k, ar, ai, wr, wi, br, bi);
                fx[o] = reals_to_chunk<P>(x);
                fr[o] = reals_to_chunk<P>(s);
                fp[o] = reals_to_chunk<P>(p);
            }
        } else if (OP == OP_XRP_UPDATE) {  // the same with a whole site-column at a time (its scale)
            R x[24], p[24], s[24], t[24], v[24];
            load_spinor<P>(a.x, i, x);
            load_spinor<P>(a.p, i, p);
            load_spinor<P>(a.s, i, s);
            load_spinor<P>(a.t, i, t);
            load_spinor<P>(a.v, i, v);
            const auto al = scalar_value(S.alpha, S.alpha32, R(0)), om = scalar_value(S.omega, S.omega32, R(0)),
                       be = scalar_value(S.beta, S.beta32, R(0));
            const R ar = al.x, ai = al.y, wr = om.x, wi = om.y, br = be.x, bi = be.y;
#pragma unroll
            for (int k = 0; k < 12; k++)
                xrp_update(x + 2 * k, p + 2 * k, s + 2 * k, t + 2 * k, v + 2 * k, ar, ai, wr, wi, br, bi);
            store_spinor<P>(a.x, i, x);
            store_spinor<P>(a.r, i, s);
            store_spinor<P>(a.p, i, p);
        } else if (OP == OP_INIT) {  // rh = r ; p = r ; x = 0
            R r[24], z[24];
            load_spinor<P>(a.r, i, r);
            store_spinor<typename ShadowOf<P>::type>(a.rh, i, r);
            store_spinor<P>(a.p, i, r);
#pragma unroll
            for (int j = 0; j < 24; j++) z[j] = R(0);
            store_spinor<P>(a.x, i, z);
        } else if (OP == OP_NORM) {  // |x|^2
            R x[24];
            load_spinor<P>(a.x, i, x);
            R n2 = 0;
#pragma unroll
            for (int j = 0; j < 24; j++) n2 += x[j] * x[j];
            nn[0] = n2;
        }
    }
    if (OP == OP_NORM) warp_partials<1>(it, tc, nn, a.part);
}

// ---------------------------------------------------- FP64 <-> storage format

struct ConvArgs {
    Launch L;
    FieldView lo;   // storage-format field
    FieldView hi;   // FP64 field
    const SolveState *st;
    int p;          // parity of the sites
    int clov;       // k_to_low: apply the clover T^-1 of the site (items that have one)
};

// The conversions between FP64 fields and FP32 run on the integer pipe (GB300 converts and
// multiplies two FP64 values per clock and SM: with 24 of each per site-column k_to_low took 119 us
// for 1.33 M site-columns in FP16, 82 this way; k_accum, 124 us, is bound by its bytes).

// v 2^m rounded to FP32; scale = 2^m.
__device__ __forceinline__ float float_of(double v, int m, double scale) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v), r = b + 0x10000000ull;
    const int e = (int)((r >> 52) & 0x7FF) + m - 896;
    const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
    if (e >= 1 && e <= 254) return __uint_as_float(sign | ((unsigned)e << 23) | ((unsigned)(r >> 29) & 0x7FFFFFu));
    return (b << 1) == 0 ? __uint_as_float(sign) : (float)(scale * v);
}
__device__ __forceinline__ int scale_exponent(double scale) { return ((__double2hiint(scale) >> 20) & 0x7FF) - 1023; }
// Storage reals of the compute precision from FP64, and back (exact).
__device__ __forceinline__ void low_of(double &w, double v, int, double scale) { w = scale * v; }
__device__ __forceinline__ void low_of(float &w, double v, int m, double scale) { w = float_of(v, m, scale); }
__device__ __forceinline__ double high_of(double w) { return w; }
__device__ __forceinline__ double high_of(float w) { return wide(w); }

// lo = scale * hi  (scale = 2 kappa / sigma: the normalised defect), times T^-1
// of the site when a.clov is set
template <class P>
__global__ void __launch_bounds__(384) k_to_low(const __grid_constant__ ConvArgs a) {
    using R = typename P::real;
    __shared__ __align__(16) Item it;
    load_item(a.L, it);
    TileCoord tc = tile_coord(it, a.L);
    if (!tc.valid) return;
    int64_t i = tc.cb + tc.h;
    const double sc = a.st[it.solve0 + tc.col].scale;
    const int m = scale_exponent(sc);
    double v[24];
    load_spinor<PF64>(a.hi, i, v);
    R w[24];
#pragma unroll
    for (int j = 0; j < 24; j++) {
        if (sc == 0.0)
            w[j] = R(0);
        else
            low_of(w[j], v[j], m, sc);
    }
    if (a.clov && it.clovinv) clover_apply<R>(it.clovinv, it.gV, site_row(it, tc.h, a.p), w);
    store_spinor<P>(a.lo, i, w);
}

// hi += sigma * lo  (FP64 accumulation of the correction)
template <class P>
__global__ void __launch_bounds__(384) k_accum(const __grid_constant__ ConvArgs a) {
    using R = typename P::real;
    __shared__ __align__(16) Item it;
    load_item(a.L, it);
    TileCoord tc = tile_coord(it, a.L);
    if (!tc.valid) return;
    int64_t i = tc.cb + tc.h;
    const double sg = a.st[it.solve0 + tc.col].sigma;
    if (sg == 0.0) return;
    R w[24];
    load_spinor<P>(a.lo, i, w);
    double v[24];
    load_spinor<PF64>(a.hi, i, v);
#pragma unroll
    for (int j = 0; j < 24; j++) v[j] = fma(sg, high_of(w[j]), v[j]);
    store_spinor<PF64>(a.hi, i, v);
}

// ------------------------------------------------------------ scalar updates

enum FinOp { FIN_BNORM = 0, FIN_RESID = 1, FIN_INIT = 2, FIN_ALPHA = 3, FIN_OMEGA = 4 };

struct FinArgs {
    SolveState *st;
    int nsolve;
    Partials A, B;  // B used by FIN_BNORM / FIN_RESID (odd parity)
    LoopCtl *ctl;
    // FIN_OMEGA decides whether an inner iteration is the last: its last block to finish also runs
    // the loop control (0: not in a loop; 1: sets the graph's WHILE condition; 2: host-polled)
    int loop_mode;
    cudaGraphConditionalHandle loop;
};

// One block per solve: fixed-order sum of the solve's tile partials (of type R), then the scalar
// recurrences of BiCGStab or of the defect correction.  FIN_OMEGA finds omega and the scalars of
// the next iteration from the five products of the (t, s) stencil (bicg_omega, which says how good
// they are), so that x, r and p are updated in one pass and an iteration has two reductions.
constexpr int FIN_THREADS = 256;
template <int FIN, typename R>
__global__ void __launch_bounds__(FIN_THREADS) k_fin(FinArgs a) {
    using T = typename SumOf<R>::type;
    constexpr int NV = FIN == FIN_OMEGA ? PART_MAX : FIN == FIN_ALPHA ? 2 : 1;
    constexpr bool two = (FIN == FIN_BNORM || FIN == FIN_RESID);
    __shared__ T sh[FIN_THREADS / 32][NV];
    const int s = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    SolveState &S = a.st[s];
    chain_wait();
    chain_next();
    const int nt = S.ntiles, active = S.active;
    const int64_t base = S.pbase;
    // the state the recurrence starts from, read while the partials are on their way
    const Cnum rho = S.rho, inv = S.inv;
    const double target2 = S.target2;
    T v[NV];
#pragma unroll
    for (int k = 0; k < NV; k++) sum_zero(v[k]);
    const bool wanted = !(FIN == FIN_ALPHA || FIN == FIN_OMEGA) || active == 1;
    if (wanted) {
        const R *A = reinterpret_cast<const R *>(a.A.d) + base * NV, *B = reinterpret_cast<const R *>(a.B.d) + base;
        for (int t = threadIdx.x; t < nt; t += FIN_THREADS) {
            R c[NV];
#pragma unroll
            for (int k = 0; k < NV; k++) c[k] = ld_field(A + (int64_t)t * NV + k);
#pragma unroll
            for (int k = 0; k < NV; k++) sum_add(v[k], c[k]);
            if (two) sum_add(v[0], ld_field(B + t));
        }
    }
    // the lanes split the values as the distance halves: value k ends in lane k * 32 / NV
    int off = 16;
#pragma unroll
    for (int n = NV; n > 1; n >>= 1, off >>= 1) {
        const bool up = lane & off;
#pragma unroll
        for (int i = 0; i < n / 2; i++) {
            const T keep = up ? v[i + n / 2] : v[i], send = up ? v[i] : v[i + n / 2];
            v[i] = sum_join(keep, sum_shfl_xor(send, off));
        }
    }
#pragma unroll
    for (; off > 0; off >>= 1) v[0] = sum_join(v[0], sum_shfl_xor(v[0], off));
    if ((lane & (32 / NV - 1)) == 0) sh[warp][lane / (32 / NV)] = v[0];
    __syncthreads();
    if (warp != 0) return;
    double q = 0.0;
    if (lane < NV) {
        T p[FIN_THREADS / 32];
#pragma unroll
        for (int k = 0; k < FIN_THREADS / 32; k++) p[k] = sh[k][lane];
#pragma unroll
        for (int n = FIN_THREADS / 64; n > 0; n >>= 1)
#pragma unroll
            for (int k = 0; k < n; k++) p[k] = sum_join(p[2 * k], p[2 * k + 1]);
        q = sum_value(p[0]);
    }
    double w[NV];
#pragma unroll
    for (int k = 0; k < NV; k++) w[k] = __shfl_sync(0xffffffffu, q, k);
    if (lane != 0) return;
    const Cnum c0 = cn(0.0, 0.0), c1 = cn(1.0, 0.0);
    if constexpr (FIN == FIN_BNORM) {
        S.bnorm2 = w[0];
        S.outer_done = S.outer_done || (w[0] == 0.0);
    } else if constexpr (FIN == FIN_RESID) {
        const double n = w[0];
        if (S.outer_done) {  // converged earlier: its residual was not recomputed
            S.sigma = 0;
            S.scale = 0;
            return;
        }
        S.rr64 = n;
        bool done = (n <= S.tol * S.tol * S.bnorm2) || !(n == n);
        S.outer_done = done ? 1 : 0;
        if (done) {
            S.sigma = 0;
            S.scale = 0;
        } else {
            // a power of two, so that the defect is scaled by its exponent (float_of)
            S.scale = __hiloint2double(__double2hiint(2.0 * S.kappa / sqrt(n)) & 0x7FF00000, 0);
            S.sigma = 2.0 * S.kappa / S.scale;
            double d = 0.5 * S.tol * sqrt(S.bnorm2 / n);
            d = fmax(d, S.floor_delta);
            S.delta = fmin(d, 0.1);
        }
    } else if constexpr (FIN == FIN_INIT) {
        S.rho = cn(w[0], 0.0);
        S.target2 = S.delta * S.delta * w[0];
        S.iters = 0;
        const bool act = (S.sigma > 0) && (w[0] > 0);
        S.active = act ? 1 : 0;
        S.status = act ? 0 : 4;
        set_scalar(S.alpha, S.alpha32, act ? c1 : c0);
        set_scalar(S.omega, S.omega32, act ? c1 : c0);
        set_scalar(S.beta, S.beta32, c0);
    } else if constexpr (FIN == FIN_ALPHA) {
        if (active == 1) {
            Cnum alpha, hv;
            if (bicg_alpha(rho, cn(w[0], w[1]), alpha, hv)) {
                S.inv = hv;
                set_scalar(S.alpha, S.alpha32, alpha);
            } else {
                S.active = 0;
                S.status = 2;
                set_scalar(S.alpha, S.alpha32, c0);
                set_scalar(S.omega, S.omega32, c0);
                set_scalar(S.beta, S.beta32, c0);
            }
        } else {
            S.active = 0;  // its last update has been made
        }
    } else if constexpr (FIN == FIN_OMEGA) {
        int going = 0;
        if (active == 1) {
            Cnum omega, rc, beta;
            int status = bicg_omega(w, target2, inv, omega, rc, beta);
            const int iters = S.iters + 1;
            S.iters = iters;
            S.total_iters++;
            if (!status && iters >= S.maxit) status = 3;
            set_scalar(S.omega, S.omega32, omega);
            if (status) {
                S.active = 2;
                S.status = status;
                set_scalar(S.beta, S.beta32, c0);
            } else {
                set_scalar(S.beta, S.beta32, beta);
                S.rho = rc;
                going = 1;
            }
        }
        if (a.loop_mode) {
            // the block that decides the last solve also decides whether the loop goes on: one
            // atomic carries both counts, so no fence is needed
            LoopCtl *c = a.ctl;
            const unsigned long long mine = 1ull + ((unsigned long long)going << 32);
            const unsigned long long sum = atomicAdd(&c->arrived, mine) + mine;
            if ((unsigned)sum == (unsigned)a.nsolve) {
                const int cont = (sum >> 32) > 0 && (++c->iter < c->maxit);
                c->arrived = 0;
                if (a.loop_mode == 1)
                    cudaGraphSetConditional(a.loop, cont ? 1u : 0u);
                else
                    c->pad = cont;
            }
        }
    }
}

// ---------------------------------------------- user layout <-> even-odd fields
//
// User spinors: [ncol][n][4][3] complex, domain-local lexicographic order.
// One launch per item; thread per (column, site).

struct PackArgs {
    Item it;
    const double2 *user;  // eta (pack) or NULL for a point source
    double2 *uout;        // unpack target
    FieldView fe, fo;     // FP64 even / odd fields
    FieldView xe, xo;     // pack: solution fields zeroed at the same sites (p == NULL: untouched)
    int src_l;            // point source local index (pack with user == NULL)
};

__device__ __forceinline__ void local_coords(const Item &it, int l, int k[4]) {
    k[3] = l % it.e[3];
    l /= it.e[3];
    k[2] = l % it.e[2];
    l /= it.e[2];
    k[1] = l % it.e[1];
    k[0] = l / it.e[1];
}

static __global__ void k_pack(PackArgs a) {
    int64_t n = 2 * (int64_t)a.it.nh;
    int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= n * a.it.ncol) return;
    int col = (int)(g / n);
    int l = (int)(g - (int64_t)col * n);
    int k[4];
    local_coords(a.it, l, k);
    int par = (a.it.par_o + k[0] + k[1] + k[2] + k[3]) & 1;
    int64_t i = a.it.fbase + (int64_t)col * a.it.nh + (l >> 1);
    double v[24];
    if (a.user) {
        const double2 *u = a.user + ((int64_t)col * n + l) * 12;
#pragma unroll
        for (int j = 0; j < 12; j++) {
            double2 c = u[j];
            v[2 * j] = c.x;
            v[2 * j + 1] = c.y;
        }
    } else {
#pragma unroll
        for (int j = 0; j < 24; j++) v[j] = 0.0;
        if (l == a.src_l) v[2 * col] = 1.0;  // column c = 3 spin + colour is component c
    }
    store_spinor<PF64>(par ? a.fo : a.fe, i, v);
    if (a.xe.p) {
#pragma unroll
        for (int j = 0; j < 24; j++) v[j] = 0.0;
        store_spinor<PF64>(par ? a.xo : a.xe, i, v);
    }
}

static __global__ void k_unpack(PackArgs a) {
    int64_t n = 2 * (int64_t)a.it.nh;
    int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= n * a.it.ncol) return;
    int col = (int)(g / n);
    int l = (int)(g - (int64_t)col * n);
    int k[4];
    local_coords(a.it, l, k);
    int par = (a.it.par_o + k[0] + k[1] + k[2] + k[3]) & 1;
    int64_t i = a.it.fbase + (int64_t)col * a.it.nh + (l >> 1);
    double v[24];
    load_spinor<PF64>(par ? a.fo : a.fe, i, v);
    double2 *u = a.uout + ((int64_t)col * n + l) * 12;
#pragma unroll
    for (int j = 0; j < 12; j++) u[j] = make_double2(v[2 * j], v[2 * j + 1]);
}

// Low-precision pack/unpack (for applying the low-precision stencil alone).
template <class P>
__global__ void k_pack_low(PackArgs a, FieldView le, FieldView lo) {
    using R = typename P::real;
    int64_t n = 2 * (int64_t)a.it.nh;
    int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= n * a.it.ncol) return;
    int col = (int)(g / n);
    int l = (int)(g - (int64_t)col * n);
    int k[4];
    local_coords(a.it, l, k);
    int par = (a.it.par_o + k[0] + k[1] + k[2] + k[3]) & 1;
    int64_t i = a.it.fbase + (int64_t)col * a.it.nh + (l >> 1);
    const double2 *u = a.user + ((int64_t)col * n + l) * 12;
    R v[24];
#pragma unroll
    for (int j = 0; j < 12; j++) {
        double2 c = u[j];
        v[2 * j] = (R)c.x;
        v[2 * j + 1] = (R)c.y;
    }
    store_spinor<P>(par ? lo : le, i, v);
}

template <class P>
__global__ void k_unpack_low(PackArgs a, FieldView le, FieldView lo) {
    using R = typename P::real;
    int64_t n = 2 * (int64_t)a.it.nh;
    int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= n * a.it.ncol) return;
    int col = (int)(g / n);
    int l = (int)(g - (int64_t)col * n);
    int k[4];
    local_coords(a.it, l, k);
    int par = (a.it.par_o + k[0] + k[1] + k[2] + k[3]) & 1;
    int64_t i = a.it.fbase + (int64_t)col * a.it.nh + (l >> 1);
    R v[24];
    load_spinor<P>(par ? lo : le, i, v);
    double2 *u = a.uout + ((int64_t)col * n + l) * 12;
#pragma unroll
    for (int j = 0; j < 12; j++) u[j] = make_double2((double)v[2 * j], (double)v[2 * j + 1]);
}

// ------------------------------------------------ FP64 hopping on the integer pipe

// An FP64 field into block fixed point (fx64.cuh), one pass; a.skip as in HopArgs.
struct FxArgs {
    Launch L;
    FieldView in, fx;
    const SolveState *st;
    int skip;
};

static __global__ void __launch_bounds__(384) k_to_fx(const __grid_constant__ FxArgs a) {
    __shared__ __align__(16) Item it;
    load_item(a.L, it);
    const TileCoord tc = tile_coord(it, a.L);
    if (!tc.valid) return;
    if (a.skip) {
        const SolveState &S = a.st[it.solve0 + tc.col];
        if (skipped(S, a.skip)) return;
    }
    double v[24];
    load_spinor<PF64>(a.in, tc.cb + tc.h, v);
    fx_store_doubles(a.fx, tc.cb + tc.h, v);
}

// A block of k_hop_fx takes the group's columns in FX_SPLIT parts, FX_MINB blocks to an SM: 16
// warps of 128 registers instead of 12 of 160 in one block (residual of 16x24^3, 12 columns, FP16
// solve 48.5 -> 47.6 ms, eighth power 10.04 -> 9.91; 2 x 6 and 3 x 4 columns of 160 registers lose
// to the links' staging, which every part repeats).
constexpr int FX_SPLIT = 3, FX_MINB = 4;
constexpr int FX_MAX_THREADS = HOP_TS * ((HOP_MAX_CG + FX_SPLIT - 1) / FX_SPLIT);
__host__ __device__ constexpr int fx_cols(int CG) { return (CG + FX_SPLIT - 1) / FX_SPLIT; }

// k_hop at FP64 accuracy: a.in is in block fixed point, the epilogue and its operands are FP64
// (OUTFX: the plain sums are stored in block fixed point instead, for the next hop).  Blocks as
// k_hop: the oriented links of a 32-site tile are staged once, as integers, for the columns.
// About 6000 instructions per site-column, 1728 of them the widening multiply-adds and 1700 not of
// the hop (staging, which each of the FX_SPLIT parts repeats, and the epilogue), instead of 864
// on the FP64 pipe at 1/32 of the rate: 2.10 -> 0.56 ms for the plain sums of 110592 sites x 12
// columns (16x24^3, one parity).  The sums alone are 48 registers, a neighbour 48, its projection
// 24, so there are few warps (16 an SM): the multiply-add pipe is 55% busy, issue 35%, the rest
// waits for neighbours (L2) and for the staging.
template <int EPI, int DOT, bool CLOV, bool OUTFX>
__global__ void __launch_bounds__(FX_MAX_THREADS, FX_MINB) k_hop_fx(const __grid_constant__ HopArgs a) {
    constexpr int TS = HOP_TS;
    // this block's columns: cgh of the group's CG, from part * cgh
    const int blk = blockIdx.x / FX_SPLIT, part = blockIdx.x % FX_SPLIT, cgh = fx_cols(a.L.CG);
    if (part * cgh >= a.L.CG) return;
    auto coord = [&](const Item &it) {
        TileCoord t = tile_coord(it, a.L, blk);
        const int cl = threadIdx.x / TS;
        t.col += part * cgh;
        t.cb += (int64_t)part * cgh * it.nh;
        t.valid = t.h < it.nh && t.col < it.ncol && part * cgh + cl < a.L.CG;
        return t;
    };
    __shared__ __align__(16) Item it;
    __shared__ int s_nb[8 * TS];
    __shared__ __align__(16) int4 s_u[8 * TS * 9];
    load_item(a.L, it, blk);
    if (a.skip) {
        const int cg = fdiv(blk - it.blk0, it.by_nt);
        const int col = cg * a.L.CG + part * cgh + (int)threadIdx.x;
        int live = 0;
        if ((int)threadIdx.x < cgh && part * cgh + (int)threadIdx.x < a.L.CG && col < it.ncol) {
            const SolveState &S = a.st[it.solve0 + col];
            live = !skipped(S, a.skip);
        }
        if (!__syncthreads_or(live)) return;
    }
    {
        const int lb = blk - it.blk0, tile = lb - fdiv(lb, it.by_nt) * it.ntiles;
        for (int q = threadIdx.x; q < 8 * TS; q += blockDim.x) {
            const int d = q / TS, h = tile * TS + (q - d * TS);
            int nb = -1;
            if (h < it.nh) {
                int64_t row = 0;
                bool neg;
                nb = hop_geometry(it, h, a.p, d, row, neg);
                if (nb >= 0) {
                    const double2 *l = reinterpret_cast<const double2 *>(it.links64) + (int64_t)(d >> 1) * 9 * it.gV + row;
                    const bool adj = d & 1;
#pragma unroll
                    for (int j = 0; j < 9; j++) {
                        const double2 c = __ldg(l + j * it.gV);
                        long long re = fx_link(c.x), im = fx_link(c.y);
                        if (neg) re = -re;
                        if (neg != adj) im = -im;  // the adjoint's conjugate, and the sign
                        int4 e;
                        fx_split(re, e.x, e.y);
                        fx_split(im, e.z, e.w);
                        s_u[q * 9 + (adj ? 3 * (j % 3) + j / 3 : j)] = e;
                    }
                }
            }
            s_nb[q] = nb;
        }
    }
    __syncthreads();
    TileCoord tc = coord(it);
    if (a.skip && tc.valid) {
        const SolveState &S = a.st[it.solve0 + tc.col];
        if (skipped(S, a.skip)) tc.valid = false;
    }
    double sums[PART_MAX] = {};
    if (tc.valid) {
        const int sl = tc.h - tc.tile * TS;
        int e[8], top = FX_ZERO;
#pragma unroll
        for (int d = 0; d < 8; d++) {
            const int nb = s_nb[d * TS + sl];
            e[d] = nb >= 0 ? __ldg(fx_exponents(a.in) + tc.cb + nb) : FX_ZERO;
            top = max(top, e[d]);
        }
        if (top != FX_RAW) {
            long long sum[24];
#pragma unroll
            for (int j = 0; j < 24; j++) sum[j] = 0;
#define DDP_FX_STEP(D)                                                                        \
            {                                                                                 \
                const int nb = s_nb[(D) * TS + sl];                                           \
                if (nb >= 0) {                                                                \
                    const int4 *b = reinterpret_cast<const int4 *>(a.in.p) + tc.cb + nb;      \
                    int4 v[12];                                                               \
                    _Pragma("unroll") for (int j = 0; j < 12; j++) v[j] = __ldg(b + j * a.in.stride); \
                    fx_hop_step<D>(v, s_u + ((D) * TS + sl) * 9, sum, min(62, top - e[D]));   \
                }                                                                             \
            }
            DDP_FX_STEP(0)
            DDP_FX_STEP(1)
            DDP_FX_STEP(2)
            DDP_FX_STEP(3)
            DDP_FX_STEP(4)
            DDP_FX_STEP(5)
            DDP_FX_STEP(6)
            DDP_FX_STEP(7)
#undef DDP_FX_STEP
            if (OUTFX) {
                fx_store_sums(a.out, tc.cb + tc.h, sum, top - FX_LINK);
            } else {
                cx<double> acc[4][3];
#pragma unroll
                for (int j = 0; j < 12; j++)
                    acc[j / 3][j % 3] = mk(fx_value(sum[2 * j], top - FX_LINK), fx_value(sum[2 * j + 1], top - FX_LINK));
                hop_store_epilogue<PF64, EPI, DOT, CLOV>(a, it, tc, acc, sums);
            }
        } else {
            double o[24];
            fx_slow<TS>(a.in, tc.cb, s_nb + sl, s_u + sl * 9, o);
            if (OUTFX) {
                fx_store_doubles(a.out, tc.cb + tc.h, o);
            } else {
                cx<double> acc[4][3];
                for (int j = 0; j < 12; j++) acc[j / 3][j % 3] = mk(o[2 * j], o[2 * j + 1]);
                hop_store_epilogue<PF64, EPI, DOT, CLOV>(a, it, tc, acc, sums);
            }
        }
    }
    if (DOT != DOT_NONE) {
        if (part * cgh + (int)(threadIdx.x / TS) >= a.L.CG) tc.col = it.ncol;  // no column: nothing to write
        warp_partials<DOT != DOT_NONE ? dot_sums(DOT) : 1>(it, tc, sums, a.part);
    }
}

// User layout <-> block fixed point (the stencil powers); unpacking multiplies by s.
static __global__ void k_pack_fx(PackArgs a, FieldView le, FieldView lo) {
    int64_t n = 2 * (int64_t)a.it.nh;
    int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= n * a.it.ncol) return;
    int col = (int)(g / n);
    int l = (int)(g - (int64_t)col * n);
    int k[4];
    local_coords(a.it, l, k);
    int par = (a.it.par_o + k[0] + k[1] + k[2] + k[3]) & 1;
    const double2 *u = a.user + ((int64_t)col * n + l) * 12;
    double v[24];
#pragma unroll
    for (int j = 0; j < 12; j++) {
        double2 c = u[j];
        v[2 * j] = c.x;
        v[2 * j + 1] = c.y;
    }
    fx_store_doubles(par ? lo : le, a.it.fbase + (int64_t)col * a.it.nh + (l >> 1), v);
}

static __global__ void k_unpack_fx(PackArgs a, FieldView le, FieldView lo, double s) {
    int64_t n = 2 * (int64_t)a.it.nh;
    int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= n * a.it.ncol) return;
    int col = (int)(g / n);
    int l = (int)(g - (int64_t)col * n);
    int k[4];
    local_coords(a.it, l, k);
    int par = (a.it.par_o + k[0] + k[1] + k[2] + k[3]) & 1;
    double v[24];
    fx_load_doubles(par ? lo : le, a.it.fbase + (int64_t)col * a.it.nh + (l >> 1), v);
    double2 *u = a.uout + ((int64_t)col * n + l) * 12;
#pragma unroll
    for (int j = 0; j < 12; j++) u[j] = make_double2(s * v[2 * j], s * v[2 * j + 1]);
}

}  // namespace ddp
