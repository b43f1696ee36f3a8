// The two contraction-shaped steps of the projector-cut factorization (Sec. 5) on the
// tensor cores with FP64-level accuracy: the time-slice sums of the colourless spinors
// (Eq. W0tbary) and the Gram blocks conj(A_i) . A_j (the pion blocks of Eq. Bpions and
// the Cholesky QR of the inverse iteration), both as one emulated-FP64 product kernel.
//
// Colourless spinors.  Per time slice the sum is a complex matrix product
//   X[(i,j)][(k,alpha)] = sum_{(x,c)} E[(i,j)][(x,c)] s_k(x)_{alpha c},
//   E[(i,j)][(x,c)] = sum_{ab} eps_abc (s_i^a)^T C g5 s_j^b          (the diquark, FP64).
// C g5 is antisymmetric, so E is symmetric in (i, j): only the m(m+1)/2 rows i <= j
// are formed and X[j][i] = X[i][j].  The complex product is one real product
// C' = A' B'^T with A' = [Re E | Im E] and the rows of B' = [Re s | -Im s] (real-part
// columns) and [Im s | Re s] (imaginary-part columns).
//
// Every row of A' and every column of B' is split into S integer slices of 7 bits
// under a shared power-of-two exponent (the splitting of Ozaki, Ogita, Oishi and Rump,
// 2012): with |a| < 2^e over the row (column), N = round(a 2^(49-e)) is written in
// balanced base 128, a = 2^(e-7) sum_p q_p 2^(-7p) + O(2^(e-50)), q_0 in [-128, 128],
// q_p in [-64, 63] for p > 0, each exact in BF16.  For every d < S the products of slices
// p + q = d are summed on the tensor cores (tcgen05.mma kind::f16, BF16 operands,
// FP32 accumulators in tensor memory, one per d).  Over KC = 448 reduction terms
// every such sum is an integer of magnitude below 9 * 2^12 * 448 < 2^24, hence
// exact in FP32; after each chunk the seven sums are converted to integers and
// added exactly into two 64-bit fixed-point accumulators per output.  Products of
// slices with p + q >= S are dropped: each term of the sum is exact to about
// 2^-47 of its row maximum times its column maximum.
//
// Operands reach the tensor cores through a five-stage pipeline of bulk copies
// (cp.async.bulk, completion on an mbarrier): the split kernels write every
// (slice, 128- or 64-row tile, 16-deep K step) block contiguously in the
// shared-memory layout the MMA descriptor describes (K-major, no swizzle: 8-row x
// 16-byte core matrices, 128 bytes apart along K, 256 bytes apart between 8-row
// groups), so that one copy per block stages it (seven for the columns of large Gram blocks).
#include <algorithm>
#include <cmath>
#include <cstring>

#include "ddp_host.h"

using namespace ddp;

namespace {

constexpr int S = 7;          // slices per operand; accumulator groups d = p + q < S
constexpr int TM = 128;       // rows of A' per tile (the MMA's M)
constexpr int TN = 64;        // rows of B' (output columns) per tile (the MMA's N)
constexpr int KSTEP = 16;     // reduction depth per pipeline stage (one MMA of K = 16 per slice pair)
constexpr int CS = 28;        // stages per exact chunk: KC = 448
constexpr int SBO = 16 * KSTEP, LBO = 128;  // bytes between 8-row groups; between K core matrices
constexpr int TILE_A = TM * KSTEP * 2, TILE_B = TN * KSTEP * 2;  // bytes
constexpr int STAGE = S * (TILE_A + TILE_B);
constexpr int NSTAGE = 5;   // operand buffers in flight
constexpr int GEMM_THREADS = 512;   // all drain; one lane loads, one issues the MMAs
constexpr int GEMM_BLOCK = GEMM_THREADS;
constexpr int MMA_WARP = 0, PRODUCER_WARP = 5;  // on different quarters of the SM
constexpr int DCOLS = TN / (GEMM_THREADS / 128);  // accumulator columns a thread drains
constexpr int TMEM_COLS = 512;  // S * TN = 448 used
constexpr int MAX_STEPS_PER_BLOCK = 1 << 16;  // keeps the fixed-point sums far below 2^63
constexpr int MMAX = TC_MMAX; // largest number of columns (the paper's 120 modes fit)
// sites per block of the diquark kernel: all m spinors of the block's sites are staged in
// shared memory, m * ES * 192 bytes (16 sites up to 32 columns, 4 beyond, plus 64 bytes
// of padding per column)
constexpr int ES_SMALL = 16, ES_LARGE = 4, ES_SMALL_MMAX = 32;
// float4 elements between the staged spinors of consecutive columns k
__host__ __device__ constexpr int colour_kstride(int es) { return 12 * es + (es == 4 ? 4 : 0); }
constexpr unsigned long long WAIT_NS = 2000000000ull;  // a wait gives up after 2 s

static_assert(S * TN <= TMEM_COLS, "accumulators exceed the tensor memory");
static_assert(4 * TN <= 256, "one MMA spans at most four B slices (N <= 256)");
static_assert(DCOLS == 16, "the drain loads 16 columns per thread");
static_assert(CS * KSTEP * 9 * 4096 < (1 << 24), "chunk sums must stay exact in FP32");

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t mma_desc(uint32_t saddr) {
    return ((uint64_t)(saddr >> 4) & 0x3FFF) | ((uint64_t)((LBO >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((SBO >> 4) & 0x3FFF) << 32) | (1ull << 46);
}

// kind::f16 instruction descriptor: FP32 accumulator, BF16 A and B, both K-major, M = TM.
__host__ __device__ constexpr uint32_t idesc_n(int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
}

__device__ __forceinline__ uint64_t globaltimer() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Bounded wait for the completion of the mbarrier phase with the given parity.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    uint64_t t0 = 0;  // read only after some tries: most waits are short
    for (uint32_t it = 0;; it++) {
        uint32_t ok;
        asm volatile("{\n .reg .pred pw;\n mbarrier.try_wait.parity.shared::cta.b64 pw, [%1], %2;\n"
                     " selp.u32 %0, 1, 0, pw;\n}\n"
                     : "=r"(ok)
                     : "r"(bar), "r"(parity)
                     : "memory");
        if (ok) return true;
        if ((it & 255u) == 255u) {
            const uint64_t t = globaltimer();
            if (t0 == 0)
                t0 = t;
            else if (t - t0 > WAIT_NS)
                return false;
        }
    }
}

__device__ __forceinline__ void atomic_max_pos(double *a, double v) {
    // non-negative doubles order like their bit patterns
    atomicMax(reinterpret_cast<unsigned long long *>(a), (unsigned long long)__double_as_longlong(v));
}

__device__ __forceinline__ int exponent_of(double mx) {
    if (!(mx > 0)) return 0;
    int e;
    frexp(mx, &e);  // mx < 2^e
    return e;
}

// The shared exponent of every row or column: e with max < 2^e, or NONFINITE for a
// row or column that holds a NaN or an infinity (its slices are zero and its outputs NaN).
constexpr int NONFINITE = -100000;
__global__ void k_exponents(const double *mx, int n, int *ex) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) ex[i] = isfinite(mx[i]) ? exponent_of(mx[i]) : NONFINITE;
}

// (i, j), i <= j, of the symmetric row r (rows ordered i-major).
__device__ __forceinline__ void pair_of(int r, int m, int &i, int &j) {
    i = 0;
    while (r >= m - i) {
        r -= m - i;
        i++;
    }
    j = i + r;
}

// ------------------------------------------------------------- pre-passes
//
// GB300 runs FP64 arithmetic at a small fraction of its FP32 rate, so the pre-passes
// avoid it: the diquarks are formed in double-FP32 arithmetic (each value an unevaluated
// sum hi + lo of two floats, 48 significant bits; Dekker's product with fused
// multiply-adds and Knuth's two-sum), and the 7-bit slices are cut from the integer
// round(v 2^(49-e)) obtained from the bit pattern of v by shifts.
//
// The diquarks are bound by the FP32 pipe (24 complex products of 24 operations on lane pairs for
// every row and site), the other pre-passes by their stores: a thread cuts 8 steps of the reduction
// and writes 16 bytes per slice.  Per time slice of 24^3 sites and 24 columns: maxima 37 -> 20 us
// (were compared in FP64), diquarks 243 -> 196 (were one lane per instruction), slices of the
// diquarks 162 -> 129 and of the spinors 93 -> 51 (were 2 bytes per store, every spinor cut twice).

// Magnitude used for the shared exponents: +inf for a non-finite value, so that a NaN or
// an infinity in the input turns the affected outputs into NaN (see k_ozaki_finish).
__device__ __forceinline__ float magf(float v) { return isfinite(v) ? fabsf(v) : INFINITY; }

// 2^k as a float, -126 <= k <= 127.
__device__ __forceinline__ float pow2f(int k) { return __int_as_float((127 + k) << 23); }

// hi + lo = v 2^-f to 48 significant bits, from the bits of v by integer operations
// (|v| < 2^f; parts below 2^-100 of 2^f, irrelevant at the 2^-49 precision of the
// slices, are dropped; a non-finite v gives NaN).
__device__ __forceinline__ float2 df_scaled(double v, int f) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const int ev = (int)((b >> 52) & 0x7FF);
    if (ev == 0x7FF) return make_float2(NAN, NAN);
    const int e = ev - 1023 - f;  // v 2^-f = 1.m 2^e
    if (ev == 0 || e < -100) return make_float2(0.f, 0.f);
    const unsigned long long m = (b & ((1ull << 52) - 1)) | (1ull << 52);
    const unsigned long long mh = (m + (1ull << 28)) >> 29;  // the significand rounded to 24 bits
    const long long rem = (long long)m - (long long)(mh << 29);  // |rem| <= 2^28
    const float sc = pow2f(e - 23);
    float hi = __uint2float_rn((unsigned)mh) * sc;                    // exact
    float lo = (__ll2float_rn(rem) * 3.7252902984619140625e-9f) * sc;  // rem 2^-28 2^(e-23) ... 2^-1
    lo *= 0.5f;                                                          // rem 2^(e-52)
    if (b >> 63) {
        hi = -hi;
        lo = -lo;
    }
    return make_float2(hi, lo);
}

// (s, e) += a * b lane by lane for double-floats a = ah + al, b = bh + bl; (s, e) is an unnormalized
// sum (Knuth's two-sum; the rounding errors are collected in e).
__device__ __forceinline__ void df2_mac(float2 &s, float2 &e, float2 ah, float2 al, float2 bh, float2 bl) {
    const float2 neg = make_float2(-1.f, -1.f);  // x - y = fma(y, -1, x)
    const float2 p = __fmul2_rn(ah, bh);
    float2 d = __ffma2_rn(ah, bh, make_float2(-p.x, -p.y));
    d = __ffma2_rn(ah, bl, d);
    d = __ffma2_rn(al, bh, d);
    const float2 t = __fadd2_rn(s, p);
    const float2 bb = __ffma2_rn(s, neg, t);
    const float2 u = __ffma2_rn(__ffma2_rn(bb, neg, t), neg, s), w = __ffma2_rn(bb, neg, p);
    e = __fadd2_rn(e, __fadd2_rn(__fadd2_rn(u, w), d));
    s = t;
}

// hi + lo = (s0 + e0) + sg (s1 + e1) of two such sums.
__device__ __forceinline__ float2 df_join(float s0, float e0, float s1, float e1, float sg) {
    s1 *= sg;
    const float s = __fadd_rn(s0, s1), bb = __fsub_rn(s, s0);
    const float err = __fadd_rn(__fsub_rn(s0, __fsub_rn(s, bb)), __fsub_rn(s1, bb));
    const float e = __fadd_rn(err, __fmaf_rn(sg, e1, e0)), h = __fadd_rn(s, e);
    return make_float2(h, __fsub_rn(e, __fsub_rn(h, s)));
}

// Column maxima of the spinors over one time slice: colmax[q], q = (k, alpha), the power of two
// (with the leading bits) of the largest |Re|, |Im| of s_k(x)_{alpha c} over x and c; infinite for a
// value that is not finite.  Compared as the integers of their high words: FP64 comparisons run on
// the FP64 pipe.
__device__ __forceinline__ unsigned mag_hi(double v) {
    const unsigned h = (unsigned)__double2hiint(v) & 0x7FFFFFFFu;
    return max(min(h, 0x7FF00000u), (unsigned)(__double2loint(v) != 0));  // bounds a subnormal too
}
__global__ void __launch_bounds__(256) k_colour_max(const double2 *A, int64_t n, int64_t site0, int64_t slice_n,
                                                    int m, double *colmax) {
    __shared__ unsigned bm[4 * MMAX];
    const int Q = 4 * m;
    for (int q = threadIdx.x; q < Q; q += blockDim.x) bm[q] = 0;
    __syncthreads();
    // consecutive threads: the spins of a site, then the next columns; groups of threads share the sites
    const int per = max(1, (int)blockDim.x / Q);
    if ((int)threadIdx.x < per * Q || per * Q > (int)blockDim.x)
        for (int q = threadIdx.x % (per * Q); q < per * Q; q += blockDim.x) {
            const int c4 = q % Q, k = c4 / 4, al = c4 % 4;
            unsigned mx = 0;
            for (int64_t x = blockIdx.x * (int64_t)per + q / Q; x < slice_n; x += (int64_t)gridDim.x * per) {
                const double2 *v = A + ((int64_t)k * n + site0 + x) * 12 + 3 * al;
                const double2 v0 = __ldg(v), v1 = __ldg(v + 1), v2 = __ldg(v + 2);
                mx = max(mx, max(max(mag_hi(v0.x), mag_hi(v0.y)), max(mag_hi(v1.x), mag_hi(v1.y))));
                mx = max(mx, max(mag_hi(v2.x), mag_hi(v2.y)));
            }
            if (mx) atomicMax(bm + c4, mx);
        }
    __syncthreads();
    for (int q = threadIdx.x; q < Q; q += blockDim.x)
        if (bm[q]) atomicMax(reinterpret_cast<unsigned *>(colmax + q) + 1, bm[q]);  // the high word
}

// f_k: |s_k(x)| < 2^f_k over the slice (the exponent of the spinor column k).
__device__ __forceinline__ int column_exponent(const double *colmax, int k) {
    return exponent_of(fmax(fmax(colmax[4 * k], colmax[4 * k + 1]), fmax(colmax[4 * k + 2], colmax[4 * k + 3])));
}

struct EArgs {
    const double2 *A;   // [m][n][12]
    int64_t n, site0, slice_n;
    int m, form, rows;  // rows = m (m + 1) / 2
    float4 *E;          // [rows][3 slice_n]: Re hi, Re lo, Im hi, Im lo of E 2^-(f_i + f_j)
    double *rowmax;     // [rows]   max |Re|, |Im| (hi parts) of the row of E 2^-(f_i + f_j)
    const double *colmax;
};

// The diquarks E^c_ij(x) = i sum over the spin pairs of Eq. W0tbary for i <= j, formed
// from the spinors scaled by 2^-f_k (so that double-FP32 arithmetic keeps its range),
// with the row maxima.  Block: ESITES sites, all rows; ESITES consecutive threads share a row.
template <int ESITES>
__global__ void __launch_bounds__(256) k_colour_E(EArgs a) {
    static_assert(ESITES >= 1 && ESITES <= 32 && (ESITES & (ESITES - 1)) == 0, "row groups within a warp");
    // [m][12][ESITES] with the site index fastest; with 4 sites the spinors of consecutive
    // k start 16 banks apart, so that the two rows a quarter-warp reads do not collide
    constexpr int KSTR = colour_kstride(ESITES);
    extern __shared__ float4 sh[];
    __shared__ int fexp[MMAX];
    const int m = a.m;
    const int64_t x0 = (int64_t)blockIdx.x * ESITES;
    const int ns = (int)min((int64_t)ESITES, a.slice_n - x0);
    for (int k = threadIdx.x; k < m; k += blockDim.x) fexp[k] = column_exponent(a.colmax, k);
    __syncthreads();
    for (int e = threadIdx.x; e < m * ns * 12; e += blockDim.x) {
        const int c = e % 12, xs = (e / 12) % ns, k = e / (12 * ns);
        const double2 v = a.A[((int64_t)k * a.n + a.site0 + x0 + xs) * 12 + c];
        float2 re = df_scaled(v.x, fexp[k]), im = df_scaled(v.y, fexp[k]);
        // the form, exactly on the parts: 1 conj then g5 (spins 0, 1 negated), 2 negation
        if (a.form == 1) im = make_float2(-im.x, -im.y);
        if ((a.form == 1 && c < 6) || a.form == 2) {
            re = make_float2(-re.x, -re.y);
            im = make_float2(-im.x, -im.y);
        }
        sh[k * KSTR + c * ESITES + xs] = make_float4(re.x, im.x, re.y, im.y);
    }
    __syncthreads();
    const int nit = a.rows * ESITES;
    for (int it0 = 0; it0 < nit; it0 += blockDim.x) {
        const int it = it0 + threadIdx.x;
        const int r = it / ESITES, xs = it % ESITES;
        float mx = 0.f;
        if (r < a.rows && xs < ns) {
            int i, j;
            pair_of(r, m, i, j);
            const float4 *si = sh + i * KSTR + xs, *sj = sh + j * KSTR + xs;
            float4 *o = a.E + (int64_t)r * 3 * a.slice_n + (x0 + xs) * 3;
            for (int c = 0; c < 3; c++) {
                const int ca = (c + 1) % 3, cb = (c + 2) % 3;
                // f(a, b) = s_i(1,a) s_j(0,b) - s_i(0,a) s_j(1,b) + s_i(3,a) s_j(2,b) - s_i(2,a) s_j(3,b);
                // E^c = i [f(ca, cb) - f(cb, ca)]
                // P = sum of Re s_i times (Re, Im) s_j, M = of Im s_i: E = i [(P.x - M.y) + i (P.y + M.x)]
                float2 P = make_float2(0.f, 0.f), Pe = P, M = P, Me = P;
                auto mac = [&](float4 x, float4 y, float sg) {  // Re hi, Im hi, Re lo, Im lo
                    const float2 yh = make_float2(y.x, y.y), yl = make_float2(y.z, y.w);
                    df2_mac(P, Pe, make_float2(sg * x.x, sg * x.x), make_float2(sg * x.z, sg * x.z), yh, yl);
                    df2_mac(M, Me, make_float2(sg * x.y, sg * x.y), make_float2(sg * x.w, sg * x.w), yh, yl);
                };
#pragma unroll
                for (int t = 0; t < 2; t++) {
                    const float sg = t ? -1.f : 1.f;
                    const int p = t ? cb : ca, q = t ? ca : cb;
                    mac(si[(3 + p) * ESITES], sj[q * ESITES], sg);
                    mac(si[p * ESITES], sj[(3 + q) * ESITES], -sg);
                    mac(si[(9 + p) * ESITES], sj[(6 + q) * ESITES], sg);
                    mac(si[(6 + p) * ESITES], sj[(9 + q) * ESITES], -sg);
                }
                const float2 R = df_join(P.x, Pe.x, M.y, Me.y, -1.f), I = df_join(P.y, Pe.y, M.x, Me.x, 1.f);
                o[c] = make_float4(-I.x, -I.y, R.x, R.y);  // times i
                mx = fmaxf(mx, fmaxf(magf(R.x), magf(I.x)));
            }
        }
        for (int off = ESITES / 2; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
        if ((threadIdx.x & (ESITES - 1)) == 0 && r < a.rows && mx > 0.f) atomic_max_pos(a.rowmax + r, (double)mx);
    }
}

// round(mant 2^(ee + k)), |result| < 2^62 by the caller's choice of k (half away from zero).
__device__ __forceinline__ long long fixed_round(unsigned long long mant, int sh, bool neg) {
    unsigned long long n;
    if (sh >= 0)
        n = mant << sh;
    else if (sh > -64)
        n = (mant + (1ull << (-sh - 1))) >> (-sh);
    else
        n = 0;
    return neg ? -(long long)n : (long long)n;
}

// round(v 2^k) from the bits of a finite double (subnormals included).
__device__ __forceinline__ long long fixed_of(double v, int k) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const int ev = (int)((b >> 52) & 0x7FF);
    const unsigned long long mant = (b & ((1ull << 52) - 1)) | (ev ? 1ull << 52 : 0ull);
    return fixed_round(mant, (ev ? ev : 1) - 1075 + k, b >> 63);
}

// round(f 2^k) from the bits of a finite float.
__device__ __forceinline__ long long fixed_of(float f, int k) {
    const unsigned b = __float_as_uint(f);
    const int ev = (int)((b >> 23) & 0xFF);
    const unsigned long long mant = (b & 0x7FFFFFu) | (ev ? 0x800000u : 0u);
    return fixed_round(mant, (ev ? ev : 1) - 150 + k, b >> 31);
}

// Digit p = 6 - k of N in balanced base 128 is bits 7k .. 7k + 6 of N + sum_k 64 128^k, less 64
// (k < 6); what lies above is digit 0.  Returned as FP32: an exact small integer.
__device__ __forceinline__ void digits7f(long long N, float q[S]) {
    constexpr unsigned long long BIAS = 64ull * (1 + (1ull << 7) + (1ull << 14) + (1ull << 21) + (1ull << 28) + (1ull << 35));
    const long long M = N + (long long)BIAS;
#pragma unroll
    for (int k = 0; k < S - 1; k++)
        q[S - 1 - k] = __int_as_float(0x4B400000 + ((int)(M >> (7 * k)) & 127)) - (12582912.f + 64.f);
    q[0] = __int_as_float(0x4B400000 + (int)(M >> 42)) - 12582912.f;
}
__device__ __forceinline__ unsigned pack_bf16(float a, float b) {
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<unsigned *>(&h);
}

// Byte offset of the 16-byte row (row r, depths 8 k8 .. 8 k8 + 7) in a tile block: 8-row groups of
// SBO bytes, core matrices of LBO.
__device__ __forceinline__ int tile_offset(int r, int k8) { return (r >> 3) * SBO + k8 * LBO + (r & 7) * 16; }
__device__ __forceinline__ void put_slices(uint8_t *base, int tile_bytes, const uint4 v[S], bool negate = false) {
    const unsigned x = negate ? 0x80008000u : 0u;
#pragma unroll
    for (int p = 0; p < S; p++)
        *reinterpret_cast<uint4 *>(base + (int64_t)p * tile_bytes) = make_uint4(v[p].x ^ x, v[p].y ^ x, v[p].z ^ x, v[p].w ^ x);
}
// The digits of two consecutive values into word j of every slice.
__device__ __forceinline__ void put_digits(uint4 v[S], int j, long long n0, long long n1) {
    float q0[S], q1[S];
    digits7f(n0, q0);
    digits7f(n1, q1);
#pragma unroll
    for (int p = 0; p < S; p++) {
        const unsigned w = pack_bf16(q0[p], q1[p]);
        if (j == 0) v[p].x = w;
        else if (j == 1) v[p].y = w;
        else if (j == 2) v[p].z = w;
        else v[p].w = w;
    }
}

struct SplitArgs {
    const float4 *E;
    const double2 *A;
    int64_t n, site0, K;  // K = 3 slice_n
    int m, form, rows;
    int MT, NT, KSh;      // tiles; K steps of one half (Re / Im) of the reduction
    const int *rexp, *cexp;  // exponents of the rows of A' and of the spinor columns (k, alpha)
    uint8_t *Aq, *Bq;        // [MT][2 KSh][S][128 x KSTEP], [NT][2 KSh][S][64 x KSTEP] BF16
};

// A' = [Re E | Im E]: thread per (row, 8 reduction steps), a 16-byte row of a core matrix of every
// slice of both halves; consecutive threads take consecutive rows, 8 of which are one core matrix.
// With |v| < 2^e for the row, v = 2^(e-49) round(v 2^(49-e)) to within half a unit.
__global__ void __launch_bounds__(256) k_split_A(SplitArgs a) {
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int rows = a.MT * TM;
    if (g >= 2 * (int64_t)a.KSh * rows) return;
    const int r = (int)(g % rows);
    const int64_t t = g / rows, ksr = t >> 1, kx = ksr * KSTEP + 8 * (t & 1);
    uint4 re[S], im[S];
#pragma unroll
    for (int p = 0; p < S; p++) re[p] = im[p] = make_uint4(0, 0, 0, 0);
    const int er = r < a.rows ? a.rexp[r] : NONFINITE;
    if (er != NONFINITE) {
        const float4 *src = a.E + (int64_t)r * a.K + kx;
        const int k = 49 - er;
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
            const float4 v0 = kx + 2 * j < a.K ? __ldg(src + 2 * j) : z, v1 = kx + 2 * j + 1 < a.K ? __ldg(src + 2 * j + 1) : z;
            put_digits(re, j, fixed_of(v0.x, k) + fixed_of(v0.y, k), fixed_of(v1.x, k) + fixed_of(v1.y, k));
            put_digits(im, j, fixed_of(v0.z, k) + fixed_of(v0.w, k), fixed_of(v1.z, k) + fixed_of(v1.w, k));
        }
    }
    // tile block (mt, K step, slice): the S slices of one step lie contiguously
    uint8_t *o = a.Aq + ((int64_t)(r / TM) * 2 * a.KSh + ksr) * S * TILE_A + tile_offset(r % TM, (int)(t & 1));
    put_slices(o, TILE_A, re);
    put_slices(o + (int64_t)a.KSh * S * TILE_A, TILE_A, im);
}

// B' rows: col < 4m: [Re s | -Im s]; 4m <= col < 8m: [Im s | Re s]; beyond: zero.  Thread per
// (spinor column q, 8 reduction steps), which serves both of its rows; and per zero row.
__global__ void __launch_bounds__(256) k_split_B(SplitArgs a) {
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int cols = a.NT * TN, Q = 4 * a.m;
    if (g >= 2 * (int64_t)a.KSh * (cols - Q)) return;
    // q < Q: spinor columns; Q <= q: the zero rows 2 Q, 2 Q + 1, ...
    const int q = (int)(g % (cols - Q));
    const int64_t t = g / (cols - Q), ksr = t >> 1, kx = ksr * KSTEP + 8 * (t & 1);
    uint4 re[S], im[S];
#pragma unroll
    for (int p = 0; p < S; p++) re[p] = im[p] = make_uint4(0, 0, 0, 0);
    const int eq = q < Q ? a.cexp[q] : NONFINITE;
    if (eq != NONFINITE) {
        const int al = q % 4, k = 49 - eq;
        const double2 *src = a.A + ((int64_t)(q / 4) * a.n + a.site0) * 12 + 3 * al;
        auto at = [&](int64_t i) {  // reduction index i = 3 x + c
            if (i >= a.K) return make_double2(0.0, 0.0);
            const int64_t x = i / 3;
            return __ldg(src + x * 12 + (i - 3 * x));
        };
        // the form's signs: conj and g5 (form 1), negation (form 2)
        const bool nre = a.form == 2 || (a.form == 1 && al < 2), nim = a.form == 2 || (a.form == 1 && al >= 2);
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const double2 v0 = at(kx + 2 * j), v1 = at(kx + 2 * j + 1);
            const long long r0 = fixed_of(v0.x, k), r1 = fixed_of(v1.x, k), i0 = fixed_of(v0.y, k), i1 = fixed_of(v1.y, k);
            put_digits(re, j, nre ? -r0 : r0, nre ? -r1 : r1);
            put_digits(im, j, nim ? -i0 : i0, nim ? -i1 : i1);
        }
    }
    const int64_t half = (int64_t)a.KSh * S * TILE_B;
    auto row = [&](int col) {
        return a.Bq + ((int64_t)(col / TN) * 2 * a.KSh + ksr) * S * TILE_B + tile_offset(col % TN, (int)(t & 1));
    };
    if (q < Q) {
        put_slices(row(q), TILE_B, re);
        put_slices(row(q) + half, TILE_B, im, true);
        put_slices(row(Q + q), TILE_B, im);
        put_slices(row(Q + q) + half, TILE_B, re);
    } else {
        put_slices(row(Q + q), TILE_B, re);
        put_slices(row(Q + q) + half, TILE_B, re);
    }
}

// -------------------------------------------------------------- the product

struct GemmArgs {
    const uint8_t *Aq, *Bq;  // Bq null: the columns are the rows of A' (gram_tc)
    int a_bytes;      // bytes of one A slice block per K step: TILE_A, or fewer rows (see gram_tc)
    int MT, NT, KS, ksplit;
    // the column tiles from NTr on are cross products (gram_tc): the first half of the reduction of A
    // against the second half of column tile nt - NTr, in ksplit / 2 ranges
    int NTr;
    int ncols;        // NT * TN
    double *part;     // [ksplit][MT * TM][ncols]: sum_d 2^-7d G_d of this block's K range
    int *err;         // set when a wait gave up
};

__device__ __forceinline__ void bulk_copy(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

// One lane of a converged warp, known to the compiler as such: operands of the MMA and copy
// instructions stay in uniform registers.
__device__ __forceinline__ bool elect_one() {
    uint32_t r;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(r));
    return r != 0;
}

// Barrier 1 over the GEMM_THREADS threads; returns the OR of v over them.
__device__ __forceinline__ bool drain_barrier_or(bool v) {
    uint32_t r;
    asm volatile("{\n .reg .pred pi, po;\n setp.ne.u32 pi, %1, 0;\n"
                 " barrier.cta.red.or.pred po, 1, %2, pi;\n selp.u32 %0, 1, 0, po;\n}\n"
                 : "=r"(r)
                 : "r"((uint32_t)v), "n"(GEMM_THREADS)
                 : "memory");
    return r != 0;
}

// One CTA per (64-column tile, 128-row tile, K range): the column tiles of one row tile
// are neighbours in the launch order, so that the CTAs streaming the same A blocks run at
// the same time and share them through L2.  One lane of PRODUCER_WARP streams the operand
// blocks of each K step into NSTAGE buffers (two bulk copies per step), one of MMA_WARP issues
// the MMAs; after every CS steps the sixteen warps drain the seven accumulators (warp w: lanes
// 32 (w % 4) .. + 31, columns DCOLS (w / 4) .. + DCOLS - 1) into exact 64-bit fixed point.
// With loads and MMAs issued by one thread in turn a step took 1550 clocks, of which 900 did not
// depend on the MMAs (896 at the tensor rate): 282 us for 24 modes on 24^3 sites, 228 with the roles
// split and five buffers instead of four (141 at the tensor rate; the operands' way from L2, 43 KB a step, is the next bound).
__global__ void __launch_bounds__(GEMM_BLOCK, 1) k_ozaki_gemm(GemmArgs a) {
    extern __shared__ __align__(128) uint8_t dsm[];
    __shared__ __align__(8) uint64_t full[NSTAGE], empty[NSTAGE];
    __shared__ uint32_t tbase;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int nt = blockIdx.x, mt = blockIdx.y, z = blockIdx.z;
    const bool cross = nt >= a.NTr;
    const int KS = cross ? a.KS / 2 : a.KS, nz = cross ? a.ksplit / 2 : a.ksplit;
    if (z >= nz) return;
    const int s0 = (int)((int64_t)KS * z / nz), s1 = (int)((int64_t)KS * (z + 1) / nz);
    const int ct = cross ? nt - a.NTr : nt;                                 // column tile
    const int64_t b0 = (a.Bq ? (int64_t)ct * a.KS : 0) + (cross ? KS : 0);  // first B block
    const int nsteps = s1 - s0;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tbase)),
                     "n"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int s = 0; s < NSTAGE; s++) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&full[s])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&empty[s])) : "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tbase;

    auto load = [&](int q) {  // producer: K step s0 + q into buffer q % NSTAGE (two bulk copies)
        const int st = q % NSTAGE;
        const uint32_t sa = smem_u32(dsm + st * STAGE), fb = smem_u32(&full[st]);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb),
                     "r"((uint32_t)(S * (a.a_bytes + TILE_B)))
                     : "memory");
        bulk_copy(sa, a.Aq + (((int64_t)mt * a.KS + s0 + q) * S) * a.a_bytes, S * a.a_bytes, fb);
        if (a.Bq) {
            bulk_copy(sa + S * a.a_bytes, a.Bq + ((b0 + s0 + q) * S) * TILE_B, S * TILE_B, fb);
        } else {  // 64 rows of each slice of A'
            const uint8_t *b = a.Aq + ((b0 + s0 + q) * S) * a.a_bytes + ct * TILE_B;
#pragma unroll
            for (int p = 0; p < S; p++) bulk_copy(sa + S * a.a_bytes + p * TILE_B, b + p * a.a_bytes, TILE_B, fb);
        }
    };
    {
        // 2^14 sum_{d<=2} 2^-7d G_d and 2^42 sum_{d>=3} 2^-7d G_d in two's complement (unsigned
        // arithmetic: exact for every accumulator row that holds a result, and defined
        // modulo 2^64 for the padding rows, whose values are discarded)
        uint64_t acc_hi[DCOLS], acc_lo[DCOLS];
#pragma unroll
        for (int c = 0; c < DCOLS; c++) acc_hi[c] = acc_lo[c] = 0;
        bool ok = true, aborted = false;
        int loaded = 0, issued = 0;  // steps the producer has loaded, steps whose MMAs were committed
        for (int j0 = 0; j0 < nsteps; j0 += CS) {
            const int je = min(j0 + CS, nsteps);
            if (warp == PRODUCER_WARP && elect_one()) {
                // the buffer of step q is free once the MMAs of step q - NSTAGE have read it: up to
                // NSTAGE steps of the next chunk are under way while this one's sums are drained
                for (; ok && loaded < min(je + NSTAGE, nsteps); loaded++) {
                    if (loaded >= NSTAGE) ok = mbar_wait(smem_u32(&empty[loaded % NSTAGE]), (loaded / NSTAGE - 1) & 1);
                    if (!ok) break;
                    load(loaded);
                }
            }
            if (warp == MMA_WARP && elect_one()) {
                for (int j = j0; j < je; j++) {
                    const int st = j % NSTAGE;
                    ok = mbar_wait(smem_u32(&full[st]), (j / NSTAGE) & 1);
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    // A slices a_bytes apart: with fewer than 128 rows stored, the MMA's
                    // remaining rows read whatever follows and only feed accumulator rows
                    // that are never drained into results
                    const uint32_t sa = smem_u32(dsm + st * STAGE), sb = sa + S * a.a_bytes;
                    const uint64_t da0 = mma_desc(sa), db0 = mma_desc(sb);
                    // The B slices of a stage lie one after another along N, so one MMA of
                    // A slice p against B slices q0 .. q0 + nq - 1 (N = 64 nq <= 256) writes the
                    // adjacent accumulators of the groups p + q0 .. p + q0 + nq - 1.
#pragma unroll
                    for (int p = 0; p < S; p++) {
#pragma unroll
                        for (int q0 = 0; q0 < S - p; q0 += 4) {
                            const int nq = (S - p - q0) < 4 ? (S - p - q0) : 4;
                            const uint32_t dcol = tmem + (uint32_t)((p + q0) * TN);
                            const uint64_t da = da0 + (uint64_t)((p * a.a_bytes) >> 4);
                            const uint64_t db = db0 + (uint64_t)((q0 * TILE_B) >> 4);
                            // the first products of a chunk (p = 0 covers every group) overwrite
                            const uint32_t accum = (j == j0 && p == 0) ? 0u : 1u;
                            asm volatile("{\n .reg .pred pa;\n setp.ne.b32 pa, %4, 0;\n"
                                         " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, pa;\n}\n"
                                         ::"r"(dcol), "l"(da), "l"(db), "r"(idesc_n(TN * nq)), "r"(accum)
                                         : "memory");
                        }
                    }
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                                 ::"r"(smem_u32(&empty[st]))
                                 : "memory");
                    issued = j + 1;
                }
            }
            if (!ok) atomicExch(a.err, 1);
            __syncwarp();
            loaded = __reduce_max_sync(0xffffffffu, loaded);
            issued = __reduce_max_sync(0xffffffffu, issued);
            {
                const int j = je - 1, st = j % NSTAGE;
                // every draining thread takes the same branch: the barrier returns the OR
                if (drain_barrier_or(!ok)) {
                    aborted = true;
                    break;
                }
                const bool done = mbar_wait(smem_u32(&empty[st]), (j / NSTAGE) & 1);
                if (!done) atomicExch(a.err, 1);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                if (done) {
                    const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;
                    const int cbase = DCOLS * (warp >> 2);
#pragma unroll
                    for (int d = 0; d < S; d++) {
                        uint32_t r[DCOLS];
                        const uint32_t taddr = tmem + lane_base + (uint32_t)(d * TN + cbase);
                        asm volatile(
                            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
                            "%15}, [%16];"
                            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                              "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
                              "=r"(r[14]), "=r"(r[15])
                            : "r"(taddr)
                            : "memory");
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                        // G_d is an integer below 2^24: the conversion is exact
                        const int sh = d <= 2 ? 14 - 7 * d : 42 - 7 * d;
#pragma unroll
                        for (int c = 0; c < DCOLS; c++) {
                            const uint64_t v = (uint64_t)(int64_t)__float2int_rn(__uint_as_float(r[c])) << sh;
                            if (d <= 2)
                                acc_hi[c] += v;
                            else
                                acc_lo[c] += v;
                        }
                    }
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                if (drain_barrier_or(!done)) {
                    aborted = true;
                    break;
                }
            }
        }
        // after a failed wait: give the copies and MMAs in flight a bounded time to land
        if (issued > 0) mbar_wait(smem_u32(&empty[(issued - 1) % NSTAGE]), ((issued - 1) / NSTAGE) & 1);
        for (int q = max(0, loaded - NSTAGE); q < loaded; q++) mbar_wait(smem_u32(&full[q % NSTAGE]), (q / NSTAGE) & 1);
        __syncwarp();
        if (!aborted) {
            const int row = mt * TM + 32 * (warp & 3) + lane;
            double *o = a.part + ((int64_t)z * a.MT * TM + row) * a.ncols + nt * TN + DCOLS * (warp >> 2);
#pragma unroll
            for (int c = 0; c < DCOLS; c++)
                o[c] = ldexp((double)(int64_t)acc_hi[c], -14) + ldexp((double)(int64_t)acc_lo[c], -42);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(TMEM_COLS) : "memory");
}

// Number of K ranges per output tile.  The product runs one CTA per SM: up to one wave,
// as many ranges as fill it; where that leaves the last wave poorly filled (few tiles
// per wave, or a ragged tail), more ranges of at least 8 chunks each are taken if they
// fill the waves better by more than 5%.  Every range stays below MAX_STEPS_PER_BLOCK.
int pick_ksplit(int tiles, int KS) {
    constexpr int NSM = 152;
    auto fill = [&](int k) {
        const int64_t ctas = (int64_t)tiles * k;
        return (double)ctas / (double)(((ctas + NSM - 1) / NSM) * NSM);
    };
    int best = std::max(1, std::min(KS, NSM / tiles));
    for (int k = best + 1; k <= 256 && k <= KS / (8 * CS); k++)
        if (fill(k) > fill(best) + 0.05) best = k;
    return std::max(best, (KS + MAX_STEPS_PER_BLOCK - 1) / MAX_STEPS_PER_BLOCK);
}

// The sums over the K ranges of a product's elements, in a fixed order.  A block of FIN_THREADS has
// FIN_THREADS / G elements; thread u E + e adds the ranges u, u + G, ... of element e, and thread e
// the G sums.  One thread adding up to 152 ranges waited for every load: Gram block of 8 columns on
// 8^3 sites 43 us, 12 with G = 8; 8 columns of colourless spinors on 4^3 sites 10 and 6.  Few ranges
// come with many elements, which fill the chip with G = 1.
constexpr int FIN_THREADS = 256;
int fin_groups(int ksplit) { return ksplit >= 16 ? 8 : 1; }
struct RangeSums {
    int E, e, u;
    __device__ explicit RangeSums(int G) : E(FIN_THREADS / G), e(threadIdx.x % E), u(threadIdx.x / E) {}
    __device__ int64_t element() const { return blockIdx.x * (int64_t)E + e; }
    // v[k] = sum of n[k] values at p[k], step apart; to be used by the threads with u = 0
    template <int NV>
    __device__ void sums(bool valid, const double *const p[NV], const int n[NV], int64_t step, double v[NV]) const {
        __shared__ double sh[NV][FIN_THREADS];
        const int G = FIN_THREADS / E;
#pragma unroll
        for (int k = 0; k < NV; k++) {
            v[k] = 0;
            if (valid)
                for (int s = u; s < n[k]; s += G) v[k] += __ldg(p[k] + s * step);
            sh[k][threadIdx.x] = v[k];
        }
        __syncthreads();
        if (u == 0)
            for (int g = 1; g < G; g++)
#pragma unroll
                for (int k = 0; k < NV; k++) v[k] += sh[k][g * E + e];
    }
};

// X[i][j][k][alpha] = X[j][i][k][alpha] = 2^(e_row + e_col - 14) sum over the K-range
// partials.
__global__ void __launch_bounds__(FIN_THREADS) k_ozaki_finish(const double *part, int ksplit, int G, int prow, int ncols, int m,
                                                              int rows, const double *rowmax, const double *colmax, double2 *X) {
    const RangeSums rs(G);
    const int64_t g = rs.element();
    const int Q = 4 * m;
    const int r = (int)(g / Q), q = (int)(g % Q);
    const double *row = part + (int64_t)r * ncols, *const p[2] = {row + q, row + Q + q};
    const int n[2] = {ksplit, ksplit};
    double v2[2];
    rs.sums<2>(r < rows, p, n, (int64_t)prow * ncols, v2);
    if (r >= rows || rs.u) return;
    // the splits carried v = 2^(e - 49) N = 2^(e - 7) sum_p q_p 2^(-7p) for each operand
    int i, j;
    pair_of(r, m, i, j);
    const int sc = exponent_of(rowmax[r]) + column_exponent(colmax, i) + column_exponent(colmax, j) +
                   exponent_of(colmax[q]) - 14;
    double2 v = make_double2(ldexp(v2[0], sc), ldexp(v2[1], sc));
    if (!isfinite(rowmax[r]) || !isfinite(colmax[q])) v = make_double2(NAN, NAN);  // a non-finite input
    X[((int64_t)i * m + j) * Q + q] = v;
    if (i != j) X[((int64_t)j * m + i) * Q + q] = v;
}

}  // namespace

namespace ddp {

// Colourless-spinor slice sums of a domain on the tensor cores (fields and forms as
// ddp_colourless_slices).  A: [m][n][12] on the device; X: L0 x m^3 x 4 complex on the
// device, slices outside the domain left untouched.
int colourless_tc(ddp_ctx *ctx, const double2 *A, int64_t n, int m, int form, int64_t slice_n, int nslice, int o0,
                  int L0, double2 *X) {
    if (m < 1 || m > MMAX) return DDP_ERR_UNSUPPORTED;
    const int rows = m * (m + 1) / 2, Q = 4 * m;
    const int MT = (rows + TM - 1) / TM;
    const int NT = (2 * Q + TN - 1) / TN;
    const int64_t K = 3 * slice_n;
    const int64_t KSh64 = (K + KSTEP - 1) / KSTEP;
    if (KSh64 > (1 << 28)) return DDP_ERR_UNSUPPORTED;
    const int KSh = (int)KSh64, KS = 2 * KSh;
    const int ksplit = pick_ksplit(MT * NT, KS);
    const int ncols = NT * TN, prow = MT * TM;
    const size_t bE = (size_t)rows * K * sizeof(float4);
    const size_t bA = (size_t)S * MT * KS * TILE_A, bB = (size_t)S * NT * KS * TILE_B;
    const size_t bP = (size_t)ksplit * prow * ncols * sizeof(double);
    Arena &ar = ctx->aux;
    ar.reset();
    DDP_CUDA(ctx, ar.reserve(bE + bA + bB + bP + (size_t)(rows + Q) * 12 + 64 + 10 * 256));
    float4 *E = (float4 *)ar.take(bE);
    uint8_t *Aq = (uint8_t *)ar.take(bA);
    uint8_t *Bq = (uint8_t *)ar.take(bB);
    double *part = (double *)ar.take(bP);
    // rows, then spinor columns
    double *rowmax = (double *)ar.take((size_t)(rows + Q) * 8), *colmax = rowmax + rows;
    int *rexp = (int *)ar.take((size_t)(rows + Q) * 4), *cexp = rexp + rows;
    int *err = (int *)ar.take(64);
    const int es = m <= ES_SMALL_MMAX ? ES_SMALL : ES_LARGE;
    const size_t esm = (size_t)m * colour_kstride(es) * sizeof(float4);
    const size_t gsm = (size_t)NSTAGE * STAGE;
    DDP_CUDA(ctx, cudaFuncSetAttribute(es == ES_SMALL ? k_colour_E<ES_SMALL> : k_colour_E<ES_LARGE>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)esm));
    DDP_CUDA(ctx, cudaFuncSetAttribute(k_ozaki_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gsm));
    cudaStream_t st = ctx->stream;
    DDP_CUDA(ctx, cudaMemsetAsync(err, 0, sizeof(int), st));
    for (int z = 0; z < nslice; z++) {
        const int64_t site0 = (int64_t)z * slice_n;
        DDP_CUDA(ctx, cudaMemsetAsync(rowmax, 0, (size_t)(rows + Q) * 8, st));
        EArgs ea;
        ea.A = A;
        ea.n = n;
        ea.site0 = site0;
        ea.slice_n = slice_n;
        ea.m = m;
        ea.form = form;
        ea.rows = rows;
        ea.E = E;
        ea.rowmax = rowmax;
        ea.colmax = colmax;
        k_colour_max<<<(unsigned)std::min<int64_t>(2 * 152, (slice_n + 1) / 2), 256, 0, st>>>(A, n, site0, slice_n,
                                                                                          m, colmax);
        if (es == ES_SMALL)
            k_colour_E<ES_SMALL><<<(unsigned)((slice_n + ES_SMALL - 1) / ES_SMALL), 256, esm, st>>>(ea);
        else
            k_colour_E<ES_LARGE><<<(unsigned)((slice_n + ES_LARGE - 1) / ES_LARGE), 256, esm, st>>>(ea);
        SplitArgs sa;
        sa.E = E;
        sa.A = A;
        sa.n = n;
        sa.site0 = site0;
        sa.K = K;
        sa.m = m;
        sa.form = form;
        sa.rows = rows;
        sa.MT = MT;
        sa.NT = NT;
        sa.KSh = KSh;
        k_exponents<<<(rows + Q + 255) / 256, 256, 0, st>>>(rowmax, rows + Q, rexp);
        sa.rexp = rexp;
        sa.cexp = cexp;
        sa.Aq = Aq;
        sa.Bq = Bq;
        const int64_t na = 2 * (int64_t)KSh * MT * TM, nb = 2 * (int64_t)KSh * (NT * TN - Q);
        k_split_A<<<(unsigned)((na + 255) / 256), 256, 0, st>>>(sa);
        k_split_B<<<(unsigned)((nb + 255) / 256), 256, 0, st>>>(sa);
        GemmArgs g;
        g.Aq = Aq;
        g.Bq = Bq;
        g.a_bytes = TILE_A;
        g.MT = MT;
        g.NT = g.NTr = NT;
        g.KS = KS;
        g.ksplit = ksplit;
        g.ncols = ncols;
        g.part = part;
        g.err = err;
        k_ozaki_gemm<<<dim3(NT, MT, ksplit), GEMM_BLOCK, gsm, st>>>(g);
        const int64_t nx = (int64_t)rows * Q;
        const int G = fin_groups(ksplit), per = FIN_THREADS / G;
        k_ozaki_finish<<<(unsigned)((nx + per - 1) / per), FIN_THREADS, 0, st>>>(
            part, ksplit, G, prow, ncols, m, rows, rowmax, colmax, X + (int64_t)((o0 + z) % L0) * m * m * Q);
        ctx->launches += 7;
        DDP_CUDA(ctx, cudaGetLastError());
    }
    int h = 0;
    DDP_CUDA(ctx, cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, st));
    DDP_CUDA(ctx, cudaStreamSynchronize(st));
    if (h) {
        snprintf(ctx->last_error, sizeof(ctx->last_error), "colourless spinors: a wait for the tensor cores gave up");
        return DDP_ERR_CUDA;
    }
    return DDP_OK;
}

}  // namespace ddp

// ------------------------------------------------------------ Gram blocks
//
// G[i][j] = sum_r conj(A_i[r]) A_j[r] over the rows r of one segment, on the same
// emulated-FP64 product, every column with its own power-of-two exponent.  With R_i and I_i the
// real and imaginary parts of column i, the reduction of A' = [R | I] runs over two halves:
//   m > 32: the real parts are A' against the columns B' = [R | I]; the imaginary parts are
//     X_ij - X_ji with X = sum R_i I_j, which is the first half of A' against the second half of B'
//     (cross tiles): three quarters of the products.  B' holds the same slices as A', so only A' is
//     stored, and a column tile is read as 64 rows of each of its slices (rows beyond R8 are those of
//     the next slice and feed columns that are never used).
//   m <= 32: real and imaginary parts share one 64-column tile, B' rows [R | I] for j < m and
//     [I | -R] beyond.
// The m <= 128 rows of A' are stored as R8 = 8 ceil(m / 8) rows per block (the MMA's other rows
// read whatever follows in shared memory and feed accumulator rows that are never used).
//
// The slices are cut in one pass that reads the columns once and writes 16 bytes per store.  Per
// time slice of 24^3 sites and 120 columns: maxima 178 -> 61 us (compared as integers: FP64
// comparisons run on the FP64 pipe), slices 650 -> 224 (were two passes with 2-byte stores and both
// operands; the bytes take 130 at the copy rate), product 456 -> 282 (188 at the tensor pipe's rate).

namespace {

// top[i] = the largest high word, without its sign, of the components of column i over the
// segment's rows; at least 1 if a component is not zero
__global__ void __launch_bounds__(256) k_gram_max(const double2 *A, int64_t cs, int64_t r0, int64_t nrow, unsigned *top) {
    const double2 *a = A + (int64_t)blockIdx.y * cs + r0;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    unsigned mx = 0, low = 0;
    int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    auto take = [&](const double2 &v) {
        mx = max(mx, max((unsigned)__double2hiint(v.x) & 0x7FFFFFFFu, (unsigned)__double2hiint(v.y) & 0x7FFFFFFFu));
        low |= (unsigned)(__double2loint(v.x) | __double2loint(v.y));
    };
    for (; r + 3 * step < nrow; r += 4 * step) {
        const double2 v0 = __ldg(a + r), v1 = __ldg(a + r + step), v2 = __ldg(a + r + 2 * step), v3 = __ldg(a + r + 3 * step);
        take(v0);
        take(v1);
        take(v2);
        take(v3);
    }
    for (; r < nrow; r += step) take(__ldg(a + r));
    mx = max(mx, (unsigned)(low != 0));  // subnormals below 2^-1042 have no bit in their high word
    mx = __reduce_max_sync(0xffffffffu, mx);
    if ((threadIdx.x & 31) == 0) atomicMax(top + blockIdx.y, mx);
}

// e with |v| < 2^e for every component of the column (0 for a column of zeros), NONFINITE if one is
// not finite.  A column of subnormals, t its largest high word: |v| < (t + 1) 2^32 2^-1074.
__global__ void k_gram_exponents(const unsigned *top, int n, int *ex) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int e = (int)(top[i] >> 20);
    ex[i] = e == 0x7FF ? NONFINITE : e ? e - 1022 : top[i] ? 32 - __clz(top[i]) - 1042 : 0;
}

struct GramSplitArgs {
    const double2 *A;
    int64_t cs, r0, nrow;  // column stride; the segment's rows
    int m, R8, KSh;
    int mixed;             // real and imaginary columns in one tile (m <= 32)
    const int *cexp;       // exponents of the columns
    uint8_t *Aq, *Bq;      // [2 KSh][S][R8 x KSTEP]; mixed: [2 KSh][S][64 x KSTEP]; BF16
};

// Thread per (column, 8 reduction steps): a 16-byte row of a core matrix of every slice.
// Consecutive threads take consecutive columns, so that 8 of them write one core matrix.
__global__ void __launch_bounds__(256) k_gram_split(GramSplitArgs a) {
    const int RB = a.mixed ? TN : a.R8;
    const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (g >= 2 * (int64_t)a.KSh * RB) return;
    const int row = (int)(g % RB);
    const int64_t t = g / RB;
    const int k8 = (int)(t & 1);
    const int64_t ksr = t >> 1, kx = ksr * KSTEP + 8 * k8;
    if (a.mixed && row >= a.m && row < 2 * a.m) return;  // written by the thread of column row - m
    uint4 re[S], im[S];
    const int er = row < a.m ? a.cexp[row] : NONFINITE;
#pragma unroll
    for (int p = 0; p < S; p++) re[p] = im[p] = make_uint4(0, 0, 0, 0);
    if (er != NONFINITE) {
        const double2 *src = a.A + (int64_t)row * a.cs + a.r0 + kx;
        const int k = 49 - er;
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const double2 z = make_double2(0.0, 0.0);
            const double2 v0 = kx + 2 * j < a.nrow ? __ldg(src + 2 * j) : z, v1 = kx + 2 * j + 1 < a.nrow ? __ldg(src + 2 * j + 1) : z;
            put_digits(re, j, fixed_of(v0.x, k), fixed_of(v1.x, k));
            put_digits(im, j, fixed_of(v0.y, k), fixed_of(v1.y, k));
        }
    }
    const int64_t sre = ksr * S, sim = (a.KSh + ksr) * S;  // first slice of the K steps of either half
    if (row < a.R8) {
        const int tile = a.R8 * KSTEP * 2;
        put_slices(a.Aq + sre * tile + tile_offset(row, k8), tile, re);
        put_slices(a.Aq + sim * tile + tile_offset(row, k8), tile, im);
    }
    if (!a.mixed) return;
    uint8_t *bre = a.Bq + sre * TILE_B, *bim = a.Bq + sim * TILE_B;
    put_slices(bre + tile_offset(row, k8), TILE_B, re);
    put_slices(bim + tile_offset(row, k8), TILE_B, im);
    if (row < a.m) {  // column m + row: [I | -R]
        put_slices(bre + tile_offset(row + a.m, k8), TILE_B, im);
        put_slices(bim + tile_offset(row + a.m, k8), TILE_B, re, true);
    }
}

// G[i][j] = 2^(e_i + e_j - 14) (sum of the K-range partials); cross > 0: the first of the cross
// products' columns, X_ij - X_ji the imaginary part, in ksplit / 2 ranges.
__global__ void __launch_bounds__(FIN_THREADS) k_gram_finish(const double *part, int ksplit, int G, int ncols, int m, int cross,
                                                             const int *cexp, double2 *out) {
    const RangeSums rs(G);
    const int g = (int)rs.element();
    const bool valid = g < m * m;
    const int i = g / m, j = g % m;
    const double *ri = part + (int64_t)i * ncols, *rj = part + (int64_t)j * ncols;
    const double *const p[3] = {ri + j, ri + (cross ? cross : m) + j, rj + cross + i};
    const int n[3] = {ksplit, cross ? ksplit / 2 : ksplit, cross ? ksplit / 2 : 0};
    double s[3];
    rs.sums<3>(valid, p, n, (int64_t)TM * ncols, s);
    if (!valid || rs.u) return;
    const int sc = cexp[i] + cexp[j] - 14;
    double2 v = make_double2(NAN, NAN);
    if (cexp[i] != NONFINITE && cexp[j] != NONFINITE) v = make_double2(ldexp(s[0], sc), ldexp(s[1] - s[2], sc));
    out[g] = v;
}

}  // namespace

namespace ddp {

// Gram blocks of nseg consecutive row segments of seg rows each on the tensor cores:
// out[z][i][j] = sum over the rows r of segment z of conj(A_i[r]) A_j[r], A_i[r] the
// complex component r of column i (column stride cs); A and out on the device, m <= 128.
int gram_tc(ddp_ctx *ctx, const double2 *A, int64_t cs, int m, int64_t seg, int nseg, double2 *out) {
    if (m < 1 || m > TM) return DDP_ERR_UNSUPPORTED;
    const int R8 = 8 * ((m + 7) / 8);
    const int a_bytes = R8 * KSTEP * 2;
    const bool mixed = 2 * m <= TN;
    const int NTr = (m + TN - 1) / TN;  // column tiles of B' (mixed: the one that holds both parts)
    const int NT = mixed ? 1 : 2 * NTr, ncols = NT * TN;
    const int64_t KSh64 = (seg + KSTEP - 1) / KSTEP;
    if (KSh64 > (1 << 28)) return DDP_ERR_UNSUPPORTED;
    const int KSh = (int)KSh64, KS = 2 * KSh;
    // one wave of CTAs: the cross tiles take half the ranges for half the reduction
    const int ksplit = mixed ? pick_ksplit(1, KS)
                             : std::max({2, std::min(2 * (152 / (3 * NTr)), 2 * KSh),
                                         2 * ((KS + 2 * MAX_STEPS_PER_BLOCK - 1) / (2 * MAX_STEPS_PER_BLOCK))});
    // the last column tile of the last slice may read up to a full tile of 128 rows
    const size_t bA = (size_t)S * KS * a_bytes + TILE_A, bB = mixed ? (size_t)S * KS * TILE_B : 0;
    const size_t bP = (size_t)ksplit * TM * ncols * sizeof(double);
    Arena &ar = ctx->aux;
    ar.reset();
    DDP_CUDA(ctx, ar.reserve(bA + bB + bP + (size_t)m * 8 + 64 + 7 * 256));
    uint8_t *Aq = (uint8_t *)ar.take(bA);
    uint8_t *Bq = mixed ? (uint8_t *)ar.take(bB) : nullptr;
    double *part = (double *)ar.take(bP);
    unsigned *top = (unsigned *)ar.take((size_t)m * 4);
    int *cexp = (int *)ar.take((size_t)m * 4);
    int *err = (int *)ar.take(64);
    const size_t gsm = (size_t)NSTAGE * STAGE;
    DDP_CUDA(ctx, cudaFuncSetAttribute(k_ozaki_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gsm));
    cudaStream_t st = ctx->stream;
    DDP_CUDA(ctx, cudaMemsetAsync(err, 0, sizeof(int), st));
    for (int z = 0; z < nseg; z++) {
        DDP_CUDA(ctx, cudaMemsetAsync(top, 0, (size_t)m * 4, st));
        const int64_t r0 = (int64_t)z * seg;
        // about 8 blocks per SM over all columns
        const unsigned nb = (unsigned)std::max<int64_t>(1, std::min<int64_t>((8 * 152 + m - 1) / m, (seg + 1023) / 1024));
        k_gram_max<<<dim3(nb, m), 256, 0, st>>>(A, cs, r0, seg, top);
        k_gram_exponents<<<1, TM, 0, st>>>(top, m, cexp);
        GramSplitArgs sa;
        sa.A = A;
        sa.cs = cs;
        sa.r0 = r0;
        sa.nrow = seg;
        sa.m = m;
        sa.R8 = R8;
        sa.KSh = KSh;
        sa.mixed = mixed ? 1 : 0;
        sa.cexp = cexp;
        sa.Aq = Aq;
        sa.Bq = Bq;
        const int64_t ns = 2 * (int64_t)KSh * (mixed ? TN : R8);
        k_gram_split<<<(unsigned)((ns + 255) / 256), 256, 0, st>>>(sa);
        GemmArgs g;
        g.Aq = Aq;
        g.Bq = Bq;
        g.a_bytes = a_bytes;
        g.MT = 1;
        g.NT = NT;
        g.NTr = mixed ? NT : NTr;
        g.KS = KS;
        g.ksplit = ksplit;
        g.ncols = ncols;
        g.part = part;
        g.err = err;
        k_ozaki_gemm<<<dim3(NT, 1, ksplit), GEMM_BLOCK, gsm, st>>>(g);
        const int G = fin_groups(ksplit), per = FIN_THREADS / G;
        k_gram_finish<<<(unsigned)((m * m + per - 1) / per), FIN_THREADS, 0, st>>>(part, ksplit, G, ncols, m, mixed ? 0 : NTr * TN,
                                                                               cexp, out + (int64_t)z * m * m);
        ctx->launches += 5;
        DDP_CUDA(ctx, cudaGetLastError());
    }
    int h = 0;
    DDP_CUDA(ctx, cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, st));
    DDP_CUDA(ctx, cudaStreamSynchronize(st));
    if (h) {
        snprintf(ctx->last_error, sizeof(ctx->last_error), "Gram blocks: a wait for the tensor cores gave up");
        return DDP_ERR_CUDA;
    }
    return DDP_OK;
}

}  // namespace ddp
