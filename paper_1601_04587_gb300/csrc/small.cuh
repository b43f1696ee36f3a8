// One correction cycle of a small domain in one kernel (16- and 32-bit storage formats, no clover
// term): right-hand side, the whole BiCGStab loop and the FP64 accumulation.
//
// A domain of at most SMALL_MAX_NH sites per parity has too little work for a launch per step: an
// iteration of eight kernels on an 8^4 block took 45 us, nearly all of it the latency of each
// kernel's start, its item, its staged links and its reductions.  Here two columns of a request
// belong to one thread-block cluster.  Each block owns up to 128 sites of either parity and holds
// on chip, for the length of the solve, the oriented links and neighbours of its sites (shared by
// the two columns), the three vectors that neighbours read (p, s = r and the odd intermediate) in
// shared memory, and the vectors only the owner needs (x, v, t, rh) in registers, one site-column
// per thread.  A block owns a sub-box of the domain, so that most neighbours are its own; the
// others are read through distributed shared memory.  An iteration has six cluster barriers, two
// of them with a reduction, whose sums every block finishes for itself in the same order, so that
// all take the same decisions.
//
// Arithmetic is FP32 on FP32 vectors for every storage format (links as stored); sums over sites
// are FP32 within a warp, three floats beyond, scalars FP64, as in the per-step kernels (recur.cuh).
//
// What bounds it is latency: a block's 8 warps spend about 5000 cycles on an application of the
// hopping term (2700 of them shared-memory wavefronts), 1000 on a barrier.  Propagators of 12
// columns, FP32, per-step kernels / this kernel: one alone 4^4 1.21 / 0.56 ms, 8x4^3 1.33 / 0.62,
// 8x8x4x4 1.34 / 0.67, 8^3x4 1.55 / 0.77; 64 in a batch 2.94 / 2.37, 4.66 / 3.84, 7.47 / 6.67, 13.9 /
// 15.9 (8 of 8^3x4 2.60 / 2.60).  The largest domains gain alone and lose in large batches of their
// like: eight blocks of one SM each wait for their slowest.  With 16 blocks a cluster an 8^4 block
// alone went 2.79 -> 1.20, 64 of them 37.4 -> 54.0, so the path ends at 8 blocks.  Two threads per
// site-column (one spin of the projection each) and one row of links rebuilt from the other two
// were slower.
//
// A request takes this path by its own size alone, so its result does not depend on what else is
// solved with it.
#pragma once

#include "ddp_kernels.cuh"

namespace ddp {

constexpr int SMALL_SITES = 128;     // sites per parity and block
constexpr int SMALL_COLS = 2;        // columns per cluster
constexpr int SMALL_THREADS = SMALL_SITES * SMALL_COLS;
constexpr int SMALL_MAX_CLUSTER = 8;
constexpr int SMALL_MAX_NH = SMALL_SITES * SMALL_MAX_CLUSTER;

struct SmallArgs {
    const Item *items;   // the items of this launch, sorted by sblk0 (clusters, in units of one)
    int nitems;
    int csize;           // blocks per cluster
    FieldView re, ro;    // FP64 defect (even, odd)
    FieldView xe, xo;    // FP64 solution, accumulated
    SolveState *st;
};

// Shared memory of a block.
struct SmallShared {
    float2 link[2][8][SMALL_SITES][9];                // the hop's oriented link, per output parity
    float4 vec[3][SMALL_COLS][6][SMALL_SITES];        // p, s (and r), odd intermediate
    short nb[2][8][SMALL_SITES];                      // -1, or block << 7 | site, | SMALL_NEG
    float4 slot[2][SMALL_MAX_CLUSTER][SMALL_COLS * PART_MAX];  // partial sums of every block, double-buffered
    float warp[SMALL_THREADS / 32][PART_MAX];
    float2 alpha[SMALL_COLS], omega[SMALL_COLS], beta[SMALL_COLS];
    int go[SMALL_COLS];                               // the column goes on iterating
    int upd[SMALL_COLS];                              // its x, r, p are updated in this iteration
    Item it;
};
static_assert(SMALL_SITES == 128 && SMALL_MAX_CLUSTER <= 16, "neighbour codes: 4 bits of block, 7 of site");
static_assert(sizeof(SmallShared) <= 227 * 1024, "one block's shared memory");
constexpr int SMALL_NEG = 1 << 12;   // the hop changes sign (antiperiodic boundary)
enum { SV_P = 0, SV_S = 1, SV_T = 2 };

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync(int csize) {
    if (csize == 1) {
        __syncthreads();
    } else {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}
// The shared-memory address of block `rank` that corresponds to this block's address a.
__device__ __forceinline__ unsigned cluster_addr(unsigned a, unsigned rank) {
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}

// Site values of a vector in shared memory.
__device__ __forceinline__ void small_put(SmallShared &sh, int vec, int col, int l, const float2 v[12]) {
#pragma unroll
    for (int j = 0; j < 6; j++) sh.vec[vec][col][j][l] = make_float4(v[2 * j].x, v[2 * j].y, v[2 * j + 1].x, v[2 * j + 1].y);
}
__device__ __forceinline__ void small_get(const SmallShared &sh, int vec, int col, int l, float2 v[12]) {
#pragma unroll
    for (int j = 0; j < 6; j++) {
        const float4 c = sh.vec[vec][col][j][l];
        v[2 * j] = f2(c.x, c.y);
        v[2 * j + 1] = f2(c.z, c.w);
    }
}

// One neighbour: its code (< 0: none) and values.
__device__ __forceinline__ int small_fetch(const SmallShared &sh, int par, int d, unsigned base, int l, float2 v[12]) {
    const int nb = sh.nb[par][d][l];
    if (nb < 0) return nb;
    // own sites are read the same way: a branch for them splits the warps on a sub-box's faces (3%)
    const unsigned a = cluster_addr(base + (unsigned)(nb & 127) * 16u, (unsigned)(nb >> 7) & 15u);
#pragma unroll
    for (int j = 0; j < 6; j++)
        asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(v[2 * j].x), "=f"(v[2 * j].y), "=f"(v[2 * j + 1].x), "=f"(v[2 * j + 1].y)
                     : "r"(a + (unsigned)(j * SMALL_SITES * 16)));
    return nb;
}

// The hopping sum at the thread's site of parity par from vector vec of its column.
__device__ __forceinline__ void small_hops(const SmallShared &sh, int par, int vec, int col, int l, float2 acc[12]) {
    const unsigned base = (unsigned)__cvta_generic_to_shared(&sh.vec[vec][col][0][0]);
    float2 s[4][3];
#pragma unroll
    for (int j = 0; j < 12; j++) s[j / 3][j % 3] = f2(0.f, 0.f);
#define DDP_SMALL_HOP(D)                                                                            \
    {                                                                                               \
        float2 v[12];                                                                               \
        const int nb = small_fetch(sh, par, D, base, l, v);                                   \
        if (nb >= 0) f2_hop_step<D, true>(v, sh.link[par][D][l], s, (nb & SMALL_NEG) ? -1.f : 1.f); \
    }
    DDP_SMALL_HOP(0)
    DDP_SMALL_HOP(1)
    DDP_SMALL_HOP(2)
    DDP_SMALL_HOP(3)
    DDP_SMALL_HOP(4)
    DDP_SMALL_HOP(5)
    DDP_SMALL_HOP(6)
    DDP_SMALL_HOP(7)
#undef DDP_SMALL_HOP
#pragma unroll
    for (int j = 0; j < 12; j++) acc[j] = s[j / 3][j % 3];
}

__device__ __forceinline__ float2 f2_cmul(float2 a, float2 b) {  // a b
    return f2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ void f2_dot(float &re, float &im, float2 a, float2 b) {  // += conj(a) b
    re = fmaf(a.x, b.x, fmaf(a.y, b.y, re));
    im = fmaf(a.x, b.y, fmaf(-a.y, b.x, im));
}

// Sums of NV values over a column's sites, over all blocks of the cluster: on return lane c * NV + k
// of warp 0 of every block holds value k of column c.  buf alternates between calls.
template <int NV>
__device__ __forceinline__ double small_sums(SmallShared &sh, float v[NV], int csize, unsigned rank, int buf) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int off = 16;
#pragma unroll
    for (int n = NV; n > 1; n >>= 1, off >>= 1) {
        const bool up = lane & off;
#pragma unroll
        for (int i = 0; i < n / 2; i++) {
            const float keep = up ? v[i + n / 2] : v[i], send = up ? v[i] : v[i + n / 2];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
#pragma unroll
    for (; off > 0; off >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
    if ((lane & (32 / NV - 1)) == 0) sh.warp[warp][lane / (32 / NV)] = v[0];
    __syncthreads();
    constexpr int NT = SMALL_COLS * NV;
    // lanes t, t + NT, ... of the first warps: value t to blocks 0, 1, ... (each forms it for itself)
    for (int q = threadIdx.x; q < NT * csize; q += SMALL_THREADS) {
        const int t = q % NT, r = q / NT, c = t / NV, k = t % NV;
        const float *w = &sh.warp[c * (SMALL_SITES / 32)][k];
        Sum3 s = {w[0], 0.f, 0.f};
#pragma unroll
        for (int n = 1; n < SMALL_SITES / 32; n++) sum_add(s, w[n * PART_MAX]);
        const unsigned a = cluster_addr((unsigned)__cvta_generic_to_shared(&sh.slot[buf][rank][t]), (unsigned)r);
        asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %3};" ::"r"(a), "f"(s.hi), "f"(s.mid), "f"(s.lo) : "memory");
    }
    cluster_sync(csize);
    if (warp != 0) return 0.0;
    {
        // two lanes per value: even and odd blocks, each as a tree
        const int t = lane & 15, odd = lane >> 4;
        Sum3 d[SMALL_MAX_CLUSTER / 2];
#pragma unroll
        for (int r = 0; r < SMALL_MAX_CLUSTER / 2; r++) {
            sum_zero(d[r]);
            if (t < NT && 2 * r + odd < csize) {
                const float4 f = sh.slot[buf][2 * r + odd][t];
                d[r] = {f.x, f.y, f.z};
            }
        }
#pragma unroll
        for (int n = SMALL_MAX_CLUSTER / 4; n > 0; n >>= 1)
            if (csize > 2 * n)
#pragma unroll
                for (int r = 0; r < n; r++) d[r] = sum_join(d[r], d[r + n]);
        return sum_value(sum_join(d[0], sum_shfl_xor(d[0], 16)));
    }
}

template <class P>
__global__ void __launch_bounds__(SMALL_THREADS, 1) k_small(const __grid_constant__ SmallArgs a) {
    extern __shared__ __align__(16) unsigned char small_raw[];
    SmallShared &sh = *reinterpret_cast<SmallShared *>(small_raw);
    const int csize = a.csize;
    const unsigned rank = csize == 1 ? 0u : cluster_rank();
    const int cl = blockIdx.x / csize;  // cluster of this launch
    if (threadIdx.x < 32) {
        int lo = 0, hi = a.nitems - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (a.items[mid].sblk0 <= cl)
                lo = mid;
            else
                hi = mid - 1;
        }
        const int4 *src = reinterpret_cast<const int4 *>(a.items + lo);
        if (threadIdx.x < sizeof(Item) / 16) reinterpret_cast<int4 *>(&sh.it)[threadIdx.x] = __ldg(src + threadIdx.x);
    }
    __syncthreads();
    const Item &it = sh.it;
    const int col0 = (cl - it.sblk0) * SMALL_COLS;
    // columns with nothing to correct (the same answer in every block of the cluster)
    bool any = false;
    for (int c = 0; c < SMALL_COLS; c++) any = any || (col0 + c < it.ncol && a.st[it.solve0 + col0 + c].sigma > 0);
    if (!any) return;
    // the block's sub-box
    const int bz = (int)rank / (it.sc[0] * it.sc[1] * it.sc[2]) * it.sb[3];
    const int b0 = (int)rank % it.sc[0] * it.sb[0], b1 = (int)rank / it.sc[0] % it.sc[1] * it.sb[1],
              b2 = (int)rank / (it.sc[0] * it.sc[1]) % it.sc[2] * it.sb[2];
    const int hx = it.sb[3] >> 1;
    // coordinates of slot l of parity p, false outside the domain
    auto coords = [&](int l, int p, int k[4]) {
        const int j = l % hx, r = l / hx, r1 = r / it.sb[2];
        k[2] = b2 + r % it.sb[2];
        k[1] = b1 + r1 % it.sb[1];
        k[0] = r1 / it.sb[1];
        const bool in = k[0] < it.sb[0];
        k[0] += b0;
        k[3] = bz + 2 * j + ((p + it.par_o + k[0] + k[1] + k[2]) & 1);
        return in && k[0] < it.e[0] && k[1] < it.e[1] && k[2] < it.e[2] && k[3] < it.e[3];
    };
    for (int q = threadIdx.x; q < 2 * 8 * SMALL_SITES; q += SMALL_THREADS) {
        const int l = q % SMALL_SITES, d = (q / SMALL_SITES) & 7, par = q / (8 * SMALL_SITES);
        int code = -1, k[4];
        if (coords(l, par, k)) {
            int64_t row = 0;
            bool neg;
            if (hop_neighbour(it, k, par, d, row, neg)) {
                const int c0 = k[0] / it.sb[0], c1 = k[1] / it.sb[1], c2 = k[2] / it.sb[2], c3 = k[3] / it.sb[3];
                const int blk = c0 + it.sc[0] * (c1 + it.sc[1] * (c2 + it.sc[2] * c3));
                const int slot = (((k[0] - c0 * it.sb[0]) * it.sb[1] + k[1] - c1 * it.sb[1]) * it.sb[2] + k[2] - c2 * it.sb[2]) * hx +
                                 ((k[3] - c3 * it.sb[3]) >> 1);
                code = (blk << 7) | slot | (neg ? SMALL_NEG : 0);
                cx<float> u[3][3];
                load_link<P>(it.links, it.gV, d >> 1, row, u);
                float2 *w = sh.link[par][d][l];
#pragma unroll
                for (int j = 0; j < 9; j++) {
                    const cx<float> c = u[j / 3][j % 3];
                    if (d & 1)
                        w[3 * (j % 3) + j / 3] = f2(c.re, -c.im);
                    else
                        w[j] = f2(c.re, c.im);
                }
            }
        }
        sh.nb[par][d][l] = (short)code;
    }
    const int cc = threadIdx.x / SMALL_SITES, l = threadIdx.x % SMALL_SITES;
    const int col = col0 + cc;
    const bool have = col < it.ncol;
    // the thread's even and odd site
    int ke[4], ko[4];
    const bool own_e = coords(l, 0, ke) && have, own_o = coords(l, 1, ko) && have;
    const int64_t cb = it.fbase + (int64_t)(have ? col : 0) * it.nh;
    const int64_t ie = cb + (own_e ? local_lex(it, ke) >> 1 : 0), io = cb + (own_o ? local_lex(it, ko) >> 1 : 0);
    const SolveState *S = a.st + it.solve0 + (have ? col : 0);
    const float kap = (float)it.kappa, k2 = -kap * kap;
    const double scale = have ? S->scale : 0.0;  // a power of two, or 0: nothing to correct
    const int m = scale_exponent(scale);
    __syncthreads();  // links and neighbours are in place
    float2 acc[12], rp[12], x[12], v[12], rh[12], t[12], s[12];
#pragma unroll
    for (int j = 0; j < 12; j++) t[j] = rp[j] = x[j] = v[j] = rh[j] = f2(0.f, 0.f);
    // normalised defect: odd part to the neighbours, r = r'_e + kappa H_eo r'_o
    if (own_o && scale != 0.0) {
        const double2 *f = reinterpret_cast<const double2 *>(a.ro.p) + io;
#pragma unroll
        for (int j = 0; j < 12; j++) {
            const double2 c = __ldg(f + j * a.ro.stride);
            t[j] = f2(float_of(c.x, m, scale), float_of(c.y, m, scale));
        }
    }
    if (own_e && scale != 0.0) {
        const double2 *f = reinterpret_cast<const double2 *>(a.re.p) + ie;
#pragma unroll
        for (int j = 0; j < 12; j++) {
            const double2 c = __ldg(f + j * a.re.stride);
            rp[j] = f2(float_of(c.x, m, scale), float_of(c.y, m, scale));
        }
    }
    small_put(sh, SV_T, cc, l, t);
    cluster_sync(csize);
    float sums[PART_MAX] = {};
    if (own_e) {
        small_hops(sh, 0, SV_T, cc, l, acc);
#pragma unroll
        for (int j = 0; j < 12; j++) {
            rp[j] = __ffma2_rn(f2(kap, kap), acc[j], rp[j]);
            rh[j] = rp[j];
            sums[0] = fmaf(rp[j].x, rp[j].x, fmaf(rp[j].y, rp[j].y, sums[0]));
        }
    }
    small_put(sh, SV_P, cc, l, rp);
    small_put(sh, SV_S, cc, l, rp);
    int buf = 0;
    // the scalars live in lane c of warp 0
    const Cnum c0 = cn(0.0, 0.0);
    Cnum rho = c0, alpha = c0, inv = c0;
    double target2 = 0.0;
    int iters = 0, maxit = 0, status = 4, running = 0;
    {
        const double q = small_sums<1>(sh, sums, csize, rank, buf);
        buf ^= 1;
        if (threadIdx.x < 32) {
            const int c = threadIdx.x & (SMALL_COLS - 1);
            const double n = __shfl_sync(0xffffffffu, q, c);
            if (threadIdx.x < SMALL_COLS) {
                const bool hc = col0 + c < it.ncol;
                const SolveState *Sc = a.st + it.solve0 + (hc ? col0 + c : 0);
                running = hc && Sc->sigma > 0 && n > 0.0;
                rho = cn(n, 0.0);
                target2 = Sc->delta * Sc->delta * n;
                maxit = Sc->maxit;
                status = running ? 0 : 4;
                sh.go[c] = running;
            }
        }
        __syncthreads();
    }
    // the block-uniform state of the loop: every block of the cluster takes the same turns
    while (sh.go[0] || sh.go[1]) {
        if (own_o) {  // odd intermediate of p
            small_hops(sh, 1, SV_P, cc, l, acc);
            small_put(sh, SV_T, cc, l, acc);
        }
        cluster_sync(csize);
        sums[0] = sums[1] = 0.f;
        if (own_e) {  // v = p - kappa^2 H_eo tmp
            small_hops(sh, 0, SV_T, cc, l, acc);
            small_get(sh, SV_P, cc, l, v);
#pragma unroll
            for (int j = 0; j < 12; j++) {
                v[j] = __ffma2_rn(f2(k2, k2), acc[j], v[j]);
                f2_dot(sums[0], sums[1], rh[j], v[j]);
            }
        }
        {
            const double q = small_sums<2>(sh, sums, csize, rank, buf);
            buf ^= 1;
            if (threadIdx.x < 32) {
                const int c = threadIdx.x & (SMALL_COLS - 1);
                const Cnum hv = cn(__shfl_sync(0xffffffffu, q, 2 * c), __shfl_sync(0xffffffffu, q, 2 * c + 1));
                if (threadIdx.x < SMALL_COLS) {
                    if (!running || !bicg_alpha(rho, hv, alpha, inv)) {
                        alpha = c0;
                        if (running) status = 2;
                        running = 0;
                    }
                    sh.alpha[c] = f2((float)alpha.x, (float)alpha.y);
                    sh.upd[c] = running;
                }
            }
            __syncthreads();
        }
        const float2 al = sh.alpha[cc];
        if (own_e) {  // s = r - alpha v
            small_get(sh, SV_S, cc, l, s);
#pragma unroll
            for (int j = 0; j < 12; j++) {
                const float2 av = f2_cmul(al, v[j]);
                s[j] = f2(s[j].x - av.x, s[j].y - av.y);
            }
            small_put(sh, SV_S, cc, l, s);
        }
        cluster_sync(csize);
        if (own_o) {  // odd intermediate of s
            small_hops(sh, 1, SV_S, cc, l, acc);
            small_put(sh, SV_T, cc, l, acc);
        }
        cluster_sync(csize);
#pragma unroll
        for (int k = 0; k < PART_MAX; k++) sums[k] = 0.f;
        if (own_e) {  // t = s - kappa^2 H_eo tmp and the five products
            small_hops(sh, 0, SV_T, cc, l, acc);
            small_get(sh, SV_S, cc, l, s);
#pragma unroll
            for (int j = 0; j < 12; j++) {
                t[j] = __ffma2_rn(f2(k2, k2), acc[j], s[j]);
                f2_dot(sums[0], sums[1], t[j], s[j]);
                f2_dot(sums[2], sums[3], rh[j], s[j]);
                f2_dot(sums[4], sums[5], rh[j], t[j]);
                sums[6] = fmaf(t[j].x, t[j].x, fmaf(t[j].y, t[j].y, sums[6]));
                sums[7] = fmaf(s[j].x, s[j].x, fmaf(s[j].y, s[j].y, sums[7]));
            }
        }
        {
            const double q = small_sums<PART_MAX>(sh, sums, csize, rank, buf);
            buf ^= 1;
            if (threadIdx.x < 32) {
                const int c = threadIdx.x & (SMALL_COLS - 1);
                double w[PART_MAX];
#pragma unroll
                for (int k = 0; k < PART_MAX; k++) w[k] = __shfl_sync(0xffffffffu, q, c * PART_MAX + k);
                if (threadIdx.x < SMALL_COLS && running) {
                    Cnum omega, rc, beta;
                    status = bicg_omega(w, target2, inv, omega, rc, beta);
                    iters++;
                    if (!status && iters >= maxit) status = 3;
                    if (status) {
                        running = 0;
                        beta = c0;
                    } else {
                        rho = rc;
                    }
                    sh.omega[c] = f2((float)omega.x, (float)omega.y);
                    sh.beta[c] = f2((float)beta.x, (float)beta.y);
                }
                if (threadIdx.x < SMALL_COLS) sh.go[c] = running;
            }
            __syncthreads();
        }
        if (own_e && sh.upd[cc]) {  // x += alpha p + omega s ; r = s - omega t ; p = r + beta (p - omega v)
            const float2 om = sh.omega[cc], be = sh.beta[cc];
            float2 p[12];
            small_get(sh, SV_P, cc, l, p);
#pragma unroll
            for (int j = 0; j < 12; j++)
                xrp_update(&x[j].x, &p[j].x, &s[j].x, &t[j].x, &v[j].x, al.x, al.y, om.x, om.y, be.x, be.y);
            small_put(sh, SV_S, cc, l, s);
            small_put(sh, SV_P, cc, l, p);
        }
        cluster_sync(csize);
    }
    // e_o = r'_o + kappa H_oe e_e and the FP64 accumulation of both parts
    small_put(sh, SV_P, cc, l, x);
    cluster_sync(csize);
    const double sigma = have ? S->sigma : 0.0;
    if (own_e && sigma != 0.0) {
        double2 *f = reinterpret_cast<double2 *>(a.xe.p) + ie;
#pragma unroll
        for (int j = 0; j < 12; j++) {
            double2 c = f[j * a.xe.stride];
            c.x = fma(sigma, high_of(x[j].x), c.x);
            c.y = fma(sigma, high_of(x[j].y), c.y);
            f[j * a.xe.stride] = c;
        }
    }
    if (own_o && sigma != 0.0) {
        small_hops(sh, 1, SV_P, cc, l, acc);
        const double2 *g = reinterpret_cast<const double2 *>(a.ro.p) + io;
        double2 *f = reinterpret_cast<double2 *>(a.xo.p) + io;
#pragma unroll
        for (int j = 0; j < 12; j++) {
            const double2 o = __ldg(g + j * a.ro.stride);
            double2 c = f[j * a.xo.stride];
            c.x = fma(sigma, high_of(fmaf(kap, acc[j].x, float_of(o.x, m, scale))), c.x);
            c.y = fma(sigma, high_of(fmaf(kap, acc[j].y, float_of(o.y, m, scale))), c.y);
            f[j * a.xo.stride] = c;
        }
    }
    cluster_sync(csize);  // no block leaves while another reads its vectors
    if (rank == 0 && threadIdx.x < SMALL_COLS && col0 + (int)threadIdx.x < it.ncol) {
        SolveState &W = a.st[it.solve0 + col0 + threadIdx.x];
        W.iters = iters;
        W.total_iters += iters;
        W.status = status;
        W.active = 0;
    }
}

}  // namespace ddp
