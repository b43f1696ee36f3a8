// Solver engine: domain propagators S = D_Gamma^{-1} eta (Sec. 2, Eq. diric)
// for a batch of independent requests.
//
// Outer loop (FP64 defect correction): r = eta - D_Gamma x with FP64 links and
// vectors; stop a column when |r| <= tol |eta|.  Otherwise solve
// (2 kappa D_Gamma) e' = 2 kappa r / |r| with the even-odd Schur complement
//   (1 - kappa^2 H_eo H_oe) e'_e = r'_e + kappa H_eo r'_o,  e'_o = r'_o + kappa H_oe e'_e
// by BiCGStab in the storage format P to a relative tolerance delta, and
// accumulate x += |r| e' in FP64.
//
// Inner loop: every column of every request iterates together; per-column
// scalars live on the device and the loop runs inside a CUDA graph whose
// conditional WHILE node is driven by the device (no host round trip per
// iteration).  Converged columns freeze (alpha = omega = 0).
#pragma once

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <type_traits>

#include "ddp_host.h"

namespace ddp {

// Launches kernel k; chained: as a programmatic dependent of the kernel before it in the stream
// (see chain_wait).
template <class Args>
inline void launch_kernel(ddp_ctx *ctx, void (*k)(Args), int nblocks, int threads, const Args &a, bool chained) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    cfg.gridDim = dim3((unsigned)nblocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = ctx->stream;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = chained ? 1 : 0;
    cudaLaunchKernelEx(&cfg, k, a);  // an error stays pending, as with <<<>>>
}

// One application of the hopping term (CL: with the clover term of the items that have one).
// FP64: the input is brought into block fixed point in fx (a field of its size) first.
// Returns the number of kernels launched.
template <class Q, int EPI, int DOT, bool CL = false>
inline int launch_hop(ddp_ctx *ctx, int nblocks, int threads, HopArgs a, const FieldView &fx, bool chained = false) {
    if constexpr (Q::IS64) {
        FxArgs c;
        c.L = a.L;
        c.in = a.in;
        c.fx = fx;
        c.st = a.st;
        c.skip = a.skip;
        k_to_fx<<<nblocks, threads, 0, ctx->stream>>>(c);
        a.in = fx;
        k_hop_fx<EPI, DOT, CL, false><<<nblocks * FX_SPLIT, HOP_TS * fx_cols(a.L.CG), 0, ctx->stream>>>(a);
        return 2;
    } else {
        (void)fx;
        for (int j = 0; j < 6; j++) a.off[j] = (int64_t)j * a.in.stride * (int64_t)sizeof(typename Q::chunk);
        launch_kernel(ctx, k_hop<Q, EPI, DOT, CL>, nblocks, threads, a, chained);
        return 1;
    }
}

template <class Q, int EPI, int DOT, bool CL>
inline const void *hop_kernel() {
    if constexpr (Q::IS64)
        return (const void *)k_hop_fx<EPI, DOT, CL, false>;
    else
        return (const void *)k_hop<Q, EPI, DOT, CL>;
}

// Preferred shared-memory carveout of the inner-loop stencils (percent of the unified
// L1/shared memory; the rest is L1 for the neighbour gathers), set outside graph capture.
template <class Q, bool CL>
inline cudaError_t set_hop_carveout(int percent) {
    if (percent < 0) return cudaSuccess;
    const void *k[3] = {hop_kernel<Q, EPI_PLAIN, DOT_NONE, CL>(), hop_kernel<Q, EPI_MHAT, DOT_RHAT, CL>(),
                        hop_kernel<Q, EPI_MHAT, DOT_TS, CL>()};
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < 3 && e == cudaSuccess; i++)
        e = cudaFuncSetAttribute(k[i], cudaFuncAttributePreferredSharedMemoryCarveout, percent);
    return e;
}

// Launch configuration of the small-domain kernel.
template <class P>
inline void small_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute attr[1], int csize, int nclusters) {
    cfg.gridDim = dim3((unsigned)(nclusters * csize));
    cfg.blockDim = dim3(SMALL_THREADS);
    cfg.dynamicSmemBytes = sizeof(SmallShared);
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)csize;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
}

// The largest cluster of the small-domain kernel this device runs (asked once per context), with
// the kernel's attributes set; 0: none.
template <class P>
inline int small_clusters(ddp_ctx *ctx) {
    if constexpr (P::IS64) {
        return 0;
    } else {
        const bool set = cudaFuncSetAttribute(k_small<P>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)sizeof(SmallShared)) == cudaSuccess;
        if (ctx->max_cluster < 0) {
            ctx->max_cluster = 0;
            for (int c = SMALL_MAX_CLUSTER; set && c > 0 && !ctx->max_cluster; c /= 2) {
                cudaLaunchConfig_t cfg = {};
                cudaLaunchAttribute attr[1];
                small_config<P>(cfg, attr, c, 1);
                int n = 0;
                if (cudaOccupancyMaxActiveClusters(&n, k_small<P>, &cfg) == cudaSuccess && n > 0) ctx->max_cluster = c;
            }
            cudaGetLastError();
        }
        return ctx->max_cluster;
    }
}

template <class P>
struct Engine {
    ddp_ctx *ctx;
    int prec;
    Plan plan;
    FieldView be, bo, xe, xo, re64, ro64;      // FP64
    FieldView r, rh, p, v, s, t, xi, tmp, ro;  // storage format P (rh: ShadowOf<P>)
    // block fixed-point input of an FP64 hop, over fields that are dead at the time: the inner
    // fields during a true residual, the FP64 residual during the inner loop of the FP64 path
    FieldView fx_outer, fx_inner;
    Partials A, B;
    Item *d_items = nullptr;
    SolveState *d_st = nullptr;
    LoopCtl *d_ctl = nullptr;
    int loop_mode = 0;  // how the iteration body being captured ends (see FinArgs)
    cudaGraphConditionalHandle loop_handle = 0;
    std::vector<SolveState> h_st;
    Launch L;
    int threads = 0;
    cudaGraphExec_t loop_exec = nullptr;
    cudaGraph_t loop_graph = nullptr;
    long launches = 0;
    bool chained = false;      // kernels are launched as dependents of one another (see chain_wait)
    int grid = 0, solves = 0;  // blocks and columns of the next launches: of all items, or of the large ones
    bool clov = false;  // some item of the plan has a clover term

    ~Engine() {
        if (loop_exec) cudaGraphExecDestroy(loop_exec);
        if (loop_graph) cudaGraphDestroy(loop_graph);
    }

    HopArgs hop_args(int par, FieldView in, FieldView out, FieldView v1, FieldView v2, FieldView rhv,
                     Partials part, int skip = 0) {
        HopArgs a;
        a.st = d_st;
        a.skip = skip;
        a.L = L;
        a.p = par;
        a.in = in;
        a.out = out;
        a.v1 = v1;
        a.v2 = v2;
        a.rh = rhv;
        a.part = part;
        return a;
    }

    template <class Q, int EPI, int DOT, bool CL = false>
    void hop(const HopArgs &a) {
        launches += launch_hop<Q, EPI, DOT, CL>(ctx, grid, threads, a, EPI == EPI_RESID ? fx_outer : fx_inner, chained);
    }

    template <class Q, int OP>
    void blas(Partials part, int skip = 1) {
        BlasArgs a;
        a.skip = skip;
        a.L = L;
        a.x = xi;
        a.r = r;
        a.rh = rh;
        a.p = p;
        a.v = v;
        a.s = s;
        a.t = t;
        a.st = d_st;
        a.part = part;
        launch_kernel(ctx, k_blas<Q, OP>, grid, threads, a, chained);
        launches++;
    }

    template <int FIN>
    void fin() {
        FinArgs a;
        a.st = d_st;
        a.nsolve = solves;
        a.A = A;
        a.B = B;
        a.ctl = d_ctl;
        a.loop_mode = FIN == FIN_OMEGA ? loop_mode : 0;
        a.loop = loop_handle;
        using R = typename std::conditional<FIN == FIN_BNORM || FIN == FIN_RESID, double, typename P::real>::type;
        launch_kernel(ctx, k_fin<FIN, R>, solves, FIN_THREADS, a, chained);
        launches++;
    }

    void norm64(FieldView f, Partials part) {
        BlasArgs a;
        memset(&a, 0, sizeof(a));
        a.skip = 0;
        a.L = L;
        a.x = f;
        a.st = d_st;
        a.part = part;
        k_blas<PF64, OP_NORM><<<grid, threads, 0, ctx->stream>>>(a);
        launches++;
    }

    // to_low: lo = scale hi (times T^-1 of the site when clov_inv); else hi += sigma lo
    void conv(bool to_low, FieldView lo, FieldView hi, int par = 0, bool clov_inv = false) {
        ConvArgs a;
        a.L = L;
        a.lo = lo;
        a.hi = hi;
        a.st = d_st;
        a.p = par;
        a.clov = clov_inv ? 1 : 0;
        if (to_low)
            k_to_low<P><<<grid, threads, 0, ctx->stream>>>(a);
        else
            k_accum<P><<<grid, threads, 0, ctx->stream>>>(a);
        launches++;
    }

    // One BiCGStab iteration on the Schur complement (van der Vorst 1992); with the
    // clover term the operator is 1 - kappa^2 T_ee^-1 H_eo T_oo^-1 H_oe.
    template <bool CL>
    void iteration_body_t() {
        FieldView none = {nullptr, nullptr, 0};
        hop<P, EPI_PLAIN, DOT_NONE, CL>(hop_args(1, p, tmp, none, none, none, A, 1));   // tmp = T^-1 H_oe p
        hop<P, EPI_MHAT, DOT_RHAT, CL>(hop_args(0, tmp, v, p, none, rh, A, 1));        // v = p - k^2 T^-1 H_eo tmp
        fin<FIN_ALPHA>();                                                               // alpha = rho / (rh, v)
        blas<P, OP_S_UPDATE>(A);                                                        // s = r - alpha v
        hop<P, EPI_PLAIN, DOT_NONE, CL>(hop_args(1, s, tmp, none, none, none, A, 1));   // tmp = T^-1 H_oe s
        hop<P, EPI_MHAT, DOT_TS, CL>(hop_args(0, tmp, t, s, none, rh, A, 1));          // t = s - k^2 T^-1 H_eo tmp
        fin<FIN_OMEGA>();                                      // omega, beta, convergence, loop control
        blas<P, OP_XRP_UPDATE>(A);                                                      // x, r, p
    }
    void iteration_body() {
        chained = !P::IS64;  // the FP64 stencil's kernels do not take part
        if (clov)
            iteration_body_t<true>();
        else
            iteration_body_t<false>();
        chained = false;
    }

    // The inner loop of the large items as a graph (nothing to build without any).
    int build_loop_graph() {
        if (!plan.nlarge) return DDP_OK;
        large_items();
        const int rc = capture_loop();
        all_items();
        return rc;
    }

    int capture_loop() {
        cudaStream_t st = ctx->stream;
        DDP_CUDA(ctx, (set_hop_carveout<P, false>(carveout_for(ctx->prm, prec))));
        DDP_CUDA(ctx, (set_hop_carveout<P, true>(carveout_for(ctx->prm, prec))));
        if (ctx->prm.use_conditional) {
            DDP_CUDA(ctx, cudaGraphCreate(&loop_graph, 0));
            cudaGraphConditionalHandle h;
            DDP_CUDA(ctx, cudaGraphConditionalHandleCreate(&h, loop_graph, 1, cudaGraphCondAssignDefault));
            // the parameter union has no default constructor: build it in zeroed storage
            alignas(cudaGraphNodeParams) unsigned char cp_buf[sizeof(cudaGraphNodeParams)];
            memset(cp_buf, 0, sizeof(cp_buf));
            cudaGraphNodeParams &cp = *reinterpret_cast<cudaGraphNodeParams *>(cp_buf);
            cp.type = cudaGraphNodeTypeConditional;
            cp.conditional.handle = h;
            cp.conditional.type = cudaGraphCondTypeWhile;
            cp.conditional.size = 1;
            cudaGraphNode_t node;
            DDP_CUDA(ctx, cudaGraphAddNode(&node, loop_graph, nullptr, nullptr, 0, &cp));
            cudaGraph_t body = cp.conditional.phGraph_out[0];
            DDP_CUDA(ctx, cudaStreamBeginCaptureToGraph(st, body, nullptr, nullptr, 0,
                                                        cudaStreamCaptureModeThreadLocal));
            loop_mode = 1;
            loop_handle = h;
            iteration_body();  // its FIN_OMEGA sets the loop condition
            loop_mode = 0;
            cudaGraph_t captured;
            cudaError_t e = cudaStreamEndCapture(st, &captured);
            if (e != cudaSuccess) return set_cuda_error(ctx, e, "capture of the inner loop");
            DDP_CUDA(ctx, cudaGraphInstantiate(&loop_exec, loop_graph, 0));
        } else {
            DDP_CUDA(ctx, cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
            loop_mode = 2;
            for (int i = 0; i < ctx->prm.host_chunk; i++) iteration_body();
            loop_mode = 0;
            cudaError_t e = cudaStreamEndCapture(st, &loop_graph);
            if (e != cudaSuccess) return set_cuda_error(ctx, e, "capture of the inner loop");
            DDP_CUDA(ctx, cudaGraphInstantiate(&loop_exec, loop_graph, 0));
        }
        return DDP_OK;
    }

    int run_inner() {
        // launches per iteration: 4 stencils (FP64: conversion and hop), 2 vector updates, 2
        // scalar-recurrence kernels (the second of which also runs the loop control)
        const long per_iter = P::IS64 ? 12 : 8;
        if (ctx->prm.use_conditional) {
            DDP_CUDA(ctx, cudaGraphLaunch(loop_exec, ctx->stream));
        } else {
            LoopCtl hc;
            for (int guard = 0; guard < 1 + ctx->prm.max_inner / std::max(1, ctx->prm.host_chunk); guard++) {
                DDP_CUDA(ctx, cudaGraphLaunch(loop_exec, ctx->stream));
                DDP_CUDA(ctx, cudaMemcpyAsync(&hc, d_ctl, sizeof(hc), cudaMemcpyDeviceToHost, ctx->stream));
                DDP_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
                if (!hc.pad) break;
            }
        }
        LoopCtl hc;
        DDP_CUDA(ctx, cudaMemcpyAsync(&hc, d_ctl, sizeof(hc), cudaMemcpyDeviceToHost, ctx->stream));
        DDP_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
        launches += per_iter * (long)hc.iter;
        return DDP_OK;
    }

    // ----------------------------------------------------------- building blocks

    // a partial slot: the most sums of a stencil in the compute precision, or one FP64 norm
    static constexpr size_t PART_BYTES = PART_MAX * sizeof(typename P::real);
    static size_t bytes_needed(int64_t cap, int64_t npart, int nitems, int nsolve) {
        return 6 * field_bytes<PF64>(cap) + 9 * field_bytes<P>(cap) +
               (size_t)npart * (PART_BYTES + sizeof(double)) + 2048 + (size_t)nitems * sizeof(Item) +
               (size_t)nsolve * sizeof(SolveState) + sizeof(LoopCtl) + 8192;
    }

    // Every field gets room for cap site-columns per parity (stride cap).
    void carve(Arena &a, int64_t cap, int64_t npart, int nitems, int nsolve) {
        a.reset();
        be = carve_field<PF64>(a, cap);
        bo = carve_field<PF64>(a, cap);
        xe = carve_field<PF64>(a, cap);
        xo = carve_field<PF64>(a, cap);
        re64 = carve_field<PF64>(a, cap);
        ro64 = carve_field<PF64>(a, cap);
        r = carve_field<P>(a, cap);
        rh = carve_field<typename ShadowOf<P>::type>(a, cap);
        p = carve_field<P>(a, cap);
        v = carve_field<P>(a, cap);
        s = carve_field<P>(a, cap);
        t = carve_field<P>(a, cap);
        xi = carve_field<P>(a, cap);
        tmp = carve_field<P>(a, cap);
        ro = carve_field<P>(a, cap);
        auto fx_over = [&](FieldView first) {
            FieldView f;
            f.stride = cap;
            f.p = first.p;
            f.scale = reinterpret_cast<float *>((char *)first.p + (size_t)cap * PFX::NCH * sizeof(PFX::chunk));
            return f;
        };
        // 196 bytes a site-column: within r, rh, p, v, s, t (240 at the least, BF16) and within
        // re64, ro64 (384), which lie one after another
        static_assert((P::NCH * 5 + ShadowOf<P>::type::NCH) * 16 >= PFX::NCH * 16 + 4, "fixed-point field over the inner fields");
        fx_outer = fx_over(r);
        fx_inner = fx_over(re64);
        A.d = a.take(npart * PART_BYTES);
        B.d = a.take(npart * sizeof(double));  // true-residual norms only
        d_items = (Item *)a.take(nitems * sizeof(Item));
        d_st = (SolveState *)a.take(nsolve * sizeof(SolveState));
        d_ctl = (LoopCtl *)a.take(sizeof(LoopCtl));
    }

    void all_items() {
        grid = plan.nblocks;
        solves = plan.nsolve;
    }
    void large_items() {
        grid = plan.nblocks_large;
        solves = plan.nsolve_large;
    }

    // Upload the work table of the current plan and the per-column states.
    int upload(const std::vector<SolveState> &states) {
        cudaStream_t st = ctx->stream;
        L = make_launch(plan, d_items);
        threads = plan.TS * plan.CG;
        all_items();
        h_st = states;
        for (SolveState &S : h_st) {
            const Item &it = plan.items[S.item];
            S.ntiles = it.ntiles;
            S.pbase = it.pbase + (int64_t)S.col * it.ntiles;
            S.kappa = it.kappa;
        }
        DDP_CUDA(ctx, cudaMemcpyAsync(d_items, plan.items.data(), plan.items.size() * sizeof(Item),
                                      cudaMemcpyHostToDevice, st));
        DDP_CUDA(ctx, cudaMemcpyAsync(d_st, h_st.data(), plan.nsolve * sizeof(SolveState), cudaMemcpyHostToDevice,
                                      st));
        LoopCtl c0 = {0, 0, ctx->prm.max_inner, 0};
        DDP_CUDA(ctx, cudaMemcpyAsync(d_ctl, &c0, sizeof(c0), cudaMemcpyHostToDevice, st));
        return DDP_OK;
    }

    SolveState fresh_state(int item, int col, double tol) const {
        SolveState S;
        memset(&S, 0, sizeof(S));
        S.item = item;
        S.col = col;
        S.tol = tol;
        S.floor_delta = ctx->prm.floor_delta[prec];
        S.maxit = ctx->prm.max_inner;
        S.status = 4;
        return S;
    }

    // eta (or the point sources) of item i into the FP64 source fields; x = 0 there.
    int pack_source(int i, const Job &job) {
        cudaStream_t st = ctx->stream;
        PackArgs pa;
        memset(&pa, 0, sizeof(pa));
        pa.it = plan.items[i];
        pa.user = (const double2 *)job.eta;
        pa.fe = be;
        pa.fo = bo;
        pa.src_l = job.src_l;
        pa.xe = xe;
        pa.xo = xo;
        int64_t nt = 2 * (int64_t)pa.it.nh * pa.it.ncol;
        k_pack<<<(unsigned)((nt + 255) / 256), 256, 0, st>>>(pa);
        launches++;
        return DDP_OK;
    }

    int unpack_result(int i, double *out) {
        PackArgs pa;
        memset(&pa, 0, sizeof(pa));
        pa.it = plan.items[i];
        pa.uout = (double2 *)out;
        pa.fe = xe;
        pa.fo = xo;
        int64_t nt = 2 * (int64_t)pa.it.nh * pa.it.ncol;
        k_unpack<<<(unsigned)((nt + 255) / 256), 256, 0, ctx->stream>>>(pa);
        launches++;
        DDP_CUDA(ctx, cudaGetLastError());
        return DDP_OK;
    }

    void source_norms() {
        norm64(be, A);
        norm64(bo, B);
        fin<FIN_BNORM>();
    }

    // r64 = eta - D_Gamma x (FP64 links and vectors); skip_hop: x is known to be 0,
    // so r64 = eta and the partials of |eta|^2 left by source_norms() are reused.
    void residual(bool skip_hop) {
        FieldView none = {nullptr, nullptr, 0};
        if (!skip_hop) {
            if (clov) {
                hop<PF64, EPI_RESID, DOT_NORM, true>(hop_args(0, xo, re64, xe, be, none, A, 2));
                hop<PF64, EPI_RESID, DOT_NORM, true>(hop_args(1, xe, ro64, xo, bo, none, B, 2));
            } else {
                hop<PF64, EPI_RESID, DOT_NORM>(hop_args(0, xo, re64, xe, be, none, A, 2));
                hop<PF64, EPI_RESID, DOT_NORM>(hop_args(1, xe, ro64, xo, bo, none, B, 2));
            }
        }
        fin<FIN_RESID>();
    }

    int download_states() {
        DDP_CUDA(ctx, cudaMemcpyAsync(h_st.data(), d_st, plan.nsolve * sizeof(SolveState), cudaMemcpyDeviceToHost,
                                      ctx->stream));
        DDP_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
        return DDP_OK;
    }

    // One correction: inner solve of the normalised defect and FP64 accumulation.
    // With 2 kappa D = [[T_ee, -k H_eo], [-k H_oe, T_oo]] and r' the normalised defect:
    //   (1 - k^2 T_ee^-1 H_eo T_oo^-1 H_oe) e_e = T_ee^-1 (r'_e + k H_eo T_oo^-1 r'_o),
    //   e_o = T_oo^-1 r'_o + k T_oo^-1 H_oe e_e   (T = 1 without the clover term).
    template <bool CL>
    int correction_t(bool r_is_eta) {
        FieldView none = {nullptr, nullptr, 0};
        conv(true, s, r_is_eta ? be : re64, 0);
        conv(true, ro, r_is_eta ? bo : ro64, 1, CL);                                  // ro = T_oo^-1 r'_o
        hop<P, EPI_RHS, DOT_NORM, CL>(hop_args(0, ro, r, s, none, none, A));         // r = T_ee^-1 (r'_e + k H_eo ro)
        blas<P, OP_INIT>(A, 0);
        DDP_CUDA(ctx, cudaMemsetAsync(d_ctl, 0, offsetof(LoopCtl, maxit), ctx->stream));
        fin<FIN_INIT>();
        DDP_CUDA(ctx, cudaGetLastError());
        int rc = run_inner();
        if (rc) return rc;
        hop<P, EPI_AXPY_K, DOT_NONE, CL>(hop_args(1, xi, tmp, ro, none, none, A));  // e_o = ro + k T^-1 H_oe e_e
        conv(false, xi, xe);
        conv(false, tmp, xo);
        return DDP_OK;
    }
    int correct_large(bool r_is_eta) {
        if (!plan.nlarge) return DDP_OK;
        large_items();
        const int rc = clov ? correction_t<true>(r_is_eta) : correction_t<false>(r_is_eta);
        all_items();
        return rc;
    }
    // The groups of small items, one per cluster size, and the large items have nothing in common
    // and each of them fills a part of the SMs only: they run beside one another, the groups on
    // streams of their own between a fork and a join of the work stream.  One after another (FP32,
    // 12 columns): clusters of 1 to 8 blocks 3.53 ms, with an 8^4 block 5.29, so 1.35 and 2.78; all by the
    // per-step kernels 1.94 and 2.73.
    int correction(bool r_is_eta) {
        if constexpr (P::IS64) {
            return correct_large(r_is_eta);
        } else {
            // the longest first; without large items one group stays on the work stream
            const int n = (int)plan.small.size(), nside = plan.nlarge ? n : std::max(0, n - 1);
            int rc = fork(nside);
            if (rc) return rc;
            for (int i = 0; i < n && !rc; i++) {
                rc = correct_small(plan.small[n - 1 - i], r_is_eta, i < nside ? ctx->side[i].stream : ctx->stream);
                if (!rc && i < nside && cudaEventRecord(ctx->side[i].done, ctx->side[i].stream) != cudaSuccess)
                    rc = set_cuda_error(ctx, cudaGetLastError(), "end of a group of small domains");
            }
            if (!rc) rc = correct_large(r_is_eta);
            for (int i = 0; i < nside; i++) {
                const cudaError_t e = rc ? cudaStreamSynchronize(ctx->side[i].stream)
                                         : cudaStreamWaitEvent(ctx->stream, ctx->side[i].done, 0);
                if (e != cudaSuccess && !rc) rc = set_cuda_error(ctx, e, "join of the small domains");
            }
            return rc;
        }
    }
    // The first n side streams wait for what the work stream has been given so far.
    int fork(int n) {
        if (!n) return DDP_OK;
        if (!ctx->ev_fork) DDP_CUDA(ctx, cudaEventCreateWithFlags(&ctx->ev_fork, cudaEventDisableTiming));
        while ((int)ctx->side.size() < n) {
            ddp_ctx::Side s;
            DDP_CUDA(ctx, cudaEventCreateWithFlags(&s.done, cudaEventDisableTiming));
            const cudaError_t e = cudaStreamCreateWithFlags(&s.stream, cudaStreamNonBlocking);
            if (e != cudaSuccess) {
                cudaEventDestroy(s.done);
                return set_cuda_error(ctx, e, "side stream");
            }
            ctx->side.push_back(s);
        }
        DDP_CUDA(ctx, cudaEventRecord(ctx->ev_fork, ctx->stream));
        for (int i = 0; i < n; i++) DDP_CUDA(ctx, cudaStreamWaitEvent(ctx->side[i].stream, ctx->ev_fork, 0));
        return DDP_OK;
    }

    // One correction of the small items of one cluster size (small.cuh), in one kernel.
    int correct_small(const Plan::Small &g, bool r_is_eta, cudaStream_t stream) {
        SmallArgs a;
        a.items = d_items + g.item0;
        a.nitems = g.nitems;
        a.csize = g.csize;
        a.re = r_is_eta ? be : re64;
        a.ro = r_is_eta ? bo : ro64;
        a.xe = xe;
        a.xo = xo;
        a.st = d_st;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        small_config<P>(cfg, attr, g.csize, g.nclusters);
        cfg.stream = stream;
        DDP_CUDA(ctx, cudaLaunchKernelEx(&cfg, k_small<P>, a));
        launches++;
        return DDP_OK;
    }

    void drop_graph() {
        if (loop_exec) cudaGraphExecDestroy(loop_exec);
        if (loop_graph) cudaGraphDestroy(loop_graph);
        loop_exec = nullptr;
        loop_graph = nullptr;
    }

    // ----------------------------------------------------------- one-shot solve

    int run(const std::vector<Job> &in, std::vector<JobInfo> &infos) {
        const EngineParams &prm = ctx->prm;
        // the work table in the order of the classes: per-step items first
        const int maxc = small_clusters<P>(ctx);
        std::vector<int> cls(in.size());
        std::vector<size_t> order(in.size());
        for (size_t i = 0; i < in.size(); i++) {
            cls[i] = job_class(in[i], prec, prm, maxc);
            order[i] = i;
        }
        std::stable_sort(order.begin(), order.end(), [&](size_t x, size_t y) { return cls[x] < cls[y]; });
        std::vector<Job> jobs;
        std::vector<int> sorted;
        for (size_t i : order) {
            jobs.push_back(in[i]);
            sorted.push_back(cls[i]);
        }
        make_plan(jobs, prec, prm, plan);
        plan_classes(sorted, maxc, plan);
        clov = false;
        for (auto &j : jobs) clov = clov || j.clov;
        DDP_CUDA(ctx, ctx->ws.reserve(bytes_needed(plan.nfield, plan.npart, (int)plan.items.size(), plan.nsolve)));
        carve(ctx->ws, plan.nfield, plan.npart, (int)plan.items.size(), plan.nsolve);
        std::vector<SolveState> states(plan.nsolve);
        for (size_t i = 0; i < plan.items.size(); i++)
            for (int c = 0; c < plan.items[i].ncol; c++)
                states[plan.items[i].solve0 + c] = fresh_state((int)i, c, jobs[i].tol);
        int rc = upload(states);
        if (rc) return rc;
        for (size_t i = 0; i < jobs.size(); i++)
            if ((rc = pack_source((int)i, jobs[i]))) return rc;
        source_norms();
        DDP_CUDA(ctx, cudaGetLastError());
        if ((rc = build_loop_graph())) return rc;
        int cycles = 0;
        for (int cyc = 0; cyc <= prm.max_outer; cyc++) {
            residual(cyc == 0);
            if ((rc = download_states())) return rc;
            bool all_done = true;
            for (auto &S : h_st) all_done = all_done && S.outer_done;
            if (all_done || cyc == prm.max_outer) break;
            cycles++;
            if ((rc = correction(cyc == 0))) return rc;
        }
        for (size_t i = 0; i < jobs.size(); i++)
            if ((rc = unpack_result((int)i, jobs[i].out))) return rc;
        DDP_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
        infos.assign(jobs.size(), JobInfo());
        for (size_t i = 0; i < jobs.size(); i++) {
            const Item &it = plan.items[i];
            JobInfo &inf = infos[order[i]];
            inf.outer = cycles;
            inf.relres.resize(it.ncol);
            bool ok = true;
            int inner = 0;
            for (int c = 0; c < it.ncol; c++) {
                const SolveState &S = h_st[it.solve0 + c];
                double rr = (S.bnorm2 > 0) ? sqrt(S.rr64 / S.bnorm2) : 0.0;
                inf.relres[c] = rr;
                ok = ok && (rr <= jobs[i].tol);
                inner = std::max(inner, S.total_iters);
                inf.column_iters += S.total_iters;
            }
            inf.inner = inner;
            inf.status = ok ? DDP_OK : DDP_ERR_NOT_CONVERGED;
        }
        ctx->launches += launches;
        launches = 0;
        return DDP_OK;
    }
};

template <class P>
int solve_jobs(ddp_ctx *ctx, int prec, std::vector<Job> &jobs, std::vector<JobInfo> &infos) {
    Engine<P> eng;
    eng.ctx = ctx;
    eng.prec = prec;
    return eng.run(jobs, infos);
}

// out = D_Gamma psi with the stencil of storage format P (App. A, Sec. 2).
template <class P>
int apply_dirac_impl(ddp_ctx *ctx, const Job &job, const double *psi, double *out, int prec) {
    std::vector<Job> jobs(1, job);
    Plan plan;
    make_plan(jobs, prec, ctx->prm, plan);
    const int64_t NF = plan.nfield;
    size_t need = 4 * field_bytes<P>(NF) + (P::IS64 ? field_bytes<PFX>(NF) : 0) + sizeof(Item) + 1024;
    DDP_CUDA(ctx, ctx->scratch.reserve(need));
    Arena &a = ctx->scratch;
    a.reset();
    FieldView ie = carve_field<P>(a, NF), io = carve_field<P>(a, NF);
    FieldView oe = carve_field<P>(a, NF), oo = carve_field<P>(a, NF);
    FieldView fx = {nullptr, nullptr, 0};
    if (P::IS64) fx = carve_field<PFX>(a, NF);
    Item *d_items = (Item *)a.take(sizeof(Item));
    cudaStream_t st = ctx->stream;
    DDP_CUDA(ctx, cudaMemcpyAsync(d_items, plan.items.data(), sizeof(Item), cudaMemcpyHostToDevice, st));
    PackArgs pa;
    memset(&pa, 0, sizeof(pa));
    pa.it = plan.items[0];
    pa.user = (const double2 *)psi;
    pa.uout = (double2 *)out;
    int64_t nt = 2 * (int64_t)pa.it.nh * pa.it.ncol;
    unsigned nb = (unsigned)((nt + 255) / 256);
    k_pack_low<P><<<nb, 256, 0, st>>>(pa, ie, io);
    const Launch L = make_launch(plan, d_items);
    FieldView none = {nullptr, nullptr, 0};
    HopArgs h;
    h.st = nullptr;
    h.skip = 0;
    h.L = L;
    h.v2 = none;
    h.rh = none;
    h.part.d = nullptr;
    h.p = 0;
    h.in = io;
    h.out = oe;
    h.v1 = ie;
    auto dirac = [&]() {
        if (job.clov)
            ctx->launches += launch_hop<P, EPI_DIRAC, DOT_NONE, true>(ctx, plan.nblocks, plan.TS * plan.CG, h, fx);
        else
            ctx->launches += launch_hop<P, EPI_DIRAC, DOT_NONE>(ctx, plan.nblocks, plan.TS * plan.CG, h, fx);
    };
    dirac();
    h.p = 1;
    h.in = ie;
    h.out = oo;
    h.v1 = io;
    dirac();
    k_unpack_low<P><<<nb, 256, 0, st>>>(pa, oe, oo);
    ctx->launches += 2;
    DDP_CUDA(ctx, cudaGetLastError());
    return DDP_OK;
}

// Timing of one inner-loop stencil variant on fields of the given domain
// (contents: zeros, which does not change the kernel's work), CUDA events on
// the context's stream around `iters` back-to-back launches after 3 warm-up
// launches.  kernel: DDP_HOP_PLAIN  tmp = H_oe p;  DDP_HOP_SCHUR_RHAT  v = p -
// kappa^2 H_eo tmp with the (rh, v) partials;  DDP_HOP_SCHUR_TS  t = s -
// kappa^2 H_eo tmp with the partials of its five products.  Algorithmic bytes per
// launch: the spinors the variant reads or writes once per output
// site-column (2, 4 and 3 of them; the shadow residual of the (rh, v) variant
// in its own storage, BF16 for FP32 storage; that of the (t, s) variant is not
// counted) plus the 8 links touching each
// output site once for all columns.
template <class P>
int time_hop_impl(ddp_ctx *ctx, const Job &job, int prec, int kernel, int iters, float *ms, double *bytes) {
    std::vector<Job> jobs(1, job);
    Plan plan;
    make_plan(jobs, prec, ctx->prm, plan);
    const int64_t NF = plan.nfield;
    size_t need = 4 * field_bytes<P>(NF) + (P::IS64 ? field_bytes<PFX>(NF) : 0) + (size_t)plan.npart * PART_MAX * 8 + 1024 +
                  sizeof(Item) + 1024;
    DDP_CUDA(ctx, ctx->scratch.reserve(need));
    Arena &a = ctx->scratch;
    a.reset();
    FieldView in = carve_field<P>(a, NF), v1 = carve_field<P>(a, NF), rhv = carve_field<P>(a, NF),
              out = carve_field<P>(a, NF);
    FieldView fx = {nullptr, nullptr, 0};
    if (P::IS64) fx = carve_field<PFX>(a, NF);
    Partials A;
    A.d = a.take(plan.npart * PART_MAX * sizeof(double));
    Item *d_items = (Item *)a.take(sizeof(Item));
    cudaStream_t st = ctx->stream;
    DDP_CUDA(ctx, cudaMemcpyAsync(d_items, plan.items.data(), sizeof(Item), cudaMemcpyHostToDevice, st));
    size_t fb = (size_t)NF * sizeof(typename P::chunk) * P::NCH;
    DDP_CUDA(ctx, cudaMemsetAsync(in.p, 0, fb, st));
    DDP_CUDA(ctx, cudaMemsetAsync(v1.p, 0, fb, st));
    DDP_CUDA(ctx, cudaMemsetAsync(rhv.p, 0, fb, st));
    if (P::SCALED) {
        DDP_CUDA(ctx, cudaMemsetAsync(in.scale, 0, NF * sizeof(float), st));
        DDP_CUDA(ctx, cudaMemsetAsync(v1.scale, 0, NF * sizeof(float), st));
        DDP_CUDA(ctx, cudaMemsetAsync(rhv.scale, 0, NF * sizeof(float), st));
    }
    const Launch L = make_launch(plan, d_items);
    HopArgs h;
    FieldView none = {nullptr, nullptr, 0};
    h.st = nullptr;
    h.skip = 0;
    h.L = L;
    h.p = (kernel == DDP_HOP_PLAIN) ? 1 : 0;
    h.in = in;
    h.out = out;
    h.v1 = (kernel == DDP_HOP_PLAIN) ? none : v1;
    h.v2 = none;
    h.rh = (kernel == DDP_HOP_PLAIN) ? none : rhv;
    h.part = A;
    DDP_CUDA(ctx, (set_hop_carveout<P, false>(carveout_for(ctx->prm, prec))));
    auto launch = [&]() {
        if (kernel == DDP_HOP_PLAIN)
            ctx->launches += launch_hop<P, EPI_PLAIN, DOT_NONE>(ctx, plan.nblocks, plan.TS * plan.CG, h, fx);
        else if (kernel == DDP_HOP_SCHUR_RHAT)
            ctx->launches += launch_hop<P, EPI_MHAT, DOT_RHAT>(ctx, plan.nblocks, plan.TS * plan.CG, h, fx);
        else
            ctx->launches += launch_hop<P, EPI_MHAT, DOT_TS>(ctx, plan.nblocks, plan.TS * plan.CG, h, fx);
    };
    cudaEvent_t e0, e1;
    DDP_CUDA(ctx, cudaEventCreate(&e0));
    DDP_CUDA(ctx, cudaEventCreate(&e1));
    for (int i = 0; i < 3; i++) launch();
    DDP_CUDA(ctx, cudaEventRecord(e0, st));
    for (int i = 0; i < iters; i++) launch();
    DDP_CUDA(ctx, cudaEventRecord(e1, st));
    DDP_CUDA(ctx, cudaEventSynchronize(e1));
    float t = 0;
    DDP_CUDA(ctx, cudaEventElapsedTime(&t, e0, e1));
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    DDP_CUDA(ctx, cudaGetLastError());
    *ms = t / iters;
    const double site_cols = (double)plan.items[0].nh * job.ncol;
    const double spinor = (double)sizeof(typename P::chunk) * P::NCH + (P::SCALED ? 4.0 : 0.0);
    const double link = P::IS64 ? 144.0 : (std::is_same<P, PF32>::value ? 48.0 : 24.0);
    using SH = typename ShadowOf<P>::type;
    const double shadow = (double)sizeof(typename SH::chunk) * SH::NCH + (SH::SCALED ? 4.0 : 0.0);
    // spinors of the storage format read or written once per output site-column, plus
    // the shadow residual (in its own format) of the (rh, v) variant
    const double per_col = (kernel == DDP_HOP_PLAIN) ? 2 * spinor
                           : (kernel == DDP_HOP_SCHUR_RHAT) ? 3 * spinor + shadow : 3 * spinor;
    // every link touching an output site: 8 per output site (4 forward + 4 backward)
    *bytes = site_cols * per_col + (double)plan.items[0].nh * 8.0 * link;
    return DDP_OK;
}

}  // namespace ddp
