// Solver engine and server instantiated for the PF64 storage format.
#include "serve_engine.cuh"

namespace ddp {
template int solve_jobs<PF64>(ddp_ctx *, int, std::vector<Job> &, std::vector<JobInfo> &);
template int apply_dirac_impl<PF64>(ddp_ctx *, const Job &, const double *, double *, int);
template int time_hop_impl<PF64>(ddp_ctx *, const Job &, int, int, int, float *, double *);
template ServerBase *make_server<PF64>(ddp_ctx *, int, uint64_t, int, int *);

// out = (kappa D_hop)^p psi on a domain in FP64 (Eq. HPEtr with the
// Dirichlet-restricted hopping term of Sec. 2): p pairs of plain hop launches
// (odd -> even, even -> odd) between two even-odd field pairs in block fixed point
// (each hop writes what the next one reads), kappa^p applied while unpacking.
// psi and out: device pointers.
int hop_power_fx(ddp_ctx *ctx, const Job &job, int p, const double *psi, double *out) {
    using P = PFX;
    if (p == 0) {
        DDP_CUDA(ctx, cudaMemcpyAsync(out, psi, (size_t)job.ncol * job.e[0] * job.e[1] * job.e[2] * job.e[3] * 12 * sizeof(double2),
                                      cudaMemcpyDeviceToDevice, ctx->stream));
        return DDP_OK;
    }
    std::vector<Job> jobs(1, job);
    Plan plan;
    make_plan(jobs, DDP_PREC_FP64, ctx->prm, plan);
    const int64_t NF = plan.nfield;
    size_t need = 4 * field_bytes<P>(NF) + sizeof(Item) + 1024;
    DDP_CUDA(ctx, ctx->scratch.reserve(need));
    Arena &a = ctx->scratch;
    a.reset();
    FieldView f[2][2] = {{carve_field<P>(a, NF), carve_field<P>(a, NF)}, {carve_field<P>(a, NF), carve_field<P>(a, NF)}};
    Item *d_items = (Item *)a.take(sizeof(Item));
    cudaStream_t st = ctx->stream;
    DDP_CUDA(ctx, cudaMemcpyAsync(d_items, plan.items.data(), sizeof(Item), cudaMemcpyHostToDevice, st));
    PackArgs pa;
    memset(&pa, 0, sizeof(pa));
    pa.it = plan.items[0];
    pa.user = (const double2 *)psi;
    pa.uout = (double2 *)out;
    const int64_t nt = 2 * (int64_t)pa.it.nh * pa.it.ncol;
    const unsigned nb = (unsigned)((nt + 255) / 256);
    k_pack_fx<<<nb, 256, 0, st>>>(pa, f[0][0], f[0][1]);
    const Launch L = make_launch(plan, d_items);
    FieldView none = {nullptr, nullptr, 0};
    HopArgs h;
    h.st = nullptr;
    h.skip = 0;
    h.L = L;
    h.v1 = none;
    h.v2 = none;
    h.rh = none;
    h.part.d = nullptr;
    int cur = 0;
    for (int k = 0; k < p; k++) {
        const int nxt = cur ^ 1;
        h.p = 0;
        h.in = f[cur][1];
        h.out = f[nxt][0];
        k_hop_fx<EPI_PLAIN, DOT_NONE, false, true><<<plan.nblocks * FX_SPLIT, HOP_TS * fx_cols(plan.CG), 0, st>>>(h);
        h.p = 1;
        h.in = f[cur][0];
        h.out = f[nxt][1];
        k_hop_fx<EPI_PLAIN, DOT_NONE, false, true><<<plan.nblocks * FX_SPLIT, HOP_TS * fx_cols(plan.CG), 0, st>>>(h);
        cur = nxt;
    }
    k_unpack_fx<<<nb, 256, 0, st>>>(pa, f[cur][0], f[cur][1], std::pow(job.kappa, p));
    ctx->launches += 2 + 2 * (long)p;
    DDP_CUDA(ctx, cudaGetLastError());
    return DDP_OK;
}
}  // namespace ddp
