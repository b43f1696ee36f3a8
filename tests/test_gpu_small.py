"""Small domains solved on chip (one kernel per correction cycle) against the per-step kernels
and the FP64 oracle (GPU required).

Both paths stop on the same FP64 true residual, 1e-10, so their columns agree with the oracle's
(solved to 1e-12) to the solver tolerance times the conditioning of these well-conditioned boxes:
the 1e-8 of the other propagator tests.
"""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
AP = oracle.BC_ANTIPERIODIC
LAT = (12, 8, 8, 10)
KAPPA = 0.12
COL_TOL = 1e-8


@pytest.fixture(scope="module")
def env():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1601_04587_gb300 import build
    build.build()
    import paper_1601_04587_gb300 as ddp
    ctx = ddp.ddp_create(0, torch.cuda.current_stream().cuda_stream)
    U = synth.gauge_field(LAT, seed=99)
    gid = ddp.ddp_load_gauge(ctx, torch.from_numpy(U).cuda(), LAT, ddp.DDP_BC_ANTIPERIODIC)
    yield ddp, ctx, U, gid
    ddp.ddp_destroy(ctx)


def _solve(env, box, eta, prec, small):
    ddp, ctx, _, gid = env
    did = ddp.ddp_set_domain(ctx, gid, *box)
    psi = torch.zeros(eta.shape, dtype=torch.complex128, device="cuda")
    ddp.ddp_set_param(ctx, "small_domain_sites", 1024 if small else 0)
    before = ddp.ddp_kernel_launches(ctx)
    try:
        rc, info = ddp.ddp_solve_sources(ctx, did, KAPPA, 0.0, torch.from_numpy(eta).cuda(), eta.shape[0], 1e-10, prec, psi)
    finally:
        ddp.ddp_set_param(ctx, "small_domain_sites", 1024)
        ddp.ddp_free_domain(ctx, did)
    assert rc == ddp.DDP_OK, ddp.info_dict(info)
    assert info.max_rel_residual <= 1e-10
    return psi.cpu().numpy(), ddp.ddp_kernel_launches(ctx) - before


# one site per parity; one block with and without free slots (128 sites per parity, 129 in two
# blocks); unrestricted directions, wrapped and across the antiperiodic boundary; odd extents cut
# unevenly; eight blocks and the first size beyond the path (1024 and 1050 sites per parity)
BOXES = [((7, 3, 1, 5), (1, 1, 1, 2)), ((0, 0, 0, 0), (4, 4, 4, 4)), ((10, 6, 5, 8), (4, 8, 2, 4)),
         ((11, 0, 0, 3), (3, 1, 3, 10)), ((1, 2, 3, 4), (7, 5, 3, 6)), ((9, 0, 0, 0), (5, 8, 8, 4)), ((3, 1, 0, 2), (3, 6, 7, 2)),
         ((2, 7, 0, 9), (8, 8, 8, 4)), ((6, 1, 2, 0), (5, 7, 6, 10)), ((0, 0, 0, 0), (12, 2, 4, 10))]


@pytest.mark.parametrize("box", BOXES)
@pytest.mark.parametrize("ncol", [1, 3])
def test_small_against_per_step_and_oracle(env, box, ncol):
    _, _, U, _ = env
    n = int(np.prod(box[1]))
    eta = synth.random_spinor(ncol, n, 7 + ncol)
    on, launches_on = _solve(env, box, eta, 1, True)
    off, launches_off = _solve(env, box, eta, 1, False)
    ref, *_ = oracle.solve(U, LAT, AP, *box, KAPPA, eta, tol=1e-12)
    for c in range(ncol):
        norm = np.linalg.norm(ref[c])
        assert np.linalg.norm(on[c] - ref[c]) < COL_TOL * norm
        assert np.linalg.norm(off[c] - ref[c]) < COL_TOL * norm
    if n // 2 <= 1024:
        assert launches_on < launches_off   # it took the one-kernel path
    else:
        assert np.array_equal(on, off)


@pytest.mark.parametrize("prec", [2, 3])
@pytest.mark.parametrize("box", [BOXES[4], BOXES[6]])
def test_small_16_bit_formats(env, prec, box):
    _, _, U, _ = env
    eta = synth.random_spinor(2, int(np.prod(box[1])), 31)
    got, _ = _solve(env, box, eta, prec, True)
    ref, *_ = oracle.solve(U, LAT, AP, *box, KAPPA, eta, tol=1e-12)
    assert max(np.linalg.norm(got[c] - ref[c]) / np.linalg.norm(ref[c]) for c in range(2)) < COL_TOL


def test_small_and_large_in_one_batch(env):
    """Cluster sizes 1 to 8 and a domain beyond them in one batch, in mixed order, with a zero
    column: each result has the bits of the same request alone."""
    ddp, ctx, _, gid = env
    reqs, outs, alone, dids = [], [], [], []
    for i, box in enumerate([BOXES[7], BOXES[1], BOXES[6], BOXES[0], BOXES[5], BOXES[4]]):
        n = int(np.prod(box[1]))
        did = ddp.ddp_set_domain(ctx, gid, *box)
        dids.append(did)
        ncol = 1 + 2 * i
        eta = synth.random_spinor(ncol, n, 50 + i)
        if i == 2:
            eta[1] = 0
        eta = torch.from_numpy(eta).cuda()
        out, one = torch.zeros_like(eta), torch.zeros_like(eta)
        reqs.append(ddp.make_req(did, KAPPA, tol=1e-10, out=out, eta=eta, ncol=ncol))
        outs.append((out, eta))
        rc, _ = ddp.ddp_solve_sources(ctx, did, KAPPA, 0.0, eta, ncol, 1e-10, 1, one)
        assert rc == ddp.DDP_OK
        alone.append(one)
    rc, infos = ddp.ddp_solve_batch(ctx, reqs, 1)
    assert rc == ddp.DDP_OK
    for d in dids:
        ddp.ddp_free_domain(ctx, d)
    for (out, _), one, info, r in zip(outs, alone, infos, reqs):
        assert info.ncol == r.ncol
        assert torch.equal(out, one)
    assert not outs[2][0][1].any()


def test_small_iteration_cap_and_parameter(env):
    ddp, ctx, _, gid = env
    box = BOXES[1]
    eta = torch.from_numpy(synth.random_spinor(2, int(np.prod(box[1])), 3)).cuda()
    psi = torch.zeros_like(eta)
    did = ddp.ddp_set_domain(ctx, gid, *box)
    ddp.ddp_set_param(ctx, "max_inner", 2)
    ddp.ddp_set_param(ctx, "max_outer", 1)
    try:
        rc, info = ddp.ddp_solve_sources(ctx, did, KAPPA, 0.0, eta, 2, 1e-10, 1, psi)
    finally:
        ddp.ddp_set_param(ctx, "max_inner", 30000)
        ddp.ddp_set_param(ctx, "max_outer", 40)
        ddp.ddp_free_domain(ctx, did)
    assert rc == ddp.DDP_ERR_NOT_CONVERGED and info.inner_iters == 2
    assert torch.isfinite(torch.view_as_real(psi)).all()
    assert ddp.ddp_get_param(ctx, "small_domain_sites") == 1024
    for bad in (-1, 1025):
        with pytest.raises(ddp.DDPError):
            ddp.ddp_set_param(ctx, "small_domain_sites", bad)
