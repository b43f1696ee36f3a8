"""FP64 stencil calls and the server at the limit of the memory they are given (GPU required).

The block fixed-point field of the FP64 hopping term comes on top of the four FP64 fields of a call
(768 bytes per site-column); where only those fit the columns are taken in parts."""
import math

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
LAT = (16, 16, 16, 16)
N = math.prod(LAT)
NCOL = 48
FIELDS = 768 * (N // 2) * NCOL


@pytest.fixture(scope="module")
def ddp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1601_04587_gb300 as m
    return m


def _context(ddp):
    ctx = ddp.ddp_create(0, torch.cuda.current_stream().cuda_stream)
    U = torch.eye(3, dtype=torch.complex128, device="cuda").expand(4, N, 3, 3)
    gid = ddp.ddp_load_gauge(ctx, U.contiguous(), LAT, ddp.DDP_BC_ANTIPERIODIC)
    return ctx, gid, ddp.ddp_set_domain(ctx, gid, (0, 0, 0, 0), LAT)


@pytest.mark.parametrize("call", ["dirac", "power"])
def test_fp64_stencil_calls_where_four_fields_fit(ddp, call):
    g = torch.Generator(device="cuda").manual_seed(4)
    psi = torch.complex(*[torch.randn((NCOL, N, 4, 3), dtype=torch.float64, device="cuda", generator=g) for _ in range(2)])
    out, want = torch.zeros_like(psi), torch.zeros_like(psi)

    def run(ctx, did, to, ncol=NCOL):
        if call == "dirac":
            ddp.ddp_apply_dirac(ctx, did, 0.13, psi, to, ncol)
        else:
            ddp.ddp_hop_power(ctx, did, 0.13, 2, psi, to, ncol)

    ctx, _, did = _context(ddp)
    run(ctx, did, want)
    ddp.ddp_destroy(ctx)
    ctx, _, did = _context(ddp)
    run(ctx, did, out, 1)                      # kernels and their stacks are resident
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    fill = torch.empty(free - FIELDS - (8 << 20), dtype=torch.uint8, device="cuda")
    try:
        run(ctx, did, out)
    finally:
        del fill
        torch.cuda.empty_cache()
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    run(ctx, did, out.zero_())                 # nothing is left over from the refused allocation
    assert torch.equal(out, want)
    ddp.ddp_destroy(ctx)


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
def test_server_holds_what_its_budget_pays_for(ddp, prec):
    """Capacity is the budget over the bytes of a site-column: six FP64 fields, nine of the storage
    format (the shadow residual of FP32 counted in full), and 48 bytes of partial sums a 32-site tile."""
    ctx, gid, _ = _context(ddp)
    stored = {0: 192, 1: 96, 2: 52, 3: 48}[prec]
    did = ddp.ddp_set_domain(ctx, gid, (0, 0, 0, 0), (8, 16, 16, 16))
    out = torch.zeros((12, N // 2, 4, 3), dtype=torch.complex128, device="cuda")
    req = ddp.make_req(did, 0.12, (4, 8, 8, 8), 1e-8, out)
    length = N // 4 * 12
    per = 6 * 192 + 9 * stored + 1.5
    ddp.ddp_serve_config(ctx, int(length * (per + 0.25)), 2, prec)
    rc, ticket = ddp.ddp_submit(ctx, req)
    assert rc == ddp.DDP_OK
    while ddp.ddp_serve_step(ctx):
        pass
    done, info = ddp.ddp_poll(ctx, ticket)
    assert done and info.status == ddp.DDP_OK
    ddp.ddp_serve_reset(ctx)
    ddp.ddp_destroy(ctx)
