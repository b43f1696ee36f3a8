"""Small domains of several cluster sizes beside one another and beside larger ones (GPU required):
each request has the bits it has alone, and a batch is not slower than by the per-step kernels."""
import time

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
LAT = (16, 16, 16, 16)
# clusters of 1 to 8 blocks, and a domain beyond them
BOXES = [(4, 4, 4, 4), (8, 4, 4, 4), (4, 4, 6, 8), (8, 8, 4, 4), (10, 4, 4, 8), (6, 4, 8, 8), (7, 4, 8, 8), (8, 8, 8, 4)]
LARGE = (8, 8, 8, 8)
KAPPA = 0.13


@pytest.fixture(scope="module")
def env():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1601_04587_gb300 as ddp
    ctx = ddp.ddp_create(0, torch.cuda.current_stream().cuda_stream)
    gid = ddp.ddp_load_gauge(ctx, torch.from_numpy(synth.gauge_field(LAT, seed=6)).cuda(), LAT, ddp.DDP_BC_ANTIPERIODIC)
    yield ddp, ctx, gid
    ddp.ddp_destroy(ctx)


def _reqs(env, boxes):
    ddp, ctx, gid = env
    out, reqs = [], []
    for i, e in enumerate(boxes):
        did = ddp.ddp_set_domain(ctx, gid, (i, 0, 2 * i, 0), e)
        S = torch.zeros((12, int(np.prod(e)), 4, 3), dtype=torch.complex128, device="cuda")
        out.append(S)
        src = tuple((o + x // 2) % 16 for o, x in zip((i, 0, 2 * i, 0), e))
        reqs.append(ddp.make_req(did, KAPPA, src, 1e-10, S))
    return reqs, out


@pytest.fixture(scope="module")
def alone(env):
    ddp, ctx, _ = env
    reqs, out = _reqs(env, BOXES + [LARGE])
    for r in reqs:
        rc, _ = ddp.ddp_solve_batch(ctx, [r], 1)
        assert rc == ddp.DDP_OK
    return [S.clone() for S in out]


@pytest.mark.parametrize("boxes", [[0, 1], [7, 0, 3], list(range(8)), [8, 0], [2, 8, 5, 1], list(range(9))])
def test_batch_of_several_sizes_has_the_bits_of_each_alone(env, alone, boxes):
    ddp, ctx, _ = env
    every = BOXES + [LARGE]
    reqs, out = _reqs(env, every)
    for _ in range(3):
        for k in boxes:
            out[k].zero_()
        rc, _ = ddp.ddp_solve_batch(ctx, [reqs[k] for k in boxes], 1)
        assert rc == ddp.DDP_OK
        for k in boxes:
            assert torch.equal(out[k], alone[k])


def test_server_with_several_sizes_has_the_bits_of_each_alone(env, alone):
    ddp, ctx, _ = env
    reqs, out = _reqs(env, BOXES + [LARGE])
    ddp.ddp_serve_config(ctx, 1 << 30, 16, 1)
    tickets = []
    for k in (8, 3, 0, 7, 1):                # the others join while these are in flight
        rc, t = ddp.ddp_submit(ctx, reqs[k])
        assert rc == ddp.DDP_OK
        tickets.append(t)
    ddp.ddp_serve_step(ctx)
    for k in (2, 4, 5, 6):
        rc, t = ddp.ddp_submit(ctx, reqs[k])
        assert rc == ddp.DDP_OK
        tickets.append(t)
    while ddp.ddp_serve_step(ctx):
        pass
    assert all(ddp.ddp_poll(ctx, t)[0] for t in tickets)
    ddp.ddp_serve_reset(ctx)
    for S, ref in zip(out, alone):
        assert torch.equal(S, ref)


@pytest.mark.parametrize("large", [False, True])
def test_batch_of_several_sizes_is_not_slower_than_the_per_step_kernels(env, large):
    """Nine requests of 12 columns: 1.35 and 2.78 ms beside one another, 1.9 and 2.7 by the per-step
    kernels; one group after another they took 3.5 and 5.3."""
    ddp, ctx, _ = env
    reqs, _ = _reqs(env, BOXES + ([LARGE] if large else []))

    def ms(sites):
        ddp.ddp_set_param(ctx, "small_domain_sites", sites)
        best = 1e9
        try:
            for _ in range(8):
                torch.cuda.synchronize()
                t = time.perf_counter()
                ddp.ddp_solve_batch(ctx, reqs, 1)
                best = min(best, time.perf_counter() - t)
        finally:
            ddp.ddp_set_param(ctx, "small_domain_sites", 1024)
        return best

    assert ms(1024) < 1.25 * ms(0)
