"""The FP64 hopping term on the integer pipe against the FP64 oracle (GPU required).

The block fixed-point sums keep 2^-55 of the largest component of a site's neighbours, the
oracle's FP64 sums of 48 products about 48 * 2^-53 of it at the worst; with the epilogue's own
rounding an output component may differ by 64 * 2^-53 = 7.1e-15 of the largest neighbour
component, taken as 1e-14 here.
"""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
AP = oracle.BC_ANTIPERIODIC
LAT = (8, 4, 4, 6)
KAPPA = 0.1315
BOUND = 1e-14


@pytest.fixture(scope="module")
def env():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1601_04587_gb300 import build
    build.build()
    import paper_1601_04587_gb300 as ddp
    ctx = ddp.ddp_create(0, torch.cuda.current_stream().cuda_stream)
    U = synth.gauge_field(LAT, seed=4321)
    gid = ddp.ddp_load_gauge(ctx, torch.from_numpy(U).cuda(), LAT, ddp.DDP_BC_ANTIPERIODIC)
    yield ddp, ctx, U, gid
    ddp.ddp_destroy(ctx)


def _dirac(env, box, psi):
    ddp, ctx, _, gid = env
    did = ddp.ddp_set_domain(ctx, gid, *box)
    out = torch.zeros(psi.shape, dtype=torch.complex128, device="cuda")
    ddp.ddp_apply_dirac(ctx, did, KAPPA, torch.from_numpy(psi).cuda(), out, psi.shape[0], ddp.DDP_PREC_FP64)
    ddp.ddp_free_domain(ctx, did)
    return out.cpu().numpy()


# whole lattice; wrapped, odd extents (a ragged tile); two sites (seven hops dropped)
BOXES = [((0, 0, 0, 0), LAT), ((5, 1, 3, 2), (3, 2, 3, 4)), ((7, 3, 1, 5), (1, 1, 1, 2)), ((6, 0, 0, 0), (5, 4, 4, 6))]


@pytest.mark.parametrize("box", BOXES)
@pytest.mark.parametrize("ncol,step", [(1, 0), (3, 12), (13, -40)])
def test_dirac_over_a_dynamic_range(env, box, ncol, step):
    """Amplitudes 2^(step t): neighbours in time differ by the whole width of a limb and
    more; every component is held to the largest component next to it."""
    _, _, U, _ = env
    o, e = box
    n = int(np.prod(e))
    psi = synth.random_spinor(ncol, n, 17 + ncol)
    amp = 2.0 ** (step * np.arange(e[0]))
    t = np.arange(n) // (n // e[0])
    psi *= amp[t][None, :, None, None]
    got, want = _dirac(env, box, psi), oracle.apply_dirac(U, LAT, AP, o, e, KAPPA, psi)
    top = np.abs(psi).max(axis=(0, 2, 3)).reshape(e[0], -1).max(axis=1)
    near = np.maximum(top, np.maximum(np.roll(top, 1), np.roll(top, -1)))[t]
    err = np.abs(got - want).max(axis=(0, 2, 3)) / near
    assert err.max() < BOUND, err.max()


@pytest.mark.parametrize("scale", [0.0, 1e-300, 1e290])
def test_dirac_extreme_scales(env, scale):
    _, _, U, _ = env
    box = BOXES[1]
    psi = synth.random_spinor(2, int(np.prod(box[1])), 5) * scale
    got, want = _dirac(env, box, psi), oracle.apply_dirac(U, LAT, AP, *box, KAPPA, psi)
    assert np.abs(got - want).max() <= BOUND * np.abs(psi).max()


def _reached(U, box, mask):
    """The components one application of the hopping term makes depend on those of mask."""
    rng = np.random.default_rng(2)
    field = np.where(mask, rng.standard_normal(mask.shape) + 1j * rng.standard_normal(mask.shape), 0)
    return np.abs(oracle.hop_power(U, LAT, AP, *box, 1.0, 1, field)) > 1e-9


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("box", BOXES[:2])
def test_non_finite_components_spread_as_in_fp64(env, box, bad):
    """One non-finite component makes exactly the outputs non-finite that depend on it, in
    one application and in the second power of the hopping term; the others stay right."""
    ddp, ctx, U, gid = env
    n = int(np.prod(box[1]))
    clean = synth.random_spinor(3, n, 23)
    psi = clean.copy()
    psi[1, n // 2, 2, 1] = bad + 0.5j
    mask = ~np.isfinite(psi)
    got, want = _dirac(env, box, psi), oracle.apply_dirac(U, LAT, AP, *box, KAPPA, clean)
    hit = _reached(U, box, mask) | mask
    assert np.array_equal(~np.isfinite(got), hit)
    assert np.abs(got[~hit] - want[~hit]).max() < BOUND * np.abs(clean).max()
    did = ddp.ddp_set_domain(ctx, gid, *box)
    out = torch.zeros(psi.shape, dtype=torch.complex128, device="cuda")
    ddp.ddp_hop_power(ctx, did, KAPPA, 2, torch.from_numpy(psi).cuda(), out, 3)
    ddp.ddp_free_domain(ctx, did)
    hit = _reached(U, box, _reached(U, box, mask))
    assert np.array_equal(~np.isfinite(out.cpu().numpy()), hit)


def test_hop_power_zero_copies(env):
    ddp, ctx, _, gid = env
    psi = synth.random_spinor(2, int(np.prod(LAT)), 3)
    psi[0, 5, 1, 1] *= 1e-30
    did = ddp.ddp_set_domain(ctx, gid, (0, 0, 0, 0), LAT)
    out = torch.zeros(psi.shape, dtype=torch.complex128, device="cuda")
    ddp.ddp_hop_power(ctx, did, KAPPA, 0, torch.from_numpy(psi).cuda(), out, 2)
    ddp.ddp_free_domain(ctx, did)
    assert np.array_equal(out.cpu().numpy(), psi)
