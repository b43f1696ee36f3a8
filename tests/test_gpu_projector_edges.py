"""Gram blocks and colourless spinors on the tensor cores at the edges of their tiles: column counts
next to 32 (where real and imaginary parts stop sharing a tile), 64 and 128, rows that end within a
16-deep reduction step, columns that read beyond the stored rows, and non-finite columns."""
import numpy as np
import pytest

import oracle
import synth
from oracle import projector

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

L = (6, 4, 4, 4)
# Each operand is cut to 2^-49 of its column (row) maximum and slice products below 2^-47 of the
# product of the maxima are dropped; with maxima up to 5 times the rms value of random fields the
# norm-wise error is below 25 * 2^-46 = 4e-13.
TOL = 1e-12


@pytest.fixture(scope="module")
def env():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1601_04587_gb300 as ddp
    ctx = ddp.ddp_create(0, torch.cuda.current_stream().cuda_stream)
    gid = ddp.ddp_load_gauge(ctx, torch.from_numpy(synth.gauge_field(L, seed=5)).cuda(), L, ddp.DDP_BC_ANTIPERIODIC)
    yield ddp, ctx, gid
    ddp.ddp_destroy(ctx)


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("bad", [False, True])
@pytest.mark.parametrize("m", [31, 32, 33, 63, 64, 65, 72, 127])
@pytest.mark.parametrize("box", [((0, 0, 0, 0), (2, 4, 4, 4)), ((1, 1, 0, 2), (2, 3, 1, 2)), ((5, 0, 0, 0), (1, 1, 1, 2))])
def test_gram_blocks_at_tile_edges(env, m, box, bad):
    ddp, ctx, gid = env
    n = oracle.box_sites(box[1])
    A = synth.random_spinor(m, n, 300 + m)
    if bad:
        A[m - 2, n - 1, 1, 2] = complex(0.0, np.inf)
    did = ddp.ddp_set_domain(ctx, gid, *box)
    M = torch.zeros((L[0], m, m), dtype=torch.complex128, device="cuda")
    ddp.ddp_gram_slices(ctx, did, torch.from_numpy(A).cuda(), m, M)
    ddp.ddp_free_domain(ctx, did)
    got = M.cpu().numpy()
    if bad:
        A[m - 2, n - 1, 1, 2] = 0.0
        last = (box[0][0] + box[1][0] - 1) % L[0]
        assert np.isnan(got[last, m - 2]).all() and np.isnan(got[last, :, m - 2]).all()
        got[last, m - 2] = got[last, :, m - 2] = 0.0
    want = projector.gram_slices(L, *box, A)
    if bad:
        want[last, m - 2] = want[last, :, m - 2] = 0.0
    assert _rel(got, want) < TOL


@pytest.mark.parametrize("form", [0, 1, 2])
@pytest.mark.parametrize("m,box", [(7, ((1, 1, 0, 2), (2, 3, 1, 2))), (17, ((5, 0, 0, 0), (2, 1, 1, 2))),
                                   (33, ((0, 0, 0, 0), (1, 1, 3, 2)))])
def test_colourless_spinors_at_tile_edges(env, m, box, form):
    ddp, ctx, gid = env
    A = synth.random_spinor(m, oracle.box_sites(box[1]), 400 + m)
    did = ddp.ddp_set_domain(ctx, gid, *box)
    X = torch.zeros((L[0], m, m, m, 4), dtype=torch.complex128, device="cuda")
    ddp.ddp_colourless_slices(ctx, did, torch.from_numpy(A).cuda(), m, form, X)
    ddp.ddp_free_domain(ctx, did)
    g5 = oracle.gamma()[4]
    s = {0: A, 1: np.einsum("ab,mnbc->mnac", g5, np.conj(A)), 2: -A}[form]
    assert _rel(X.cpu().numpy(), projector.colourless_spinors(L, *box, s)) < TOL


@pytest.mark.parametrize("m", [5, 33])      # one shared tile, and cross products
def test_gram_of_subnormal_columns_with_large_ones(env, m):
    """Columns of subnormals, of all sizes and below 2^-1042 only, against one of size 1e150: their
    products are ordinary numbers."""
    ddp, ctx, gid = env
    box = ((0, 0, 0, 0), (2, 4, 4, 4))
    n = oracle.box_sites(box[1])
    A = synth.random_spinor(m, n, 77)
    rng = np.random.default_rng(1)
    for c, bits in ((0, 52), (1, 30)):
        k = rng.integers(-(1 << bits) + 1, 1 << bits, size=(2,) + A[c].shape).astype(np.float64)
        A[c] = k[0] * 5e-324 + 1j * (k[1] * 5e-324)
    A[2] *= 1e150
    did = ddp.ddp_set_domain(ctx, gid, *box)
    M = torch.zeros((L[0], m, m), dtype=torch.complex128, device="cuda")
    ddp.ddp_gram_slices(ctx, did, torch.from_numpy(A).cuda(), m, M)
    ddp.ddp_free_domain(ctx, did)
    got = M.cpu().numpy()
    B = A.copy()
    B[:2] *= 2.0 ** 1000                    # exact
    for t in range(2):
        rows = slice(64 * t, 64 * (t + 1))
        for c in (0, 1):
            x, y = B[c, rows].reshape(-1), B[2, rows].reshape(-1)
            want = np.vdot(x, y)
            size = np.linalg.norm(x) * np.linalg.norm(y)
            assert abs(got[t, c, 2] * 2.0 ** 1000 - want) < TOL * size
            assert abs(got[t, 2, c] * 2.0 ** 1000 - np.conj(want)) < TOL * size
