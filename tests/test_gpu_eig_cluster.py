"""The cluster eigensolver of the mode Grams (pivoted Cholesky + one-sided Jacobi) at the edges of its blocks: orders
around multiples of the lanes of a pair, of the cluster and of its largest sizes, against the oracle's ST-HOSVD.

Bounds.  A Gram of ||Z|| = 1 carries rounding errors of about sqrt(M) u; a kept direction of size sigma moves by that
over sigma.  The smallest kept sigma is above eps / (2 M), so the truncated tensors agree to about
2 M^1.5 u / eps; ten times that is allowed, which stays below 1e-7 in FP64 for the eps here.  In FP32 the kernel works
on G less a Cholesky remainder of up to a hundredth of the budget eps^2 / 3, which turns a kept direction by at most a
hundredth of eps; eps / 50 is allowed on the tensor, beside the rounding term."""
import numpy as np
import pytest

from oracle import rounding, tucker
from tests.gpu_helpers import rel

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

U64 = 2.0 ** -53


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2306_00632_gb300 import api as a
    from paper_2306_00632_gb300 import lib
    lib.load()
    return a


def _tensor(n, ranks, fall, seed):
    """Factors of orthonormal columns (so Z is the core up to rotations), a core whose entries fall to `fall`."""
    g = np.random.default_rng(seed)
    w = [fall ** (np.arange(r) / max(r - 1, 1)) for r in ranks]
    core = g.standard_normal(ranks) * w[0][:, None, None] * w[1][None, :, None] * w[2][None, None, :]
    return core, [np.linalg.qr(g.standard_normal((n, r)))[0] for r in ranks]


def _gap_eps(Y, eps):
    """A tolerance near eps whose budget lies in the middle of a gap of every mode's tail energies."""
    (G, U) = Y
    Z = tucker.full(Y)
    tails = []
    for t in range(3):
        s = np.linalg.svd(np.moveaxis(Z, t, 0).reshape(Z.shape[t], -1), compute_uv=False)
        c = np.cumsum(s[::-1] ** 2) / np.sum(s ** 2)
        tails.append(np.log(c[c > 1e-28]))
    tails = np.concatenate(tails)
    e = eps * 1.5 ** np.linspace(-1, 1, 101)
    return float(e[np.argmax(np.abs(np.log(e * e / 3)[:, None] - tails[None]).min(1))])


@pytest.mark.parametrize("n,ranks", [(4, (1, 1, 1)), (6, (2, 3, 6)), (20, (15, 16, 17)), (34, (31, 33, 34)),
                                     (40, (40, 8, 3)), (66, (63, 17, 32)), (97, (97, 20, 20)), (128, (128, 64, 12)),
                                     (130, (129, 16, 24)), (200, (200, 15, 15)), (256, (256, 20, 13))])
def test_f64_edges(api, n, ranks):
    Y = _tensor(n, ranks, 1e-4, seed=n)
    eps = _gap_eps(Y, 1e-3)
    ref, inf = rounding.t_rel(Y, eps, return_info=True)
    y = api.Tucker.from_numpy(Y[0], Y[1], cap=n, core_cap=n * max(ranks) ** 2)
    ctx = api.Ctx(n, n, min(n, 256))
    info = torch.zeros(6, dtype=torch.float64, device="cuda")
    api.tucker_round(ctx, y, eps, info=info)
    G, U = y.to_numpy()
    assert G.shape == ref[0].shape
    M = max(ranks)
    assert rel(tucker.full((G, U)), tucker.full(ref)) <= 20 * M ** 1.5 * U64 / eps
    h = info.cpu().numpy()
    assert abs(h[1] - inf["discarded"]) <= 10 * M * U64 * inf["norm2"] + 1e-8 * inf["discarded"]
    for t in range(3):
        assert np.abs(U[t].T @ U[t] - np.eye(U[t].shape[1])).max() < 1e-11


def test_f64_strict_keeps_all(api):
    """eps = 0: nothing may be dropped, also directions far below what the Gram resolves."""
    n, ranks = 48, (40, 30, 20)
    Y = _tensor(n, ranks, 1e-9, seed=3)
    y = api.Tucker.from_numpy(Y[0], Y[1], cap=n, core_cap=n ** 3)
    ctx = api.Ctx(n, n, n)
    api.tucker_round(ctx, y, 0.0)
    G, U = y.to_numpy()
    assert G.shape == ranks
    assert rel(tucker.full((G, U)), tucker.full(Y)) <= 1e-14


def test_f64_strict_clipped_by_the_cap(api):
    """A strict truncation of a tensor of numerical rank 4 clipped to more columns than the Gram resolves: the
    completed basis is orthonormal and holds the tensor."""
    n, r, cap = 48, 40, 24
    core, U = _tensor(n, (r, r, r), 1.0, seed=5)
    small = np.full(core.shape, 1e-13)
    small[:4, :4, :4] = 1.0
    Y = (core * small, U)
    y = api.Tucker.from_numpy(Y[0], Y[1], cap=n, core_cap=n ** 3)
    ctx = api.Ctx(n, n, n)
    api.tucker_round(ctx, y, 0.0, rank_cap=cap)
    G, V = y.to_numpy()
    assert G.shape == (cap, cap, cap)
    assert rel(tucker.full((G, V)), tucker.full(Y)) <= 1e-10
    for t in range(3):
        assert np.abs(V[t].T @ V[t] - np.eye(cap)).max() < 1e-11


def test_f64_nan_stays_visible(api):
    n, ranks = 12, (5, 4, 3)
    core, U = _tensor(n, ranks, 1e-2, seed=9)
    core[0, 0, 0] = np.nan
    y = api.Tucker.from_numpy(core, U, cap=n, core_cap=n ** 3)
    ctx = api.Ctx(n, n, n)
    api.tucker_round(ctx, y, 1e-3)
    assert not np.isfinite(float(api.tucker_dot(ctx, y, y)))


@pytest.mark.parametrize("n,ranks", [(4, (1, 1, 1)), (6, (2, 3, 6)), (20, (15, 16, 17)), (34, (31, 33, 34)),
                                     (66, (63, 17, 32)), (97, (97, 20, 20)), (127, (127, 65, 12)),
                                     (128, (128, 24, 24))])
def test_f32_edges(api, n, ranks):
    Y = _tensor(n, ranks, 0.05, seed=n)
    Y = (Y[0].astype(np.float32).astype(float), [u.astype(np.float32).astype(float) for u in Y[1]])
    eps = _gap_eps(Y, 0.1)
    ref = rounding.t_rel(Y, eps)
    y = api.Tucker.from_numpy(Y[0], Y[1], cap=n, core_cap=n * max(ranks) ** 2, dtype=1)
    ctx = api.Ctx(n, n, n, dtype=1)
    api.tucker_round(ctx, y, eps)
    G, U = y.to_numpy()
    assert G.shape == ref[0].shape
    M = max(ranks)
    assert rel(tucker.full((G, U)), tucker.full(ref)) <= 20 * M ** 1.5 * 2.0 ** -24 / eps + eps / 50
    for t in range(3):
        assert np.abs(U[t].T @ U[t] - np.eye(U[t].shape[1])).max() < 1e-5
