"""Kept factors stay orthonormal where the singular values of a mode nearly coincide: triples within 1e-2 to 1e-13 of each
other, orders on every shape of the eigensolvers.

The tensor is a superdiagonal core of those values turned by orthogonal matrices in every mode, so that the mode Grams are
dense, with factors of orthonormal columns.  Nothing is discarded.

Bounds.  The last sweep leaves cosines of at most tau (1e-14; FP32 5e-7) and, from wide turns, twice the largest remaining
cosine times the largest tan(theta / 2) it allows: 2e-14 (FP32 9e-6).  The QR of k columns and the product with it round by
about 20 k u (FP64) and, FP32 sums over the lanes of a warp, 2 k u."""
import numpy as np
import pytest

from tests.gpu_helpers import rel

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2306_00632_gb300 import api as a
    from paper_2306_00632_gb300 import lib
    lib.load()
    return a


def _tensor(n, k, gap, g):
    m = (k + 2) // 3
    s = np.repeat(0.1 ** (np.arange(m) / max(m - 1, 1)), 3)[:k]
    s = s * (1 + gap * g.uniform(0, 1, k) * 10.0 ** g.uniform(-3, 0, k))
    core = np.zeros((k, k, k))
    core[np.arange(k), np.arange(k), np.arange(k)] = s
    for t in range(3):
        w = np.linalg.qr(g.standard_normal((k, k)))[0]
        core = np.moveaxis(np.tensordot(w, core, (1, t)), 0, t)
    return core, [np.linalg.qr(g.standard_normal((n, k)))[0] for _ in range(3)]


def _worst(api, n, k, gap, dtype, draws, eps):
    g = np.random.default_rng(1000 * n + k)
    ctx = api.Ctx(n, n, min(n, 96) if dtype == 0 and n > 256 else n, dtype=dtype)
    worst = 0.0
    for _ in range(draws):
        Y = _tensor(n, k, gap, g)
        y = api.Tucker.from_numpy(Y[0], Y[1], cap=n, core_cap=k ** 3, dtype=dtype)
        api.tucker_round(ctx, y, eps)
        G, U = y.to_numpy()
        assert G.shape == (k, k, k)
        worst = max([worst] + [np.abs(u.T @ u - np.eye(k)).max() for u in U])
    # compared in the last draw's own factors: |full(Y) - full(G, U)| without the full tensors
    C = [u.T @ v for u, v in zip(Y[1], U)]
    back = G
    for t in range(3):
        back = np.moveaxis(np.tensordot(C[t], back, (1, t)), 0, t)
    assert rel(back, Y[0]) <= eps
    return worst


@pytest.mark.parametrize("gap", [1e-4, 1e-9])
@pytest.mark.parametrize("n,k,draws", [(9, 9, 100), (32, 24, 40), (64, 48, 20), (97, 60, 12), (200, 80, 8)])
def test_f64(api, n, k, gap, draws):
    assert _worst(api, n, k, gap, 0, draws, 1e-6) <= 1e-13 + 20 * k * 2.0 ** -53


@pytest.mark.parametrize("gap", [1e-2, 1e-4, 1e-6])
@pytest.mark.parametrize("n,k,draws", [(9, 9, 60), (32, 24, 40), (97, 48, 20), (128, 72, 12)])
def test_f32(api, n, k, gap, draws):
    assert _worst(api, n, k, gap, 1, draws, 1e-3) <= 1e-5 + 2 * k * 2.0 ** -24


@pytest.mark.parametrize("gap", [1e-2, 1e-4, 1e-6])
@pytest.mark.parametrize("n,k,draws", [(130, 24, 40), (160, 48, 20), (160, 96, 12)])
def test_f32_large_contexts(api, n, k, gap, draws):
    """Contexts above n = 128, whose FP32 Grams and Ritz matrices have an eigensolver of their own (tau 2e-6)."""
    assert _worst(api, n, k, gap, 1, draws, 1e-3) <= 1.2e-5 + 2 * k * 2.0 ** -24
