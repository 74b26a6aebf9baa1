"""The QR of the factors at the edges of its shapes (rows per lane, columns per warp, CTAs per mode): a truncation of a
tensor whose factors have fewer columns than rows keeps orthonormal factors and, up to its tolerance, the tensor.
Factors are random, nearly dependent (the second half of the columns repeats the first up to 1e-9) or tiny.

Bound: Householder reflectors are orthogonal to a few u each; k of them and the eigenvectors leave U^T U within
20 k u + 1e-11 (FP64) or 1e-5 (FP32) of the identity and the tensor within eps + 20 k u."""
import numpy as np
import pytest

from oracle import tucker
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


def _input(n, ks, kind, seed):
    g = np.random.default_rng(seed)
    U = []
    for k in ks:
        u = g.standard_normal((n, k)) / np.sqrt(n)
        if kind == "dependent" and k > 1:
            h = k // 2
            u[:, k - h:] = u[:, :h] + 1e-9 * u[:, k - h:]
        if kind == "tiny":
            u *= 1e-17
        U.append(u)
    w = [0.8 ** np.arange(k) for k in ks]
    core = g.standard_normal(ks) * w[0][:, None, None] * w[1][None, :, None] * w[2][None, None, :]
    return core, U


@pytest.mark.parametrize("kind", ["random", "dependent", "tiny"])
@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("n,ks", [(2, (1, 1, 1)), (33, (32, 31, 1)), (32, (17, 31, 2)), (64, (63, 33, 5)), (65, (64, 3, 9)),
                                  (128, (127, 97, 33)), (129, (120, 65, 3)), (256, (100, 65, 33)), (300, (90, 12, 17))])
def test_qr_edges(api, n, ks, dtype, kind):
    Y = _input(n, ks, kind, seed=n)
    y = api.Tucker.from_numpy(Y[0], Y[1], cap=max(ks), core_cap=int(np.prod(ks)), dtype=dtype)
    cap = min(n, 128)
    ctx = api.Ctx(n, n, cap, dtype)
    eps = 3e-3 if dtype else 1e-6
    api.tucker_round(ctx, y, eps)
    G, U = y.to_numpy()
    u = 2.0 ** -24 if dtype else 2.0 ** -53
    scale = [1e17 if kind == "tiny" else 1.0] * 3   # (the products of three tiny factors leave FP32's range)
    want = tucker.full((Y[0], [a * s for a, s in zip(Y[1], scale)]))
    if kind == "tiny" and dtype == 1:
        assert G.size == 0   # a zero tensor in FP32: no NaN has made it anything else
        return
    for t in range(3):
        assert np.abs(U[t].T @ U[t] - np.eye(U[t].shape[1])).max() < 20 * max(ks) * u + (1e-5 if dtype else 1e-11)
    if kind != "tiny":
        assert rel(tucker.full((G, U)), want) <= eps + 20 * max(ks) * u
    else:
        assert rel(tucker.full((G * 1e51, U)), want) <= eps + 20 * max(ks) * u
