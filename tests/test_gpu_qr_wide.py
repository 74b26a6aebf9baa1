"""The QR of the factors where its warps hold two columns (more columns than the cluster has warps), and where a factor's
squares leave the exponent's range: one mode's factor is scaled down, the core up by the inverse, so that the tensor is
representable.

Bounds: as for Householder reflectors at other sizes, U^T U within 20 k u + 1e-11 (FP64; FP32 1e-5) of the identity and the
tensor within eps + 20 k u."""
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


def _input(n, ks, seed):
    g = np.random.default_rng(seed)
    U = [g.standard_normal((n, k)) / np.sqrt(n) for k in ks]
    w = [0.8 ** np.arange(k) for k in ks]
    core = g.standard_normal(ks) * w[0][:, None, None] * w[1][None, :, None] * w[2][None, None, :]
    return core, U


def _times(core, mats):
    for t, a in enumerate(mats):
        core = np.moveaxis(np.tensordot(a, core, (1, t)), 0, t)
    return core


def _check(api, n, ks, dtype, scale, mode):
    core, U = _input(n, ks, seed=n + mode)
    V = [u * (scale if t == mode else 1.0) for t, u in enumerate(U)]
    y = api.Tucker.from_numpy(core / scale, V, cap=max(ks), core_cap=int(np.prod(ks)), dtype=dtype)
    ctx = api.Ctx(n, n, min(n, 96), dtype)
    eps = 3e-3 if dtype else 1e-6
    api.tucker_round(ctx, y, eps)
    G, W = y.to_numpy()
    u = 2.0 ** -24 if dtype else 2.0 ** -53
    k = max(ks)
    for w in W:
        assert np.abs(w.T @ w - np.eye(w.shape[1])).max() < 20 * k * u + (1e-5 if dtype else 1e-11)
    # compared in bases of the factors of both tensors
    B = [np.linalg.qr(np.hstack([a, b]))[0] for a, b in zip(U, W)]
    got = _times(G, [b.T @ w for b, w in zip(B, W)])
    want = _times(core, [b.T @ a for b, a in zip(B, U)])
    assert rel(got, want) <= eps + 20 * k * u


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("n,ks", [(200, (130, 12, 60)), (256, (200, 30, 255)), (300, (299, 257, 9)), (512, (300, 12, 40)),
                                  (512, (20, 511, 8))])
def test_two_columns_a_warp(api, n, ks, dtype):
    _check(api, n, ks, dtype, 1.0, 0)


@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("dtype,scale", [(0, 1e-150), (0, 1e-170), (1, 1e-17), (1, 1e-25)])
@pytest.mark.parametrize("n,ks", [(24, (20, 9, 7)), (97, (60, 33, 50)), (256, (70, 40, 20))])
def test_tiny_factor(api, n, ks, dtype, scale, mode):
    _check(api, n, ks, dtype, scale, mode)
