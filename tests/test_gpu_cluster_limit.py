"""The shapes that stand in where a device has no clusters of 16 CTAs (TPCG_OPT_CLUSTER 8): truncations with Grams above
order 64 and factors above 128 rows, and scalar products of small contexts.

Bounds as for the other shapes: nothing is discarded at eps = 1e-6, so the tensor stays within eps; kept factors are
orthonormal to 1e-11 (FP32 1e-5) beside 20 k u of the QR; scalar products round by about (5 n + 3) u of the norms."""
import numpy as np
import pytest

import synth
from oracle import tucker
from tests.graph_helpers import kernels
from tests.gpu_helpers import rel

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def mods():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2306_00632_gb300 import api, lib
    lib.load()
    yield api, lib
    api.set_option(lib.OPT_CLUSTER, 16)


@pytest.mark.parametrize("limit", [8, 16])
@pytest.mark.parametrize("n,ranks,dtype", [(65, (65, 20, 9), 0), (97, (97, 50, 20), 0), (128, (128, 127, 3), 0), (129, (60, 129, 7), 0),
                                           (200, (200, 90, 12), 0), (256, (256, 11, 33), 0), (257, (90, 40, 30), 1),
                                           (300, (90, 60, 20), 0)])
def test_truncation(mods, n, ranks, dtype, limit):
    api, lib = mods
    g = np.random.default_rng(n)
    core = g.standard_normal(ranks)
    U = [np.linalg.qr(g.standard_normal((n, r)))[0] @ np.linalg.qr(g.standard_normal((r, r)))[0] for r in ranks]
    ctx = api.Ctx(n, n, 96 if n > 256 else n, dtype=dtype)
    api.set_option(lib.OPT_CLUSTER, limit)

    def call():
        api.tucker_round(ctx, y, eps)

    eps = 1e-3 if dtype else 1e-6
    y = api.Tucker.from_numpy(core, U, cap=n, core_cap=int(np.prod(ranks)), dtype=dtype)
    call()
    G, V = y.to_numpy()
    u = 2.0 ** -24 if dtype else 2.0 ** -53
    for v in V:
        assert np.abs(v.T @ v - np.eye(v.shape[1])).max() < 20 * max(ranks) * u + (1e-5 if dtype else 1e-11)
    for t in range(3):
        G = np.moveaxis(np.tensordot(U[t].T @ V[t], G, (1, t)), 0, t)
    assert rel(G, core) <= eps
    largest = max(c for *_, c in kernels(call))   # (FP32 above n = 256 has one-CTA kernels only in place of 16)
    assert largest == 16 if limit == 16 else largest <= 8


@pytest.mark.parametrize("limit", [8, 16])
@pytest.mark.parametrize("dtype", [0, 1])
def test_scalar_product(mods, dtype, limit):
    api, lib = mods
    n = 40
    X = synth.random_tucker((n, n, n), (31, 6, 17), seed=1)
    Y = synth.random_tucker((n, n, n), (8, 32, 5), seed=2)
    x, y = (api.Tucker.from_numpy(T[0], T[1], dtype=dtype) for T in (X, Y))
    ctx = api.Ctx(n, n, 32, dtype=dtype)
    api.set_option(lib.OPT_CLUSTER, limit)
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    assert max(c for *_, c in kernels(lambda: api.tucker_dot(ctx, x, y, out=out))) == limit
    u = 2.0 ** -24 if dtype else 2.0 ** -53
    assert abs(api.tucker_dot(ctx, x, y).item() - tucker.dot(X, Y)) <= (5 * n + 3) * u * tucker.norm(X) * tucker.norm(Y)


def test_other_values_are_refused(mods):
    api, lib = mods
    for v in (0, 4, 12, 32):
        with pytest.raises(lib.TpcgError):
            api.set_option(lib.OPT_CLUSTER, v)
