"""The plain FP64 rule at a tolerance whose budget is below what rounding leaves of the Gram outside the Cholesky columns:
nothing can be discarded then, so the directions far below the budget are kept, and kept factors are orthonormal.

The tensor has a block of rows of lower rank (its Gram's rounding noise is the remainder, about u times the trace, against a
budget of 1e-18 times it) and a block whose singular values are 1e-12 of the others.

Bounds: orthonormal to tau = 1e-14 and the roundings of products of n terms, 20 n u."""
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
    a.set_option(lib.OPT_ROUND_RULE, 0)
    yield a
    a.set_option(lib.OPT_ROUND_RULE, -1)


@pytest.mark.parametrize("n,rank,small", [(24, 5, 8), (32, 6, 8), (64, 12, 10), (97, 20, 17), (160, 20, 12)])
def test_kept_columns_below_the_budget_are_orthonormal(api, n, rank, small):
    g = np.random.default_rng(n)
    big = n - small
    s = np.zeros(n)
    s[:rank] = g.uniform(0.5, 1.0, rank)
    s[big:] = 1e-12 * g.uniform(0.5, 1.0, small)
    core = np.zeros((n, n, n))
    core[np.arange(n), np.arange(n), np.arange(n)] = s
    U = []
    for _ in range(3):
        u = np.zeros((n, n))
        u[:big, :big] = np.linalg.qr(g.standard_normal((big, big)))[0]
        u[big:, big:] = np.linalg.qr(g.standard_normal((small, small)))[0]
        U.append(u)
    y = api.Tucker.from_numpy(core, U, cap=n, core_cap=n ** 3)
    ctx = api.Ctx(n, n, n)
    api.tucker_round(ctx, y, 2e-9)
    G, V = y.to_numpy()
    for v in V:
        assert np.abs(v.T @ v - np.eye(v.shape[1])).max() <= 1e-13 + 20 * n * 2.0 ** -53
    C = [u.T @ v for u, v in zip(U, V)]
    for t in range(3):
        G = np.moveaxis(np.tensordot(C[t], G, (1, t)), 0, t)
    assert rel(G, core) <= 1e-8
