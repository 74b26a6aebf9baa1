"""The flat-list contractions at the edges of their tiles, through a truncation that drops nothing it can see: ranks
around multiples of 32, 64 and 128, long and short reductions, odd leading dimensions (no 16-byte copies) and aligned
ones, many small blocks and few large ones, against the oracle's Tucker arithmetic.

Bound: the truncated tensor differs from the input by at most eps ||y|| plus the rounding of the three contractions, at
most 10 u sqrt(K) with K the longest reduction (n^2); eps = 1e-6 in FP64 and 2e-3 in FP32 (whose rule resolves about
1e-3)."""
import numpy as np
import pytest

from oracle import tucker
from tests.gpu_helpers import identity_tables, random_banded_terms, rel

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


def _input(n, ranks, seed):
    g = np.random.default_rng(seed)
    w = [0.7 ** np.arange(r) for r in ranks]
    core = g.standard_normal(ranks) * w[0][:, None, None] * w[1][None, :, None] * w[2][None, None, :]
    return core, [np.linalg.qr(g.standard_normal((n, r)))[0] for r in ranks]


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("n,ranks,R", [(5, (1, 1, 1), 1), (17, (4, 3, 2), 3), (33, (16, 17, 5), 2), (64, (6, 5, 4), 11),
                                       (65, (33, 31, 32), 2), (97, (9, 8, 7), 13), (128, (7, 6, 5), 19),
                                       (129, (40, 3, 2), 3), (200, (5, 4, 3), 41)])
def test_operator_product_truncation(api, dtype, n, ranks, R):
    if dtype and n > 128 and R * max(ranks) > 128:
        pytest.skip("FP32 Grams above order 128 keep at most 128 directions (tucker_round)")
    p = min(2, n - 2)
    terms = random_banded_terms(n, p, R, seed=n)
    X = _input(n, ranks, seed=n + 1)
    f = _input(n, (1, 1, 1), seed=n + 2)
    pb = api.tpcg_problem_create(n, p, terms, f[0], f[1], identity_tables(n), dtype=dtype)
    x = api.Tucker.from_numpy(*X, dtype=dtype)
    cap = min(n, 256)
    y = api.Tucker(n, R * max(ranks), cap ** 3, dtype)
    ctx = api.Ctx(n, max(R * max(ranks), cap), cap, dtype)
    api.tucker_apply(pb, x, y)
    eps = 2e-3 if dtype else 1e-6
    api.tucker_round(ctx, y, eps)
    G, U = y.to_numpy()
    want = sum(w * tucker.full((X[0], [K[t] @ X[1][t] for t in range(3)])) for w, K in terms)
    u = 2.0 ** -24 if dtype else 2.0 ** -53
    assert rel(tucker.full((G, U)), want) <= eps + 10 * u * n


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("n,rx,ry", [(7, (1, 1, 1), (2, 2, 1)), (32, (6, 5, 3), (9, 8, 7)), (65, (33, 2, 31), (32, 33, 1)),
                                     (130, (65, 17, 33), (31, 64, 5))])
def test_dot(api, dtype, n, rx, ry):
    X, Y = _input(n, rx, 1), _input(n, ry, 2)
    ctx = api.Ctx(n, 2 * min(n, 96), min(n, 96), dtype)
    x, y = (api.Tucker.from_numpy(*t, dtype=dtype) for t in (X, Y))
    got = float(api.tucker_dot(ctx, x, y))
    want = float(np.sum(tucker.full(X) * tucker.full(Y)))
    u = 2.0 ** -24 if dtype else 2.0 ** -53
    scale = np.linalg.norm(X[0]) * np.linalg.norm(Y[0])
    assert abs(got - want) <= 10 * u * np.sqrt(n) * scale * max(rx + ry)


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("sx,sy", [(1e-15, 1e-17), (1e-24, 1e-20), (1e20, 1e21), (1e25, 1e-25)])
def test_dot_keeps_products_outside_fp32s_range(api, dtype, sx, sy):
    n = 33
    X, Y = _input(n, (9, 8, 7), 1), _input(n, (6, 9, 5), 2)
    ctx = api.Ctx(n, 2 * n, n, dtype)
    x = api.Tucker.from_numpy(X[0] * sx, X[1], dtype=dtype)
    y = api.Tucker.from_numpy(Y[0] * sy, Y[1], dtype=dtype)
    got = float(api.tucker_dot(ctx, x, y)) / sx / sy
    want = float(np.sum(tucker.full(X) * tucker.full(Y)))
    u = 2.0 ** -24 if dtype else 2.0 ** -53
    assert abs(got - want) <= 10 * u * np.sqrt(n) * np.linalg.norm(X[0]) * np.linalg.norm(Y[0]) * 9


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("n,rx,ry", [(2, (1, 1, 1), (1, 1, 1)), (9, (8, 9, 1), (1, 2, 9)), (32, (32, 32, 32), (32, 32, 32)),
                                     (32, (31, 1, 17), (2, 32, 16)), (200, (17, 16, 32), (15, 9, 32)), (64, (5, 4, 3), (6, 5, 2))])
def test_dot_in_one_launch(api, dtype, n, rx, ry):
    X, Y = _input(n, rx, 3), _input(n, ry, 4)
    cap = min(n, 32)   # the bound on the ranks that selects the single launch
    ctx = api.Ctx(n, 2 * cap, cap, dtype)
    x, y = (api.Tucker.from_numpy(*t, cap=max(rx + ry), dtype=dtype) for t in (X, Y))
    want = float(np.sum(tucker.full(X) * tucker.full(Y)))
    u = 2.0 ** -24 if dtype else 2.0 ** -53
    bound = 10 * u * np.sqrt(n) * np.linalg.norm(X[0]) * np.linalg.norm(Y[0]) * max(rx + ry)
    assert abs(float(api.tucker_dot(ctx, x, y)) - want) <= bound
    assert abs(float(api.tucker_dot(ctx, y, x)) - want) <= bound
