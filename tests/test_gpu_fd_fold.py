"""The preconditioner by the two half sine matrices against the dense sine product, at the edges of its tiles: odd and even
lengths n1, one to three tiles of input columns, output tiles that straddle two terms, the largest n1 the halves take and the
first that goes to the FFTs, one and two kinds of ends (unlike ends have no halves), a tensor of two blocks.

Bound: both transforms are sums of n1 products of rounded values, two in a row, so the factors agree to 16 (n + 8) u of
their norm; descriptors are equal."""
import numpy as np
import pytest

import synth
from tests.gpu_helpers import gpu_problem, rel

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2306_00632_gb300 import api as a
    from paper_2306_00632_gb300 import lib
    lib.load()
    yield a
    a.set_option(lib.OPT_DST, 1)


def _both(api, pb, ctx, s, cap):
    from paper_2306_00632_gb300 import lib
    out = []
    for kind in (1, 0):
        api.set_option(lib.OPT_DST, kind)
        v = api.Tucker(s.n, cap=cap, core_cap=1, dtype=s.dtype)
        api.fd_precond_apply(pb, ctx, s, v)
        out.append(v.to_numpy(others=[s]))
    return out


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("n,p,ranks", [(4, 1, (1, 2, 4)), (5, 2, (5, 1, 3)), (9, 3, (9, 8, 1)), (33, 3, (33, 32, 31)),
                                       (64, 1, (1, 63, 17)), (65, 2, (65, 7, 33)), (66, 4, (2, 11, 64)), (128, 3, (44, 43, 41)),
                                       (256, 2, (31, 3, 64)), (256, 3, (2, 33, 1)), (257, 2, (3, 1, 2))])
def test_halves_match_dense(api, n, p, ranks, dtype):
    pb = gpu_problem("cube", 0.0, n, p, dtype=dtype)
    S = synth.random_tucker((n, n, n), ranks, seed=n)
    s = api.Tucker.from_numpy(S[0], S[1], dtype=dtype)
    cap = pb.info.RP * max(ranks)
    ctx = api.Ctx(n, cap, min(n, 96), dtype)
    (g, f), (gd, fd) = _both(api, pb, ctx, s, cap)
    u = 2.0 ** -24 if dtype else 2.0 ** -53
    assert rel(g, gd) == 0.0
    for t in range(3):
        assert f[t].shape == fd[t].shape
        assert rel(f[t], fd[t]) <= 16 * (n + 8) * u


def test_output_over_capacity_is_flagged(api):
    n = 17
    pb = gpu_problem("cube", 0.0, n, 3)
    S = synth.random_tucker((n, n, n), (3, 2, 4), seed=1)
    s = api.Tucker.from_numpy(S[0], S[1])
    ctx = api.Ctx(n, 4 * pb.info.RP, n)
    v = api.Tucker(n, cap=3 * pb.info.RP, core_cap=1)   # the third mode needs 4 per term
    api.fd_precond_apply(pb, ctx, s, v)
    assert v.read_desc()[0] == 0
