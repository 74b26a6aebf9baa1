"""The preconditioner's FFT sine transforms (TPCG_OPT_DST 2) at the lengths whose default are the half sine matrices: FFT
sizes 16 to 1024, odd and even lengths, doubled lengths with a large prime factor, against the dense sine product and, for
small n, the oracle.

Bound: the dense product's sums of n1 rounded products, twice in a row, agree to 16 (n + 8) u of their norm, and the FFTs'
6 log2(4 n) + 12 roundings a transform are fewer.  The oracle's eigenvectors are interpolated to 1e-11."""
import pytest

import synth
from tests.graph_helpers import kernels
from tests.gpu_helpers import gpu_problem, oracle_problem, rel

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def mods():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2306_00632_gb300 import api, lib
    lib.load()
    yield api, lib
    api.set_option(lib.OPT_DST, 1)


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("n,p,ranks", [(5, 2, (2, 1, 5)), (17, 2, (3, 2, 4)), (24, 3, (8, 1, 3)), (33, 4, (3, 17, 4)), (66, 4, (9, 2, 4)),
                                       (128, 3, (20, 33, 1)), (256, 3, (3, 2, 4)), (257, 2, (5, 3, 1))])
def test_ffts_match_dense_and_oracle(mods, n, p, ranks, dtype):
    api, lib = mods
    pb = gpu_problem("cube", 0.0, n, p, dtype=dtype)
    S = synth.random_tucker((n, n, n), ranks, seed=23)
    s = api.Tucker.from_numpy(S[0], S[1], dtype=dtype)
    cap = pb.info.RP * max(ranks)
    ctx = api.Ctx(n, cap, max(ranks), dtype)
    out = {}
    for kind in (2, 0):
        api.set_option(lib.OPT_DST, kind)
        v = api.Tucker(n, cap=cap, core_cap=1, dtype=dtype)
        names = [k for k, *_ in kernels(lambda: api.fd_precond_apply(pb, ctx, s, v))]
        assert any("chirp" in k for k in names) == (kind == 2) and not any("fold" in k for k in names), names
        api.fd_precond_apply(pb, ctx, s, v)
        out[kind] = v.to_numpy(others=[s])
    u = 2.0 ** -24 if dtype else 2.0 ** -53
    assert rel(out[2][0], out[0][0]) == 0.0
    for t in range(3):
        assert rel(out[2][1][t], out[0][1][t]) <= 16 * (n + 8) * u
    if n <= 70 and dtype == 0:
        ref = oracle_problem("cube", 0.0, n, p)[2].apply(S)
        for t in range(3):
            assert rel(out[2][1][t], ref[1][t]) < 1e-11
