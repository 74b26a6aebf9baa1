"""What the process-wide options reach, read from the kernels that a call enqueues."""
import pytest

import synth
from oracle import tucker
from tests.graph_helpers import kernels

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def mods():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2306_00632_gb300 import api, lib
    lib.load()
    return api, lib


@pytest.mark.parametrize("dtype,name", [(0, "gemm64_kernel"), (1, "gemm32_kernel")])
def test_ctas_per_sm_reaches_both_types(mods, dtype, name):
    """CTAs of 256 threads an SM; the contractions' CTAs of 128 threads count half."""
    api, lib = mods
    n = 64
    Y = synth.random_tucker((n, n, n), (20, 21, 22), seed=3)
    y = api.Tucker.from_numpy(Y[0], Y[1], cap=n, core_cap=n ** 3, dtype=dtype)
    ctx = api.Ctx(n, n, n, dtype=dtype)
    sms = torch.cuda.get_device_properties(0).multi_processor_count

    def largest():
        return max(g[0] * g[1] * g[2] * b[0] for k, g, b, _ in kernels(lambda: api.tucker_round(ctx, y, 1e-3)) if name in k)

    try:
        for budget in (1, 2, 3):
            api.set_option(lib.OPT_GEMM_CTAS_PER_SM, budget)
            assert largest() <= budget * sms * 256
        api.set_option(lib.OPT_GEMM_CTAS_PER_SM, 0)
        assert largest() > 3 * sms * 256
    finally:
        api.set_option(lib.OPT_GEMM_CTAS_PER_SM, 2)


def test_tensor_cores_reach_small_scalar_products(mods):
    api, lib = mods
    n = 24
    X = synth.random_tucker((n, n, n), (5, 6, 7), seed=5)
    Y = synth.random_tucker((n, n, n), (8, 3, 4), seed=6)
    try:
        api.set_option(lib.OPT_TC, 1)
        for dtype in (0, 1):
            x, y = (api.Tucker.from_numpy(T[0], T[1], dtype=dtype) for T in (X, Y))
            ctx = api.Ctx(n, n, 16, dtype=dtype)
            out = torch.zeros(1, dtype=torch.float64, device="cuda")
            names = [k for k, *_ in kernels(lambda: api.tucker_dot(ctx, x, y, out=out))]
            assert any("gemm_tc" in k for k in names) == (dtype == 1), names
            # 22 bits of each operand over the sums of five contractions
            assert abs(api.tucker_dot(ctx, x, y).item() - tucker.dot(X, Y)) <= 1e-5 * tucker.norm(X) * tucker.norm(Y)
    finally:
        api.set_option(lib.OPT_TC, 0)
