"""The corrected reciprocals of recip.cuh against CUDA's divisions and roots, over the exponents they are used at (the ends
among them) and mantissas, and the conversions by moving bits.

Bounds in units of u = 2^-53 (relative): the FMA that ends the FP64 reciprocal rounds once, the series' end is 0.05, and the
IEEE division rounds once: 2.2.  FP32 (u = 2^-24) against FP64: one rounding, 1.1; the root's 1 - d y^2 carries the rounding
of d y besides, half of which reaches the result: 1.6."""
import ctypes as C
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SRC = r"""
#include "recip.cuh"
using namespace tpcg;
__global__ void k(const double* d, int n, double* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double v = d[i];
    const float f = (float)v;
    const double o[7] = {recip_mid(v), 1.0 / v, (double)rsqrt_from(f, rsqrtf(f)), (double)recip_from(f, __fdividef(1.f, f)),
                         (double)bits_to_float(v), bits_to_double(f), bits_to_double(f, 100)};
    for (int q = 0; q < 7; ++q) out[(long long)q * n + i] = o[q];
}
extern "C" int run(const double* d, int n, double* out) {
    k<<<(n + 255) / 256, 256>>>(d, n, out);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2306_00632_gb300 import build
    t = tmp_path_factory.mktemp("recip")
    (t / "k.cu").write_text(SRC)
    so = str(t / "librecip.so")
    subprocess.run([build.NVCC, *build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I" + build.CSRC,
                    str(t / "k.cu"), "-o", so], check=True)
    lib = C.CDLL(so)

    def f(d):
        x = torch.tensor(d, dtype=torch.float64, device="cuda")
        out = torch.empty((7, len(d)), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert lib.run(C.c_void_p(x.data_ptr()), len(d), C.c_void_p(out.data_ptr())) == 0
        return out.cpu().numpy()

    return f


def _mantissas(g, per):
    m = 1.0 + g.uniform(0, 1, per)
    m[:6] = [1.0, 1.0 + 2.0 ** -52, 2.0 - 2.0 ** -52, 1.5, 1.0 + 2.0 ** -23, 2.0 - 2.0 ** -24]
    return m


def _off(a, b):
    return np.max(np.abs(a / b - 1.0))


def test_corrections_and_conversions(run):
    g = np.random.default_rng(2)
    e = np.repeat(np.arange(-126, 127), 1024)
    d = np.ldexp(np.concatenate([_mantissas(g, 1024) for _ in range(253)]), e)
    o = run(d)
    mid = np.abs(e) <= 124
    assert _off(o[0][mid], o[1][mid]) <= 2.2 * 2.0 ** -53
    f = d.astype(np.float32).astype(np.float64)
    assert _off(o[2], 1.0 / np.sqrt(f)) <= 1.6 * 2.0 ** -24
    assert _off(o[3][mid], 1.0 / f[mid]) <= 1.1 * 2.0 ** -24
    # mantissas cut to 24 bits, and back
    assert np.array_equal(o[4], np.ldexp(np.floor(np.ldexp(d, 23 - e)), e - 23))
    assert np.array_equal(o[5], f)
    assert np.array_equal(o[6], np.ldexp(f, 100))


def test_below_single_precision(run):
    assert not run(np.ldexp(1.7, np.arange(-1000, -126)))[4].any()
