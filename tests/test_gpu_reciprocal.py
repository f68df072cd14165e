"""The reciprocals of pp_internal.cuh (face densities), compiled from the
header: FP64 against exact fractions over the exponents and mantissas, FP32
against its instruction's bound, and the values beside the normal numbers."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PROBE = r"""
#include "pp_internal.cuh"
__global__ void k64(const double* x, double* y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = pp::rcp_f64(x[i]);
}
__global__ void k32(const float* x, float* y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = pp::rcp_f32(x[i]);
}
extern "C" int rcp64(const double* x, double* y, int n) {
  k64<<<(n + 255) / 256, 256>>>(x, y, n);
  return (int)cudaDeviceSynchronize();
}
extern "C" int rcp32(const float* x, float* y, int n) {
  k32<<<(n + 255) / 256, 256>>>(x, y, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_2005_11806_gb300 import build_ext
    d = tmp_path_factory.mktemp("rcp")
    src, lib = str(d / "rcp.cu"), str(d / "rcp.so")
    with open(src, "w") as f:
        f.write(PROBE)
    subprocess.run([build_ext._nvcc(), *build_ext.ARCH, *build_ext.FLAGS, "-I", build_ext.CSRC, "-shared", src, "-o",
                    lib], check=True, capture_output=True)
    assert os.path.exists(lib)
    return ctypes.CDLL(lib)


def _run(f, x):
    a = torch.from_numpy(x).cuda()
    y = torch.empty_like(a)
    torch.cuda.synchronize()
    assert f(ctypes.c_void_p(a.data_ptr()), ctypes.c_void_p(y.data_ptr()), x.size) == 0
    return y.cpu().numpy()


def _mantissas(rng, n, bits):
    """Random mantissas in [1, 2), and those around the ends and around the 20 bits of the estimate."""
    ulp = 2.0 ** -bits
    edge = np.concatenate([1.0 + k * ulp * np.arange(64) for k in (1.0, 2.0 ** (bits - 20))])
    return np.concatenate([1.0 + rng.random(n), edge, 2.0 - ulp * np.arange(1, 65)])


def test_fp64(probe):
    rng = np.random.default_rng(11)
    m = _mantissas(rng, 20000, 52)
    e = rng.integers(-1021, 1021, m.size)  # x and 1 / x normal
    x = np.ldexp(m, e) * rng.choice([-1.0, 1.0], m.size)
    y = _run(probe.rcp64, x)
    assert np.isfinite(y).all()
    worst = max(abs(Fraction(float(b)) * Fraction(float(a)) - 1) / (Fraction(float(np.spacing(abs(b)))) * abs(Fraction(float(a))))
                for a, b in zip(x, y))
    assert worst <= Fraction(57, 100)  # ulp
    # and over many more: never more than the neighbour of the rounded quotient
    m = 1.0 + rng.random(4_000_000)
    x = np.ldexp(m, rng.integers(-1021, 1021, m.size))
    y, ref = _run(probe.rcp64, x), 1.0 / x
    assert (np.abs(y.view(np.int64) - ref.view(np.int64)) <= 1).all()


def test_fp64_beside_the_normal_numbers(probe):
    inf, nan, tiny = np.inf, np.nan, 5e-324
    x = np.array([0.0, -0.0, inf, -inf, nan, tiny, -tiny, 2.0 ** -1023, 1.5 * 2.0 ** 1022, -1.5 * 2.0 ** 1023])
    y = _run(probe.rcp64, x)
    want = np.array([inf, -inf, 0.0, -0.0, nan, inf, -inf, inf, 0.0, -0.0])
    assert np.array_equal(y, want, equal_nan=True)
    assert np.array_equal(np.signbit(y)[:4], np.signbit(want)[:4])


def test_fp32(probe):
    rng = np.random.default_rng(12)
    m = _mantissas(rng, 2_000_000, 23)
    x = np.ldexp(m, rng.integers(-125, 125, m.size)).astype(np.float32)
    y = _run(probe.rcp32, x)
    exact = 1.0 / x.astype(np.float64)
    # one unit in the last place (the instruction's bound)
    assert (np.abs(y.astype(np.float64) - exact) <= np.spacing(np.abs(exact).astype(np.float32)).astype(np.float64)).all()
    assert np.array_equal(_run(probe.rcp32, np.array([np.inf, 0.0], dtype=np.float32)), [0.0, np.inf])
