"""silu(g) * u as the projection kernels' epilogues compute it, against float64 and against the division operator, over every
magnitude of g: the range where the reciprocal of the denominator is subnormal, infinities and NaN among them."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2510_04147_b200 import build

pytestmark = pytest.mark.gpu

SOURCE = """
#include "kernels.h"
__global__ void both(const float* g, const float* u, float* a, float* b, int n) {
  const int i = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
  if (i + 1 >= n) return;
  ssd::swiglu2(g[i], g[i + 1], u[i], u[i + 1], a[i], a[i + 1]);
  for (int j = i; j < i + 2; ++j) b[j] = g[j] / (1.f + expf(-g[j])) * u[j];
}
extern "C" int run(const float* g, const float* u, float* a, float* b, int n) {
  both<<<(n / 2 + 255) / 256, 256>>>(g, u, a, b, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def swiglu(tmp_path_factory):
    d = tmp_path_factory.mktemp("swiglu")
    (d / "swiglu.cu").write_text(SOURCE)
    flags = [f for f in build.NVCC_FLAGS if f not in ("-Xptxas", "-v")]
    subprocess.run([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), *flags, "-shared", "-I", build.CSRC, "-o", str(d / "swiglu.so"),
                    str(d / "swiglu.cu")], check=True)
    lib = ctypes.CDLL(str(d / "swiglu.so"))

    def run(g, u):
        assert len(g) % 2 == 0
        dev = [torch.from_numpy(np.ascontiguousarray(x, np.float32)).cuda() for x in (g, u, g, u)]
        torch.cuda.synchronize()
        assert lib.run(*[ctypes.c_void_p(t.data_ptr()) for t in dev], len(g)) == 0
        return dev[2].cpu().numpy(), dev[3].cpu().numpy()

    return run


def _gates():
    powers = np.float32(2.0) ** np.arange(-149, 128, dtype=np.float32)
    near = np.concatenate([np.linspace(lo, lo + 4, 200001) for lo in (-91.0, -88.0, 85.0)])
    g = np.concatenate([np.linspace(-110, 110, 2000001), near, powers, -powers, [0.0, -0.0, np.finfo(np.float32).max, -np.finfo(np.float32).max]])
    return g[:len(g) // 2 * 2].astype(np.float32)


@pytest.mark.parametrize("u", [1.0, -0.73, 3.0e5])
def test_swiglu_over_all_magnitudes(swiglu, u):
    g = _gates()
    got, div = swiglu(g, np.full_like(g, u))
    assert np.array_equal(np.isfinite(got), np.isfinite(div))
    with np.errstate(over="ignore"):
        exact = g.astype(np.float64) / (1.0 + np.exp(-g.astype(np.float64))) * u
    # expf 2 ulp, the sum, the quotient and the product half a unit each: 3.5 * 2^-23 of the value.  Past e^-g = 2^128 the
    # denominator is infinite and the result 0, also with `/`; results below the normal range keep the distance of a subnormal.
    low = np.abs(u) * 89 * 2.0 ** -128 * (g < -88.7) + 2.0 ** -148 * max(1.0, abs(u))
    fits = np.abs(exact) < np.finfo(np.float32).max
    assert (np.abs(got[fits] - exact[fits]) <= (3.5 * 2.0 ** -23 * np.abs(exact) + low)[fits]).all()
    # a last place of the quotient, carried through the product
    assert (np.abs(got[fits].astype(np.float64) - div[fits]) <= 2.0 ** -22 * np.abs(div[fits]) + 2.0 ** -148 * max(1.0, abs(u))).all()
    assert (got[g <= -89] == 0).all()


def test_swiglu_of_what_is_not_finite(swiglu):
    inf, nan = np.float32(np.inf), np.float32(np.nan)
    g = np.array([inf, inf, inf, -inf, -inf, nan, nan, 1.0, -100.0, -100.0], np.float32)
    u = np.array([2.0, -2.0, 0.0, 2.0, inf, 1.0, inf, nan, 2.0, inf], np.float32)
    got, div = swiglu(g, u)
    assert np.array_equal(got, div, equal_nan=True), (got, div)
