"""The FP32 kernels' reciprocal, square root and log1p (lbm_device.cuh) against 64 bits, scalar and
in pairs, over the arguments the equations of state, the collision and the links give them.

Bounds, in units of the result's last place (ulp):
  recip, root   0.5 for the last rounding and e^2 2^24 of it for what the Newton step leaves of the
                approximation's error e = 2^-22: 0.5001; 0.501 asserted.
  log1p         f's rounding: half an ulp of f, which is a whole one of the result where the logarithm
                falls below the binade of f (f in [0.25, 0.284)), over 1 + f: 0.8; the last rounding
                0.5; the roundings in f^2 Q (f^2 Q = 0.03 there, two roundings and the polynomial's own
                5e-9, in ulps of 2^-26): 0.3.  1.6 without a power of two.  With one (f < 0 next to
                e ln 2 > 0.34 and the reverse) f's rounding is 0.5 / 0.707, the sum f + f^2 Q rounds
                once more, and the constant ln 2 is 2^-25 of 0.69 off at the most: 2.4."""
from __future__ import annotations

import ctypes
import os
import re
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2203_04508_gb300", "csrc")

SOURCE = r"""
#include "lbm_device.cuh"
using namespace lbmgb;
template <typename V>
__device__ V apply(int op, V a, V b) {
  return op == 0 ? recip(a) : op == 1 ? root(a) : log1p_product(a, b);
}
// y[i]: element i alone; z: two at a time; w: log1pf of the rounded product
__global__ void k(int op, int n, const float* a, const float* b, float* y, float* z, float* w) {
  const int i = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
  if (i + 1 >= n) return;
  for (int j = i; j < i + 2; ++j) {
    y[j] = apply(op, a[j], b[j]);
    w[j] = log1pf(__fmul_rn(a[j], b[j]));
  }
  const float2 p = apply(op, make_float2(a[i], a[i + 1]), make_float2(b[i], b[i + 1]));
  z[i] = p.x;
  z[i + 1] = p.y;
}
extern "C" int run(int op, int n, const float* a, const float* b, float* y, float* z, float* w) {
  k<<<(n / 2 + 255) / 256, 256>>>(op, n, a, b, y, z, w);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def device_math(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2203_04508_gb300 import build
    d = tmp_path_factory.mktemp("math")
    (d / "m.cu").write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, *build.COMMON, "-shared", "-o", str(d / "m.so"), str(d / "m.cu")],
                   check=True)
    lib = ctypes.CDLL(str(d / "m.so"))

    def run(op, a, b=None):
        n = a.size // 2 * 2
        b = np.ones_like(a) if b is None else b
        t = [torch.tensor(v[:n], device="cuda") for v in (a, b)] + [torch.empty(n, device="cuda") for _ in range(3)]
        torch.cuda.synchronize()
        assert lib.run(op, n, *[ctypes.c_void_p(v.data_ptr()) for v in t]) == 0
        y, z, w = (v.cpu().numpy() for v in t[2:])
        assert np.array_equal(y, z, equal_nan=True)   # a pair: each half as the scalar
        return y.astype(np.float64), w.astype(np.float64)
    return run


def _ulps(y, exact):
    return np.abs(y - exact) / np.spacing(np.abs(exact).astype(np.float32)).astype(np.float64)


N = 1 << 20


@pytest.mark.gpu
@pytest.mark.parametrize("lo,hi", [(1e-6, 1e-3), (1e-3, 1.0), (1.0, 2.0), (2.0, 4000.0)])
def test_reciprocal_and_root(device_math, lo, hi):
    """Densities, 1 - b rho / 4, 2 q, and the pseudopotential's square."""
    a = np.exp(np.random.default_rng(1).uniform(np.log(lo), np.log(hi), N)).astype(np.float32)
    assert _ulps(device_math(0, a)[0], 1.0 / a.astype(np.float64)).max() <= 0.501
    assert _ulps(device_math(0, -a)[0], -1.0 / a.astype(np.float64)).max() <= 0.501
    assert _ulps(device_math(1, a)[0], np.sqrt(a.astype(np.float64))).max() <= 0.501


@pytest.mark.gpu
@pytest.mark.parametrize("lo,hi,bound", [(-0.9999, -0.9, 2.4), (-0.9, -0.3, 2.4), (-0.29, 0.41, 1.6), (-0.05, 0.05, 1.6),
                                         (-1e-4, 1e-4, 1.6), (0.41, 1.0, 2.4), (1.0, 12.0, 2.4), (12.0, 300.0, 2.4)])
def test_log1p_of_a_product(device_math, lo, hi, bound):
    """(rho - rho0) / rho0 from the gas at the coexistence density's nearer side to the liquid."""
    rng = np.random.default_rng(2)
    b = np.exp(rng.uniform(np.log(0.1), np.log(1e3), N)).astype(np.float32)
    a = (rng.uniform(lo, hi, N) / b.astype(np.float64)).astype(np.float32)
    exact = np.log1p(a.astype(np.float64) * b.astype(np.float64))
    y, w = device_math(2, a, b)
    e, e_library = _ulps(y, exact), _ulps(w, exact)
    print(f"[{lo}, {hi}]: max {e.max():.2f} rms {np.sqrt((e * e).mean()):.3f}; log1pf of the product "
          f"max {e_library.max():.2f} rms {np.sqrt((e_library ** 2).mean()):.3f}")
    assert e.max() <= bound


@pytest.mark.gpu
def test_log1p_over_a_mixture_is_no_worse_than_the_library(device_math):
    """All densities between a gas and a liquid with a ratio of 130, against the nearer of the two."""
    r0 = np.array([0.003, 0.4])
    r = np.exp(np.random.default_rng(3).uniform(np.log(r0[0] * 0.8), np.log(r0[1] * 1.1), N)).astype(np.float32)
    near = r0.astype(np.float32)[(r.astype(np.float64) > np.sqrt(r0.prod())).astype(int)]
    a, b = (r - near).astype(np.float32), (1.0 / near.astype(np.float64)).astype(np.float32)
    exact = np.log1p(a.astype(np.float64) * b.astype(np.float64))
    y, w = device_math(2, a, b)
    rms = [np.sqrt((_ulps(v, exact)[exact != 0] ** 2).mean()) for v in (y, w)]
    print(rms)
    assert rms[0] <= rms[1]


@pytest.mark.gpu
def test_logarithm_of_what_is_not_positive(device_math):
    a = np.array([-1.0, -1.5, -3.0, np.nan, -np.inf, 0.0], np.float32)
    y, _ = device_math(2, a)
    assert np.isnan(y[:5]).all() and y[5] == 0.0


def test_the_polynomial_holds_its_stated_error():
    """The coefficients in the source, in 64 bits: relative error of f + f^2 Q(f) at most 5e-9."""
    text = open(os.path.join(CSRC, "lbm_device.cuh")).read()
    body = text[text.index("V log1p_product(V a, V b)"):]
    c = [np.float64(np.float32(v)) for v in re.findall(r"K\((-?0\.\d{10})f\)", body[:body.index("LogParts::checked")])]
    assert len(c) == 9
    f = np.linspace(np.sqrt(0.5) - 1, np.sqrt(2.0) - 1, 200001)
    f = f[np.abs(f) > 1e-7]
    q = np.polyval(c, f)
    assert np.abs((f + f * f * q) / np.log1p(f) - 1).max() <= 5e-9
