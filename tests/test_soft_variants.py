"""The forms of csrc/wb_soft.cuh that the sweeps run (products of finite factors with
what is known of them, reciprocals and roots of inputs known to be normal), on the
host and, where the product is PTX of its own, on the device, against the FP64
multiply and the forms that test_soft_fp64.py holds against exact integers."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_1701_07452_gb300 import _build
from test_soft_fp64 import Fraction, root, samples, ulps

SRC = r"""
#include "wb_soft.cuh"
constexpr int kOut = 13;
WB_HD void forms(double x, double y, double* o) {
  o[0] = wb_smul(x, y);
  o[1] = wb_smul_finite<0>(x, y);
  o[2] = wb_smul_finite<1>(x, y);
  o[3] = wb_smul_finite<2>(x, y);
  o[4] = wb_smul_finite<7>(x, y);
  const WbRoots r = wb_roots(x), s = wb_roots_sure(x);
  o[5] = r.rsq; o[6] = r.sq; o[7] = r.rcp;
  o[8] = s.rsq; o[9] = s.sq; o[10] = s.rcp;
  o[11] = wb_rcp(x);
  o[12] = wb_rcp_sure(x);
}
#ifdef DEVICE
__global__ void k_forms(int n, const double* x, const double* y, double* o) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) forms(x[i], y[i], o + (size_t)kOut * i);
}
extern "C" int run_forms(int n, const double* x, const double* y, double* o) {
  double *dx = nullptr, *dy = nullptr, *dout = nullptr;
  const size_t bytes = sizeof(double) * n;
  cudaError_t e = cudaMalloc(&dx, bytes);
  if (e == cudaSuccess) e = cudaMalloc(&dy, bytes);
  if (e == cudaSuccess) e = cudaMalloc(&dout, kOut * bytes);
  if (e == cudaSuccess) e = cudaMemcpy(dx, x, bytes, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(dy, y, bytes, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    k_forms<<<(n + 255) / 256, 256>>>(n, dx, dy, dout);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(o, dout, kOut * bytes, cudaMemcpyDeviceToHost);
  cudaFree(dx);
  cudaFree(dy);
  cudaFree(dout);
  return (int)e;
}
#else
extern "C" int run_forms(int n, const double* x, const double* y, double* o) {
  for (int i = 0; i < n; ++i) forms(x[i], y[i], o + (size_t)kOut * i);
  return 0;
}
#endif
"""


@pytest.fixture(scope="module", params=["host", pytest.param("device", marks=pytest.mark.gpu)])
def forms(request, tmp_path_factory):
    """f(x, y) -> the 13 outputs, one row each."""
    flags = []
    if request.param == "device":
        torch = pytest.importorskip("torch")
        if not torch.cuda.is_available():
            pytest.skip("no CUDA device")
        flags = [*_build.ARCH, "-DDEVICE"]
    d = tmp_path_factory.mktemp("forms")
    src, so = d / "forms.cu", d / "libforms.so"
    src.write_text(SRC)
    subprocess.run([_build.nvcc(), "-std=c++17", "-O3", *flags, "-Xcompiler", "-fPIC", "-shared", "-I", _build.CSRC,
                    str(src), "-o", str(so)], check=True, capture_output=True)
    L = ctypes.CDLL(str(so))

    def run(x, y):
        x, y = np.ascontiguousarray(x), np.ascontiguousarray(y)
        assert x.size == y.size
        out = np.empty((x.size, 13))
        dp = ctypes.POINTER(ctypes.c_double)
        assert L.run_forms(x.size, *[a.ctypes.data_as(dp) for a in (x, y, out)]) == 0
        return out.T
    return run


def pairs(lo, hi, seed):
    """Factors of exponent fields lo..hi: random and short significands (ties and
    exact products among them), both signs."""
    rng = np.random.default_rng(seed)
    x = np.concatenate([samples(20000, lo, hi, s) for s in range(5)])
    y = rng.permutation(x) * rng.choice([-1.0, 1.0], x.size)
    keep = np.uint64(0xFFFFFFFFFFFFFFFF) << rng.integers(0, 53, x.size).astype(np.uint64)
    x = (x.view(np.uint64) & np.where(rng.random(x.size) < 0.5, keep, ~np.uint64(0))).view(np.float64)
    return x * rng.choice([-1.0, 1.0], x.size), y


def bits(a):
    return np.ascontiguousarray(a).view(np.uint64)


@pytest.mark.parametrize("lo,hi", [(1003, 1043), (513, 1533), (400, 1533)])
def test_products(forms, lo, hi):
    """Bits of the FP64 multiply for magnitudes of 2^-1021 and up; zero below 2^-1022,
    one or the other in the binade between; exact zeros of either sign."""
    x, y = pairs(lo, hi, lo)
    x[1::501], y[::501], y[3::501] = -0.0, 0.0, 1.0
    out = forms(x, y)
    with np.errstate(under="ignore", over="ignore"):
        want = x * y
    mag = np.abs(want)
    assert mag.max() < 2.0 ** 1023
    ok = mag >= 2.0 ** -1021
    zero = (bits(x) << np.uint64(1) == 0), (bits(y) << np.uint64(1) == 0)
    for row, domain in ((0, ok | (mag == 0.0)), (1, ok | (mag == 0.0)), (2, ~zero[0]), (3, ~zero[1]),
                        (4, ok)):
        got, exact = out[row][domain & ok], want[domain & ok]
        assert np.array_equal(bits(got), bits(exact)), row
        if row < 4:
            low = domain & ~ok
            flushed = bits(out[row][low]) == bits(np.copysign(0.0, want[low]))
            assert np.all(flushed | ((out[row][low] == want[low]) & (mag[low] >= 2.0 ** -1022))), row


@pytest.mark.parametrize("lo,hi", [(1, 2044), (1013, 1033)])
def test_roots_and_reciprocals(forms, lo, hi):
    """The sure forms have the bits of the checked ones for positive normal x below
    2^1022, where the reciprocal is normal too, and both are within the bounds of
    the fixed-point steps (see test_soft_fp64.py)."""
    x = np.concatenate([samples(4000, lo, hi, s) for s in range(5)])
    out = forms(x, np.ones_like(x))
    for sure, checked in ((8, 5), (9, 6), (10, 7), (12, 11)):
        assert np.array_equal(bits(out[sure]), bits(out[checked])), sure
    for i in range(0, x.size, 23):
        f = Fraction(float(x[i]))
        r = root(f)
        assert ulps(float(out[5][i]), 1 / r) < 0.52 and ulps(float(out[6][i]), r) < 0.52
        assert ulps(float(out[7][i]), 1 / f) < 0.53 and ulps(float(out[11][i]), 1 / f) < 0.52


def test_sure_reciprocal_of_negative_values(forms):
    x = -samples(4000, 1, 2044, 7)
    out = forms(x, np.ones_like(x))
    assert np.array_equal(bits(out[12]), bits(out[11])) and np.all(out[12] < 0)
