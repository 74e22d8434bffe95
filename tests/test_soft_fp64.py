"""FP64 arithmetic on the integer pipes (csrc/wb_soft.cuh), compiled for the
host: the same integer operations as on the device, against exact integers."""
import ctypes
import math
import os
import struct
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_1701_07452_gb300 import _build

SRC = r"""
#include "wb_soft.cuh"
extern "C" void soft_roots(int n, const double* x, double* rsq, double* sq, double* rc, double* rcp) {
  for (int i = 0; i < n; ++i) {
    const WbRoots r = wb_roots(x[i]);
    rsq[i] = r.rsq; sq[i] = r.sq; rc[i] = r.rcp; rcp[i] = wb_rcp(x[i]);
  }
}
extern "C" void soft_mul(int n, const double* x, const double* y, double* p) {
  for (int i = 0; i < n; ++i) p[i] = wb_smul(x[i], y[i]);
}
"""


@pytest.fixture(scope="module", params=[-1, 0, 1])
def soft(request, tmp_path_factory):
    """The host build, with the FP32 seeds moved by a unit of 2^-23 (one to two
    ulp of the approximations, whose documented errors are below that)."""
    d = tmp_path_factory.mktemp("soft")
    src, so = d / "soft.cu", d / "libsoft.so"
    src.write_text(SRC)
    subprocess.run([_build.nvcc(), "-std=c++17", "-O2", "-Xcompiler", "-fPIC", "-shared", "-I", _build.CSRC,
                    f"-DWB_SEED_ULPS={request.param}", str(src), "-o", str(so)], check=True, capture_output=True)
    assert os.path.exists(so)
    return ctypes.CDLL(str(so))


def call(fn, n, *arrays):
    fn(n, *[a.ctypes.data_as(ctypes.POINTER(ctypes.c_double)) for a in arrays])


def from_bits(b):
    return struct.unpack("<d", struct.pack("<Q", int(b)))[0]


def samples(n, lo, hi, seed):
    """Doubles with exponent fields lo..hi: random significands and the ends of a binade."""
    rng = np.random.default_rng(seed)
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    m[::7] = [0, 1, 2, (1 << 52) - 1, (1 << 52) - 2][seed % 5]
    m[1::7] &= np.uint64(0xFFFFF00000000)
    e = rng.integers(lo, hi + 1, n).astype(np.uint64)
    e[2::97], e[3::97] = lo, hi
    return (e << np.uint64(52) | m).view(np.float64).copy()


def ulps(got, exact):
    """|got - exact| in units of exact's last place, exact a Fraction > 0."""
    e = math.floor(math.log2(float(exact))) if exact > Fraction(1, 1 << 1021) else -1022
    while Fraction(2) ** (e + 1) <= exact:
        e += 1
    while e > -1022 and Fraction(2) ** e > exact:
        e -= 1
    return abs(Fraction(got) - exact) / Fraction(2) ** (e - 52)


def root(x):
    """sqrt of a Fraction to 2^-160 relative."""
    k = 400 - (x.numerator.bit_length() - x.denominator.bit_length()) // 2
    return Fraction(math.isqrt((x.numerator << 2 * k) // x.denominator if k >= 0
                               else x.numerator // (x.denominator << -2 * k)), 1) / Fraction(2) ** k


@pytest.mark.parametrize("lo,hi", [(1, 2046), (1013, 1033)])
def test_roots_and_reciprocals_round_once(soft, lo, hi):
    """Truncations of the fixed-point steps stay below 2^-60 of y, that is
    0.008 ulp of 1/sqrt(x), 0.016 ulp of sqrt(x), 0.023 ulp of its square and
    0.008 ulp of the plain reciprocal, on top of the final half."""
    x = np.concatenate([samples(700, lo, hi, s) for s in range(5)])
    out = [np.empty_like(x) for _ in range(4)]
    call(soft.soft_roots, len(x), x, *out)
    for i, v in enumerate(x):
        f = Fraction(float(v))
        r = root(f)
        assert ulps(float(out[0][i]), 1 / r) < 0.52, (v, out[0][i])
        assert ulps(float(out[1][i]), r) < 0.52, (v, out[1][i])
        assert ulps(float(out[2][i]), 1 / f) < 0.53, (v, out[2][i])
        assert ulps(float(out[3][i]), 1 / f) < 0.52, (v, out[3][i])


def test_reciprocal_sign_and_bad_inputs(soft):
    """A negative x gives the negated reciprocal; zero, subnormals, infinities
    and NaN (and negative x for the roots) give NaN."""
    x = np.array([-3.0, -1.0, -1e300, 0.0, -0.0, 5e-324, 2.2e-308, np.inf, -np.inf, np.nan])
    out = [np.empty_like(x) for _ in range(4)]
    call(soft.soft_roots, len(x), x, *out)
    for o in out[:3]:
        assert np.all(np.isnan(o)), o
    assert out[3][0] == 1 / -3.0 and out[3][1] == -1.0 and out[3][2] == 1 / -1e300
    assert np.all(np.isnan(out[3][3:]))


@pytest.mark.parametrize("lo,hi", [(1003, 1043), (400, 1600), (1, 2046)])
def test_products_have_the_bits_of_the_fp64_multiply(soft, lo, hi):
    """Random and short significands (ties and exact products among them), both
    signs, zeros: the bits of the FP64 product wherever its magnitude is zero or
    in [2^-1021, 2^1023); zero below the normal range, NaN above it."""
    x = np.concatenate([samples(20000, lo, hi, s) for s in range(5)])
    rng = np.random.default_rng(lo)
    y = rng.permutation(x) * rng.choice([-1.0, 1.0], x.size)
    keep = (np.uint64(0xFFFFFFFFFFFFFFFF) << rng.integers(0, 53, x.size).astype(np.uint64))
    x = (x.view(np.uint64) & np.where(rng.random(x.size) < 0.5, keep, ~np.uint64(0))).view(np.float64)
    y[::501], x[1::501], y[3::501] = 0.0, -0.0, 1.0
    p = np.empty_like(x)
    call(soft.soft_mul, x.size, x, y, p)
    with np.errstate(over="ignore", under="ignore"):
        want = x * y
    mag = np.abs(want)
    low, high = mag < 2.0 ** -1021, mag >= 2.0 ** 1023
    mid = ~low & ~high
    assert np.array_equal(p[mid].view(np.uint64), want[mid].view(np.uint64))
    # at the ends of the range the exponents' sum decides: flushed (NaN) or exact
    flushed = p[low].view(np.uint64) == np.copysign(0.0, want[low]).view(np.uint64)
    assert np.all(flushed | ((p[low] == want[low]) & (mag[low] >= 2.0 ** -1022)))
    assert np.all(np.isnan(p[high]) | (p[high] == want[high]))
    if (lo, hi) == (1003, 1043):
        assert np.all(mid | (want == 0.0))


def test_products_of_bad_factors_are_nan(soft):
    """Infinities and NaN give NaN with any factor but a subnormal or zero one,
    where NaN too; subnormal factors count as zero."""
    bad = np.array([np.inf, -np.inf, np.nan])
    for other in (1.0, -3e-200, 2e200, 0.0, 5e-324, np.inf):
        p = np.empty(3)
        call(soft.soft_mul, 3, bad, np.full(3, other), p)
        assert np.all(np.isnan(p)), other
    p = np.empty(2)
    call(soft.soft_mul, 2, np.array([5e-324, -2e-308]), np.array([1e300, 1e300]), p)
    assert p[0] == 0.0 and p[1] == 0.0 and np.signbit(p[1])
