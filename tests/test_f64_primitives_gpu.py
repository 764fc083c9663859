"""The FP64 reciprocal, root and quotient that start from FP32 ones
(csrc/lbmhd_f64.cuh rcp64, sqrt64; csrc/lbmhd_narrow.cuh divide_all), against the
exact values in rational arithmetic.

Bounds, in units of the last place, from the method: an FP32 start with
|e| <= 2^-22 (a reciprocal good to an FP32 ulp of an operand cut to 24 bits) and
the third-order step y (1 + e + e^2) leave e^3 = 2^-66, 2^-13 ulp, before the last
rounding; the root and the quotient end in a correction by their exact
remainder.  So none is off by more than 0.501 ulp.  Operands beyond the range of
the FP32 start take the IEEE operation and must equal it.
"""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from conftest import ROOT

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "lbmhd_f64.cuh"
#include "lbmhd_narrow.cuh"
using namespace lbmhd;
__global__ void eval(int op, const double* x, const double* y, double* out, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (op == 0) out[i] = rcp64(x[i]);
    if (op == 1) out[i] = sqrt64(x[i]);
    if (op == 2) {
        const double a[2] = {x[i], -x[i]};
        double q[2];
        divide_all<2>(a, y[i], q);
        out[i] = q[0] == -q[1] || q[0] != q[0] ? q[0] : 1e308;  // both signs alike
    }
}
extern "C" int run(int op, const double* x, const double* y, double* out, int n) {
    double* d = nullptr;
    const size_t b = (size_t)n * sizeof(double);
    if (cudaMalloc((void**)&d, 3 * b) != cudaSuccess) return 1;
    cudaMemcpy(d, x, b, cudaMemcpyHostToDevice);
    cudaMemcpy(d + n, y, b, cudaMemcpyHostToDevice);
    eval<<<(n + 255) / 256, 256>>>(op, d, d + n, d + 2 * n, n);
    const cudaError_t e = cudaMemcpy(out, d + 2 * n, b, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return e != cudaSuccess;
}
"""


@pytest.fixture(scope="module")
def ev(tmp_path_factory):
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1607_08675_gb300 import build

    d = tmp_path_factory.mktemp("f64")
    src, lib = d / "f64.cu", d / "f64.so"
    src.write_text(SOURCE)
    flags = [f for f in build.FLAGS if f != "-lineinfo"]
    subprocess.run([build.nvcc(), *build.ARCH, *flags, "-I", build.CSRC, "-shared", str(src), "-o", str(lib)],
                   check=True, capture_output=True)
    f = ctypes.CDLL(str(lib)).run

    def ev(op, x, y=None):
        x = np.ascontiguousarray(x, dtype=np.float64)
        y = np.ones_like(x) if y is None else np.ascontiguousarray(y, dtype=np.float64)
        out = np.empty_like(x)
        p = [a.ctypes.data_as(ctypes.c_void_p) for a in (x, y, out)]
        assert f({"rcp": 0, "sqrt": 1, "div": 2}[op], *p, x.size) == 0
        return out

    return ev


def operands(lo, hi):
    """Every exponent of [lo, hi], with mantissas at and beside powers of two, at
    the ends of 24 bits, and random ones."""
    g = np.random.default_rng(3)
    e = np.arange(lo, hi + 1)
    m = [1.0, 1 + 2.0**-52, 2 - 2.0**-52, 1.5, 1 + 2.0**-23, 1 + 2.0**-23 - 2.0**-52, 2 - 2.0**-23, 2 - 2.0**-24]
    m = np.concatenate([np.tile(m, (e.size, 1)), 1 + g.random((e.size, 8))], axis=1)
    with np.errstate(over="ignore"):
        return np.ldexp(m, e[:, None]).ravel()


def ulps(got, exact):
    """|got - exact| in units of the last place of exact (a Fraction > 0)."""
    n, d = exact.numerator, exact.denominator
    e = n.bit_length() - d.bit_length()
    if Fraction(2) ** e > exact:
        e -= 1
    return abs(Fraction(got) - exact) / Fraction(2) ** (e - 52)


IN = 119  # exponents well inside the FP32 start's range, 2^-120 to 2^120


def test_reciprocal(ev):
    x = operands(-IN, IN)
    x[::3] *= -1
    r = ev("rcp", x)
    assert max(ulps(abs(float(a)), 1 / abs(Fraction(float(b)))) for a, b in zip(r, x)) <= Fraction("0.501")
    assert np.array_equal(np.signbit(r), np.signbit(x))


def test_root(ev):
    x = operands(-IN, IN)
    r = ev("sqrt", x)
    half = Fraction("0.501")
    for a, b in zip(r, x):
        a, b = Fraction(float(a)), Fraction(float(b))
        u = Fraction(float(np.spacing(float(a)))) * half
        assert (a - u) ** 2 <= b <= (a + u) ** 2


def test_quotient(ev):
    d = operands(-59, 59)  # the range of its FP32 start, 2^-60 to 2^60
    g = np.random.default_rng(4)
    n = np.ldexp(1 + g.random(d.size), g.integers(-126, 128, d.size))  # sums of FP32 values
    d[::3] *= -1
    q = ev("div", n, d)
    assert max(ulps(abs(float(a)), Fraction(float(b)) / abs(Fraction(float(c)))) for a, b, c in zip(q, n, d)) <= Fraction("0.501")
    assert np.array_equal(ev("div", np.zeros(4), np.array([1.0, -3.0, 1e-10, 2e17])), np.zeros(4))


def test_operands_beyond_the_fp32_start_take_the_ieee_operation(ev):
    far = np.concatenate([operands(-1074, -122), operands(122, 1023)])
    far = far[np.isfinite(far) & (far > 0)]
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan])
    with np.errstate(all="ignore"):
        for x in (far, -far, special):
            assert np.array_equal(ev("rcp", x), 1.0 / x, equal_nan=True)
            assert np.array_equal(ev("sqrt", x), np.sqrt(x), equal_nan=True)
            assert np.array_equal(np.signbit(ev("rcp", special[:4])), np.signbit(1.0 / special[:4]))
        neg = -operands(-IN, IN)
        assert np.all(np.isnan(ev("sqrt", neg)))
        d = np.concatenate([operands(-1000, -62), operands(62, 1000), special, [1e-300]])
        n = np.full(d.size, 0.7)
        assert np.array_equal(ev("div", n, d), n / d, equal_nan=True)


def test_the_switch_of_range(ev):
    """On both sides of 2^-120, 2^120 (reciprocal, root) and 2^-60, 2^60 (quotient)."""
    for op, k in (("rcp", 120), ("sqrt", 120), ("div", 60)):
        x = np.concatenate([operands(-k - 2, -k + 2), operands(k - 2, k + 2)])
        one = np.full(x.size, 0.9)
        r = ev(op, x) if op != "div" else ev(op, one, x)
        ref = {"rcp": lambda: 1 / x, "sqrt": lambda: np.sqrt(x), "div": lambda: one / x}[op]()
        assert np.max(np.abs(r - ref) / np.spacing(ref)) <= 1
