"""The table functions of the synthetic solve (csrc/special.cuh) and recip64
against 45-digit values: every table interval, the interval ends, the whole range
of binades, and the arguments that go to the library's functions.

Bounds, in units in the last place (u) of the result:
  exp_tab    0.5 for the final sum, 0.32 for the omitted r^6/720 (|r| <= ln 2/128, near
             the upper end of a binade), 0.03 for the rest: 0.85
  log_tab    0.55 u + 2^-58: r^7/7 with |r| < 2^-8 is 2^-58.8, the same near log x = 0, where the
             table value cancels e ln 2 and the error is absolute
  mills      4: the table's recursion (its errors are those of the compiled-in table), 0.5 for
             the final sum
  recip64    1: the second Newton step's rounding
  T^0.81     5 for 0.05 <= T <= 20: the exponent's rounding (up to 2^-52 of 2.4) and the two
             functions'"""
import ctypes
import decimal
import math
import subprocess
from decimal import Decimal as D

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "special.cuh"
using namespace gsis;
__global__ void k(int which, int n, const double* x, double* y) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double v = x[i];
    y[i] = which == 0 ? exp_tab(v) : which == 1 ? log_tab(v) : which == 2 ? mills(v) : which == 3 ? recip64(v)
         : which == 4 ? exp_tab(0.81 * log_tab(v)) : which == 5 ? exp(v) : log(v);
}
extern "C" int evaluate(int which, int n, const double* x, double* y) {
    double* d = nullptr;
    if (cudaMalloc(&d, 2 * n * sizeof(double)) != cudaSuccess) return 1;
    cudaMemcpy(d, x, n * sizeof(double), cudaMemcpyHostToDevice);
    k<<<(n + 127) / 128, 128>>>(which, n, d, d + n);
    cudaMemcpy(y, d + n, n * sizeof(double), cudaMemcpyDeviceToHost);
    cudaFree(d);
    return (int)cudaGetLastError();
}
"""
EXP, LOG, MILLS, RECIP, POW, LIBRARY_EXP, LIBRARY_LOG = range(7)


@pytest.fixture(scope="module")
def evaluate(tmp_path_factory):
    from paper_2501_02245_gb300 import build
    d = tmp_path_factory.mktemp("special")
    (d / "s.cu").write_text(SOURCE)
    subprocess.run([build._nvcc()] + build.ARCH + build.FLAGS + ["-I" + build.CSRC, "-shared", str(d / "s.cu"), "-o",
                                                                str(d / "s.so")], check=True)
    lib = ctypes.CDLL(str(d / "s.so"))
    p = ctypes.POINTER(ctypes.c_double)

    def f(which, x):
        x = np.ascontiguousarray(x, dtype=np.float64)
        y = np.empty_like(x)
        assert lib.evaluate(which, x.size, x.ctypes.data_as(p), y.ctypes.data_as(p)) == 0
        return y

    return f


def _worst(x, y, exact, absolute=0.0):
    """Largest error beyond `absolute`, in units in the last place of the exact value."""
    worst = 0.0
    with decimal.localcontext() as c:
        c.prec = 45
        for a, b in zip(x.tolist(), y.tolist()):
            e = exact(D(a))
            worst = max(worst, float((abs(D(b) - e) - D(absolute)) / D(math.ulp(float(e)))))
    return worst


def _spread(rng, lo, hi, n):
    return rng.uniform(lo, hi, n)


def test_exp(evaluate):
    r = np.random.default_rng(1)
    ends = (np.arange(-130, 130) + 0.5) * math.log(2.0) / 64.0   # where k changes
    x = np.concatenate([ends, np.nextafter(ends, 9e9), _spread(r, -3.0, 3.0, 1500), _spread(r, -50.0, 0.0, 1500),
                        _spread(r, -699.9, 699.9, 1000), [0.0, -0.0, 1e-300, -699.999, 699.999]])
    assert _worst(x, evaluate(EXP, x), lambda a: a.exp()) < 0.85
    far = np.array([700.0, -700.0, 745.0, -745.0, 710.0, -800.0, np.inf, -np.inf, np.nan])
    assert np.array_equal(evaluate(EXP, far), evaluate(LIBRARY_EXP, far), equal_nan=True)


def test_log(evaluate):
    r = np.random.default_rng(2)
    m = 1.0 + np.arange(128) / 128.0                              # where the table entry changes
    x = np.concatenate([m, np.nextafter(m, 0.0), np.nextafter(m, 9.0), m / 2.0, m * 4.0, _spread(r, 0.05, 20.0, 2500),
                        np.exp2(_spread(r, -1021.9, 1023.9, 500)), 1.0 + _spread(r, -1e-3, 1e-3, 300),
                        [np.nextafter(2.0, 0.0), 2.0 ** -1022, 1.7976931348623157e308]])
    assert _worst(x, evaluate(LOG, x), lambda a: a.ln(), 2.0 ** -58) < 0.55
    far = np.array([0.0, -0.0, -1.0, 5e-324, 1e-310, np.inf, -np.inf, np.nan])
    assert np.array_equal(evaluate(LOG, far), evaluate(LIBRARY_LOG, far), equal_nan=True)


def _half_erfcx(t):
    """(1/2) erfc(t/sqrt 2) exp(t^2/2), from 1/2 - the odd series of the normal integral."""
    with decimal.localcontext() as c:
        c.prec = 90   # exp(50) cancels at t = 10
        pi = D("3.14159265358979323846264338327950288419716939937510582097494459230781640628620899862803482534211706798")
        s = term = t
        n = 1
        while abs(term) > D(10) ** -85:   # sum of t^(2n+1) / (1 3 5 .. (2n+1)), times the density
            n += 2
            term = term * t * t / n
            s += term
        return (t * t / 2).exp() / 2 - s / (2 * pi).sqrt()


def test_mills(evaluate):
    r = np.random.default_rng(3)
    ends = (np.arange(640) + 0.5) / 64.0
    x = np.concatenate([ends, np.nextafter(ends, 9e9), _spread(r, 0.0, 10.0, 500), _spread(r, 0.0, 1.0, 300),
                        [0.0, 1e-300, 10.0, np.nextafter(10.0, 0.0)]])
    assert _worst(x, evaluate(MILLS, x), _half_erfcx) < 4.0
    far = np.array([np.nextafter(10.0, 20.0), 11.0, 1e300, np.inf])
    assert np.array_equal(evaluate(MILLS, far), np.repeat(evaluate(MILLS, np.array([10.0])), far.size))


def test_reciprocal(evaluate):
    r = np.random.default_rng(4)
    x = np.concatenate([_spread(r, 1.0, 2.0, 3000), np.exp2(_spread(r, -1021.0, 1021.0, 1000)) * r.choice([-1.0, 1.0], 1000),
                        [1.0, np.nextafter(2.0, 0.0), np.nextafter(1.0, 2.0), 2.0 ** -1022, 2.0 ** 1021]])
    assert _worst(x, evaluate(RECIP, x), lambda a: 1 / a) < 1.0


def test_power(evaluate):
    r = np.random.default_rng(5)
    x = np.concatenate([_spread(r, 0.05, 20.0, 2500), _spread(r, 0.9, 1.1, 500)])
    assert _worst(x, evaluate(POW, x), lambda a: (a.ln() * D(0.81)).exp()) < 5.0
