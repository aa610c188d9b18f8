"""The FP64 functions of csrc/rt_math.cuh lose no precision to their tables and
FP32 terms: little but the rounding of the result itself (at most 1/2 ulp,
1/sqrt(12) ulp rms) is left, against extended precision, the same source
compiled as C++.  What may be added to it: the rounding of the part beyond the
exact one, 2^-63 against a result above 0.0117 (an ulp of 2^-59) or 2^-62 above
0.0156 (2^-58) and above 0.034 (2^-57), and the FP32 tails of the series, 7.5e-8
of r^5 / 6 with |r| <= 3/256 and of r^5 / 720 with |r| <= 0.035 (0.03 ulp): at
most 1/10 ulp."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1410_1629_gb300", "csrc")
EXTRA = 0.1


@pytest.fixture(scope="module")
def math_lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("math")
    src = d / "shim.cpp"
    calls = {"exp": "rtk::one_minus_exp(x[i])", "log": "rtk::neg_log_one_minus(x[i])", "up": "rtk::exp_minus_one(x[i])",
             "bose": "rtk::bose(x[i], 3.7)"}
    src.write_text(f'#include "{CSRC}/rt_math.cuh"\n' + "".join(
        f'extern "C" void run_{k}(const double* x, double* y, long n) {{ for (long i = 0; i < n; ++i) y[i] = {c}; }}\n'
        for k, c in calls.items()))
    so = d / "shim.so"
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", str(src), "-o", str(so)], check=True)
    return ctypes.CDLL(str(so))


def _errors(lib, which, x, ref):
    """Error in ulps of the result's binade."""
    y = np.empty_like(x)
    getattr(lib, f"run_{which}")(ctypes.c_void_p(x.ctypes.data), ctypes.c_void_p(y.ctypes.data), ctypes.c_long(x.size))
    assert np.all(np.isfinite(y))
    return ((y.astype(np.longdouble) - ref) / np.spacing(np.minimum(ref.astype(np.float64), y))).astype(np.float64)


def _arguments(lo, hi, step, n):
    """Spread over the logarithm, and both sides of the tables' borders."""
    x = np.exp(np.random.default_rng(17).uniform(np.log(lo), np.log(hi), n))
    k = np.arange(1, 200_000) * step
    k = k[(k > lo) & (k < hi)][:5000]
    return np.concatenate([x, np.nextafter(k, 0), k, np.nextafter(k, np.inf)])


RANGES = [("exp", 1e-12, 1e-3), ("exp", 1e-3, 0.01), ("exp", 0.01, 0.1), ("exp", 0.1, 1.0), ("exp", 1.0, 10.0),
          ("exp", 10.0, 37.0), ("exp", 37.0, 38.0), ("log", 1e-12, 1e-3), ("log", 1e-3, 0.02), ("log", 0.02, 0.5),
          ("log", 0.5, 0.999999), ("up", 1e-12, 1e-3), ("up", 1e-3, 0.01), ("up", 0.01, 0.7), ("up", 0.7, 1.4),
          ("up", 1.4, 40.0), ("up", 40.0, 709.0), ("up", 709.0, 709.78271289338397)]


@pytest.mark.parametrize("which,lo,hi", RANGES)
def test_little_but_the_own_rounding(math_lib, which, lo, hi):
    x = _arguments(lo, hi, 1.0 / 256.0 if which == "log" else np.log(2.0) / 256.0, 200_000)
    xl = x.astype(np.longdouble)
    ref = {"exp": lambda: -np.expm1(-xl), "log": lambda: -np.log1p(-xl), "up": lambda: np.expm1(xl)}[which]()
    err = _errors(math_lib, which, x, ref)
    assert np.abs(err).max() <= 0.5 + EXTRA
    assert np.sqrt(np.mean(err[:200_000] ** 2)) <= np.sqrt(1.0 / 12.0 + EXTRA ** 2)


@pytest.mark.parametrize("lo,hi", [(1e-9, 1e-3), (1e-3, 0.7), (0.7, 40.0), (40.0, 700.0), (700.0, 708.0)])
def test_emission_factor(math_lib, lo, hi):
    """a / (exp(x) - 1): the divisor's error (doubled where the quotient's binade
    begins) and the quotient's rounding."""
    x = _arguments(lo, hi, np.log(2.0) / 256.0, 200_000)
    ref = np.longdouble(3.7) / np.expm1(x.astype(np.longdouble))
    assert np.abs(_errors(math_lib, "bose", x, ref)).max() <= 0.5 + 2.0 * (0.5 + EXTRA)
