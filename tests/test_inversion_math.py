"""The FP64 exponential and logarithm of the forced-scattering inversion
(csrc/rt_math.cuh) against extended precision: the same source compiled as
C++.  The bound is the sum of the roundings on the way to the result: the
result's own (1/2 ulp), and for the series' leading term its argument's, its
own and its scale's (1/2 ulp each of a value at most the result)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1410_1629_gb300", "csrc")
ULP = 2.0


@pytest.fixture(scope="module")
def math_lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("math")
    src = d / "shim.cpp"
    src.write_text(f'#include "{CSRC}/rt_math.cuh"\n'
                   'extern "C" void run_bose(const double* x, double* y, long n) {\n'
                   "  for (long i = 0; i < n; ++i) y[i] = rtk::bose(x[i]);\n}\n"
                   'extern "C" void run(const double* x, double* e, double* l, long n) {\n'
                   "  for (long i = 0; i < n; ++i) {\n"
                   "    if (e) e[i] = rtk::one_minus_exp(x[i]);\n"
                   "    if (l) l[i] = rtk::neg_log_one_minus(x[i]);\n  }\n}\n")
    so = d / "shim.so"
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", str(src), "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))
    lib.run_bose.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_long]
    lib.run.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_long]
    return lib


def _call(lib, x, which):
    x = np.ascontiguousarray(x, dtype=np.float64)
    out = np.empty_like(x)
    lib.run(x.ctypes.data, out.ctypes.data if which == "exp" else None, out.ctypes.data if which == "log" else None, x.size)
    return out


@pytest.mark.parametrize("which,lo,hi", [("exp", 1e-12, 1e-3), ("exp", 1e-3, 0.1), ("exp", 0.1, 40.0), ("exp", 40.0, 1e4),
                                         ("log", 1e-12, 1e-3), ("log", 1e-3, 0.02), ("log", 0.02, 0.999999)])
def test_against_extended_precision(math_lib, which, lo, hi):
    rng = np.random.default_rng(11)
    x = np.exp(rng.uniform(np.log(lo), np.log(hi), 200_000))
    if which == "exp":  # the borders of the table's intervals, and the two ends
        k = np.arange(1, 4000) * (np.log(2.0) / 256.0)
        x = np.concatenate([x, np.nextafter(k, 0), k, np.nextafter(k, 100), [0.0, 1e-300, 64.0, np.nextafter(64.0, 65.0)]])
        ref = -np.expm1(-x.astype(np.longdouble))
    else:
        k = np.arange(1, 256) / 256.0
        x = np.concatenate([x, np.nextafter(k, 0), k, np.nextafter(k, 1), [0.0, 1e-300, 2.0 ** -54, 1 - 2.0 ** -33, 1 - 2.0 ** -53]])
        ref = -np.log1p(-x.astype(np.longdouble))
    got = _call(math_lib, x, which)
    err = np.abs(got.astype(np.longdouble) - ref) / np.spacing(np.maximum(ref.astype(np.float64), 1e-300))
    assert np.all(np.isfinite(got)) and float(err.max()) <= ULP


def test_bose_against_extended_precision(math_lib):
    """1 / (exp(x) - 1): the leading roundings are those of 1 - exp(-x) and
    exp(-x) (2 ulp each) and of the quotient; zero where exp(x) overflows."""
    rng = np.random.default_rng(12)
    x = np.concatenate([np.exp(rng.uniform(np.log(1e-9), np.log(700.0), 200_000)), np.arange(1, 4000) * (np.log(2.0) / 256.0)])
    y = np.empty_like(x)
    math_lib.run_bose(x.ctypes.data, y.ctypes.data, x.size)
    ref = 1.0 / np.expm1(x.astype(np.longdouble))
    assert float((np.abs(y.astype(np.longdouble) - ref) / ref).max()) <= 5.0 * 2.0 ** -53
    ends = np.array([709.0, 709.7, 709.79, 1e4, np.inf, np.nan])
    y = np.empty_like(ends)
    math_lib.run_bose(ends.ctypes.data, y.ctypes.data, ends.size)
    np.testing.assert_allclose(y[:2], 1.0 / np.expm1(ends[:2]), rtol=1e-15)
    assert np.all(y[2:] == 0.0)
