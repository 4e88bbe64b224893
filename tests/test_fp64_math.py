"""FP64 reciprocal and roots by integers (fp64_math.cuh), as the host compiler builds them: within the stated
0.52 units in the last place of values formed in extended precision, over mantissas next to 1 and 2, random ones
and all exponents; special arguments as the language's operations give them."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include <math.h>
#include "fp64_math.cuh"
extern "C" void math(const double* a, double* r, long long n) {
  for (long long i = 0; i < n; ++i) {
    r[i] = flexi::fp64_rcp(a[i]);
    r[n + i] = flexi::fp64_sqrt(a[i]);
    r[2 * n + i] = flexi::fp64_rsqrt(a[i]);
  }
}
"""


def arguments(rng, n, lo, hi):
    """Values of both halves of the mantissa range and of exponents lo to hi - 1."""
    m = 1.0 + rng.random(n)
    k = n // 8
    m[:k] = 1.0 + rng.integers(0, 64, k) * 2.0 ** -52
    m[k:2 * k] = 2.0 - rng.integers(1, 64, k) * 2.0 ** -52
    return np.ldexp(m, rng.integers(lo, hi, n))


def ulps(got, ref):
    """|got - ref| in units in the last place of ref (long double)."""
    return np.abs((got.astype(np.longdouble) - ref)) / np.spacing(np.abs(ref).astype(np.float64)).astype(np.longdouble)


SPECIAL = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -5e-324, 2.2e-308, 1.7e308, -1.7e308, 2.0 ** 1022, 2.0 ** -1022,
                    2.0 ** 1021, 1.0, 4.0, -4.0, -1.0])


def reference(x):
    with np.errstate(all="ignore"):
        y = x.astype(np.longdouble)
        return 1 / y, np.sqrt(y), 1 / np.sqrt(y)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cuda = next((d for d in (os.environ.get("CUDA_HOME", ""), "/usr/local/cuda") if os.path.exists(os.path.join(d, "include", "cuda_runtime.h"))), None)
    if shutil.which("g++") is None or cuda is None:
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("fp64_math")
    src, out = d / "m.cpp", d / "m.so"
    src.write_text(SOURCE)
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-I", os.path.join(cuda, "include"), "-I",
                        os.path.join(ROOT, "paper_1910_02858_gb300", "csrc"), str(src), "-o", str(out)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    return ctypes.CDLL(str(out))


def _call(lib, x):
    x = np.ascontiguousarray(x)
    out = np.empty((3, x.size))
    p = ctypes.POINTER(ctypes.c_double)
    lib.math(x.ctypes.data_as(p), out.ctypes.data_as(p), ctypes.c_longlong(x.size))
    return out


def test_host_form_within_its_bound(lib):
    x = arguments(np.random.default_rng(1), 1_000_000, -1020, 1020)
    for got, ref in zip(_call(lib, x), reference(x)):
        assert ulps(got, ref).max() <= 0.52


def test_host_form_special_arguments(lib):
    with np.errstate(all="ignore"):
        expect = 1 / SPECIAL, np.sqrt(SPECIAL), 1 / np.sqrt(SPECIAL)
    for got, e in zip(_call(lib, SPECIAL), expect):
        assert np.array_equal(np.isnan(got), np.isnan(e)) and np.array_equal(np.isinf(got), np.isinf(e))
        f = np.isfinite(e)
        assert (np.abs(got[f] - e[f]) <= np.spacing(np.abs(e[f]))).all() and np.array_equal(np.signbit(got[f]), np.signbit(e[f]))
