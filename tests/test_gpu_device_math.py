"""Device functions of the FP64 form's integer arithmetic, each against a value of higher precision
or the FP64 expression that it stands for: fp64_rcp, fp64_sqrt, fp64_rsqrt, dg_div (fp64_math.cuh)
and fx_visc_normal (fx.cuh).  A small library of wrapper kernels is compiled from the headers."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "dg_common.cuh"
#include "fx.cuh"
using namespace flexi;
__global__ void k_math(const double* a, const double* b, double* r, long long n) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  r[i] = fp64_rcp(a[i]);
  r[n + i] = fp64_sqrt(a[i]);
  r[2 * n + i] = fp64_rsqrt(a[i]);
  r[3 * n + i] = dg_div(a[i], b[i]);
}
__global__ void k_visc(const double* in, double* fixed, double* fp64, long long n) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double W[5], G[15], nv[3], f[5];
  for (int c = 0; c < 5; ++c) W[c] = in[c * n + i];
  for (int c = 0; c < 15; ++c) G[c] = in[(5 + c) * n + i];
  for (int c = 0; c < 3; ++c) nv[c] = in[(20 + c) * n + i];
  Phys<double> ph{};
  ph.mu = 0.75;
  ph.lam_th = 1.5;
  const double ir = 1.0 / W[0];
  fx_visc_normal(W, ir, G, nv, fx_normal(nv), ph, f);
  for (int c = 0; c < 5; ++c) fixed[c * n + i] = f[c];
  visc_normal(W, ir, G, nv, ph, f);
  for (int c = 0; c < 5; ++c) fp64[c * n + i] = f[c];
}
template <typename Launch>
static int run(const double* in, long long nin, double* out, long long nout, Launch launch) {
  double *di = nullptr, *dout = nullptr;
  int err = cudaMalloc(&di, nin * 8);
  if (!err) err = cudaMalloc(&dout, nout * 8);
  if (!err) err = cudaMemcpy(di, in, nin * 8, cudaMemcpyHostToDevice);
  if (!err) {
    launch(di, dout);
    err = cudaGetLastError();
  }
  if (!err) err = cudaMemcpy(out, dout, nout * 8, cudaMemcpyDeviceToHost);
  cudaFree(di);
  cudaFree(dout);
  return err;
}
extern "C" int math(const double* in, double* out, long long n) {
  return run(in, 2 * n, out, 4 * n, [n](double* i, double* o) { k_math<<<(unsigned)((n + 127) / 128), 128>>>(i, i + n, o, n); });
}
extern "C" int visc(const double* in, double* out, long long n) {
  return run(in, 23 * n, out, 10 * n, [n](double* i, double* o) { k_visc<<<(unsigned)((n + 127) / 128), 128>>>(i, o, o + 5 * n, n); });
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_1910_02858_gb300 import build

    d = tmp_path_factory.mktemp("device_math")
    src, out = d / "device_math.cu", d / "device_math.so"
    src.write_text(SOURCE)
    cmd = [build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC", "-shared", "-I",
           build.CSRC, "-I", os.path.join(build.HERE, "..", "include"), str(src), "-o", str(out)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    return ctypes.CDLL(str(out))


def _call(fn, rows, nout):
    x = np.ascontiguousarray(np.stack(rows))
    out = np.empty((nout, x.shape[1]))
    p = ctypes.POINTER(ctypes.c_double)
    assert fn(x.ctypes.data_as(p), out.ctypes.data_as(p), ctypes.c_longlong(x.shape[1])) == 0
    return out


def test_viscous_flux_of_unequal_gradients(lib):
    """Each stress sum within the roundings of its own terms: mu times at most ten roundings of 2^-53 (FP64) plus the
    fixed-point quantum, less than two more, relative to sum_d (|G_dc| + |G_cd|) |n_d| + 2/3 sum |G_kk| |n_c|."""
    rng = np.random.default_rng(3)
    n = 200_000
    W = [rng.uniform(0.5, 2, n), *rng.uniform(-1, 1, (3, n)), rng.uniform(0.5, 2, n)]
    G = rng.uniform(-1, 1, (15, n)) * 2.0 ** rng.integers(-40, 41, (15, n))
    nv = rng.standard_normal((3, n)) * 2.0 ** rng.integers(-40, 1, (3, n))
    nv[:, : n // 4] = np.eye(3)[rng.integers(0, 3, n // 4)].T  # faces along the axes
    nv /= np.sqrt((nv * nv).sum(0))
    out = _call(lib.visc, [*W, *G, *nv], 10)
    g = np.abs(G.reshape(3, 5, n)[:, 1:4])  # [d, c]
    div = g[0, 0] + g[1, 1] + g[2, 2]
    T = np.stack([0.75 * (((g[:, c] + g[c]) * np.abs(nv)).sum(0) + 2.0 / 3.0 * div * np.abs(nv[c])) for c in range(3)])
    for c in range(3):
        assert (np.abs(out[1 + c] - out[6 + c]) <= 12 * 2.0 ** -53 * T[c]).all(), c
    heat = 1.5 / W[0] * (np.abs(G[4::5]) + W[4] / W[0] * np.abs(G[0::5])).T.dot(np.ones(3))
    T4 = (T * np.abs(W[1:4])).sum(0) + heat
    assert (np.abs(out[4] - out[9]) <= 16 * 2.0 ** -53 * T4).all()


def test_viscous_flux_special_values(lib):
    """Zero gradients, an infinity, a NaN and gradients beyond the fixed-point range: as the FP64 sums."""
    rng = np.random.default_rng(4)
    G = rng.uniform(-1, 1, (15, 5))
    G[:, 0] = 0.0
    G[2, 1], G[8, 2], G[3, 3] = np.inf, np.nan, 2.0 ** 950
    nv = np.array([0.6, 0.0, 0.8]).reshape(3, 1).repeat(5, 1)
    out = _call(lib.visc, [np.ones(5), *rng.uniform(-1, 1, (3, 5)), np.ones(5), *G, *nv], 10)
    assert np.array_equal(out[:5, :4], out[5:, :4], equal_nan=True)
    assert (out[:4, 0] == 0.0).all()


def test_reciprocal_roots_and_quotient(lib):
    """The device form, whose FP32 seeds differ from the host's: 0.52 units in the last place for the three functions,
    and one for the quotient with its residual taken out, over all exponents whose results are normal."""
    from test_fp64_math import arguments, reference, ulps

    rng = np.random.default_rng(2)
    n = 1_000_000
    a, b = arguments(rng, n, -1020, 1020), arguments(rng, n, -500, 500)
    out = _call(lib.math, [a, b], 4)
    for got, ref in zip(out[:3], reference(a)):
        assert ulps(got, ref).max() <= 0.52
    q = a.astype(np.longdouble) / b.astype(np.longdouble)
    ok = (np.abs(q) > 2.0 ** -1021) & (np.abs(q) < 2.0 ** 1023)
    assert ulps(out[3][ok], q[ok]).max() <= 1.0


def test_special_arguments(lib):
    from test_fp64_math import SPECIAL

    a, b = (x.ravel() for x in np.meshgrid(SPECIAL, SPECIAL))
    out = _call(lib.math, [a, b], 4)
    with np.errstate(all="ignore"):
        expect = 1 / a, np.sqrt(a), 1 / np.sqrt(a), a / b
    for got, e in zip(out, expect):
        assert np.array_equal(np.isnan(got), np.isnan(e)) and np.array_equal(np.isinf(got), np.isinf(e))
        f = np.isfinite(e)
        assert (np.abs(got[f] - e[f]) <= np.spacing(np.abs(e[f]))).all()
