"""csrc/reciprocal.cuh against CUDA's own 1 / x and 1 / sqrt(x) (IEEE division and square
root) and against the long-double value, over the exponents whose reciprocal is a normal
number, at random and at extreme significands, both signs.

Bounds, in units in the last place of the result.  recip: the iteration leaves the rounding
of its last fused multiply-add (1/2) and a remainder below 2^-3 (FP32: e^2 with e of 2^-22;
FP64: e^3 with e below 2^-19), so within 1 of the value and of its rounding, which is CUDA's
quotient.  rcp: the same in FP64; in FP32 the approximation as it is, documented to 2^-23 for
x in 1..2, i.e. two units (and half a unit more from CUDA's rounding).  inv_norm: FP64 rounds
x y (2^-54 of the result) and the last step, 1.5 units, so within 2, and within 3 of CUDA's
rounded quotient of a rounded root; FP32's rsqrtf is documented to 2."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include "reciprocal.cuh"
template <typename R> __global__ void k(const R *x, R *out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  out[i] = lbmk::recip(x[i]);
  out[n + i] = lbmk::rcp(x[i]);
  out[2 * n + i] = (R)1 / x[i];
  out[3 * n + i] = lbmk::inv_norm(x[i] < 0 ? -x[i] : x[i]);
  out[4 * n + i] = (R)1 / sqrt(x[i] < 0 ? -x[i] : x[i]);
}
template <typename R> int run(const R *x, R *out, int n) {
  R *d = nullptr, *o = nullptr;
  cudaError_t e = cudaMalloc(&d, sizeof(R) * n);
  if (e == cudaSuccess) e = cudaMalloc(&o, sizeof(R) * 5 * n);
  if (e == cudaSuccess) e = cudaMemcpy(d, x, sizeof(R) * n, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) k<R><<<(n + 255) / 256, 256>>>(d, o, n);
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpy(out, o, sizeof(R) * 5 * n, cudaMemcpyDeviceToHost);
  cudaFree(d);
  cudaFree(o);
  return (int)e;
}
extern "C" int run64(const double *x, double *out, int n) { return run(x, out, n); }
extern "C" int run32(const float *x, float *out, int n) { return run(x, out, n); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2302_04120_gb300 import build
    d = tmp_path_factory.mktemp("reciprocal")
    src, so = str(d / "r.cu"), str(d / "r.so")
    with open(src, "w") as fh:
        fh.write(SRC)
    subprocess.run([build._nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-I" + build.CSRC, "-shared", src, "-o", so],
                   check=True, capture_output=True)
    assert os.path.exists(so)
    return C.CDLL(so)


def _inputs(dtype):
    """Every exponent whose reciprocal is normal, 64 significands each, both signs."""
    lo, hi = (-1021, 1021) if dtype == np.float64 else (-125, 125)
    bits = 52 if dtype == np.float64 else 23
    rng = np.random.default_rng(3)
    e = np.repeat(np.arange(lo, hi), 64)
    m = rng.uniform(1.0, 2.0, e.size)
    m[0::64] = 1.0
    m[1::64] = 2.0 - 2.0 ** -bits
    m[2::64] = 1.0 + 2.0 ** -bits
    return np.ldexp(m.astype(dtype) * np.where(rng.random(e.size) < 0.5, -1, 1).astype(dtype), e).astype(dtype)


def _ulps(a, ref, dtype):
    unit = np.spacing(np.abs(ref.astype(dtype))).astype(np.longdouble)
    return float(np.max(np.abs(a.astype(np.longdouble) - ref) / unit))


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_against_cuda_and_long_double(lib, dtype):
    x = _inputs(dtype)
    n = x.size
    out = np.empty((5, n), dtype)
    f = lib.run64 if dtype == np.float64 else lib.run32
    assert f(x.ctypes.data_as(C.c_void_p), out.ctypes.data_as(C.c_void_p), n) == 0
    inv = 1 / x.astype(np.longdouble)
    root = 1 / np.sqrt(np.abs(x).astype(np.longdouble))
    cuda = out[2].astype(np.longdouble)
    got = {k: (_ulps(out[j], inv, dtype), _ulps(out[j], cuda, dtype)) for j, k in enumerate(("recip", "rcp"))}
    assert max(got["recip"]) <= 1.0, got
    assert max(got["rcp"]) <= (1.0 if dtype == np.float64 else 2.5), got
    ok = np.abs(x) > 1e-300  # FP64: smaller |g|^2 counts as zero
    got = dict(exact=_ulps(out[3][ok], root[ok], dtype), cuda=_ulps(out[3][ok], out[4][ok].astype(np.longdouble), dtype))
    assert got["exact"] <= 2.0 and got["cuda"] <= 3.0, got
    assert np.all(out[3][~ok] == 0)


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_norm_of_zero_and_nonfinite(lib, dtype):
    x = np.array([0.0, np.inf, np.nan, 1.0], dtype)
    out = np.empty((5, 4), dtype)
    f = lib.run64 if dtype == np.float64 else lib.run32
    assert f(x.ctypes.data_as(C.c_void_p), out.ctypes.data_as(C.c_void_p), 4) == 0
    assert out[3][0] == 0 and out[3][3] == 1  # no gradient, no normal
    assert not np.isfinite(out[0][0]) and np.isnan(out[0][2]) and out[0][3] == 1  # a bad cell stays one
