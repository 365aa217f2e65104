"""The reciprocals of the element kernels (csrc/elem.cuh) one by one: FP32 recip rounds correctly, the
FP64 recip and inv_sqrt (a hardware estimate and one third-order step) stay within their bounds over
the normal numbers, and around powers of two.

Bounds in units of the last place, with e the relative error of the estimate (2^-19 or less) and
2^-53 of each rounding. recip: the step leaves e^3 = 2^-57 (0.06 units) and rounds once (0.5):
0.6 from the exact value, so at most one number beside the correctly rounded one. inv_sqrt: the
step leaves 5/16 e^3 (0.04), the product x y of its residual is rounded (0.5) and so is the result
(0.5): 1.1."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SRC = r"""
#include "elem.cuh"
template <class T>
__global__ void k(const T* x, T* r, T* s, long n) {
  const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (i < n) { r[i] = chns::recip(x[i]); s[i] = chns::inv_sqrt(x[i]); }
}
template <class T>
int run(const T* x, T* r, T* s, long n) {
  k<T><<<(unsigned)((n + 255) / 256), 256>>>(x, r, s, n);
  return (int)cudaDeviceSynchronize();
}
extern "C" int run32(const float* x, float* r, float* s, long n) { return run(x, r, s, n); }
extern "C" int run64(const double* x, double* r, double* s, long n) { return run(x, r, s, n); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2107_05123_gb300 import build as b
    d = tmp_path_factory.mktemp("recip")
    src, out = d / "recip.cu", d / "recip.so"
    src.write_text(SRC)
    subprocess.run([b._nvcc(), *b.ARCH, *b.FLAGS, "-shared", "-I", b.CSRC, "-I",
                    os.path.join(os.path.dirname(b.HERE), "include"), "-o", str(out), str(src)],
                   check=True, capture_output=True)
    return ctypes.CDLL(str(out))


def _eval(lib, x):
    xd = torch.as_tensor(x, device="cuda")
    r, s = torch.empty_like(xd), torch.empty_like(xd)
    fn = lib.run32 if x.dtype == np.float32 else lib.run64
    assert fn(*(ctypes.c_void_p(t.data_ptr()) for t in (xd, r, s)), ctypes.c_long(x.size)) == 0
    return r.cpu().numpy(), s.cpu().numpy()


def _numbers(dtype, lo, hi):
    """Random mantissas over the exponents lo..hi, and each power of two with its neighbours."""
    rng = np.random.default_rng(3)
    e = rng.integers(lo, hi, 1 << 20)
    x = np.ldexp(rng.uniform(1.0, 2.0, e.size).astype(dtype), e)
    p = np.ldexp(dtype(1.0), np.arange(lo + 1, hi))
    near = [np.nextafter(p, dtype(0)), p, np.nextafter(p, dtype(np.inf))]
    unit = rng.uniform(1.0, 4.0, 1 << 20).astype(dtype)
    return np.concatenate([x, *near, unit]).astype(dtype)


def test_recip_fp32_rounds_correctly(lib):
    x = _numbers(np.float32, -126, 125)
    x = np.concatenate([x, -x])
    r, _ = _eval(lib, x)
    assert np.array_equal(r, np.float32(1.0) / x)


def test_recip_fp64(lib):
    x = _numbers(np.float64, -1022, 1020)
    x = np.concatenate([x, -x])
    r, _ = _eval(lib, x)
    exact = 1.0 / x
    assert np.abs(r.view(np.int64) - exact.view(np.int64)).max() <= 1
    assert np.isnan(_eval(lib, np.array([np.nan]))[0]).all()


def test_inv_sqrt_fp64(lib):
    x = _numbers(np.float64, -1022, 1023)
    _, s = _eval(lib, x)
    exact = 1 / np.sqrt(x.astype(np.longdouble))
    err = np.abs(s.astype(np.longdouble) - exact) / np.spacing(exact.astype(np.float64))
    assert float(err.max()) <= 1.1
    assert _eval(lib, np.array([np.inf]))[1][0] == 0.0
    assert np.isnan(_eval(lib, np.array([np.nan]))[1]).all()
