"""The scalar device functions of the kernels, compiled on their own and
compared with IEEE arithmetic over the whole range of their arguments."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "small_dense.cuh"
namespace gbcca {
void set_last_error(const std::string&) {}
std::atomic<long long> g_launches{0};
}
__global__ void rcp_k(const double* x, double* y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = gbcca::rcp_nr(x[i]);
}
__global__ void widen_k(const float* x, double* y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = gbcca::widen(x[i]);
}
extern "C" int widen(const float* x, double* y, int n) {
  widen_k<<<(n + 255) / 256, 256>>>(x, y, n);
  return (int)cudaDeviceSynchronize();
}
extern "C" int rcp(const double* x, double* y, int n) {
  rcp_k<<<(n + 255) / 256, 256>>>(x, y, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2106_12060_gb300 import build as b
    d = tmp_path_factory.mktemp("device_math")
    (d / "t.cu").write_text(SOURCE)
    subprocess.run([b.nvcc(), *b.ARCH, *b.FLAGS, "-I", b.CSRC, "-shared", "-o", str(d / "t.so"), str(d / "t.cu")],
                   check=True)
    return ctypes.CDLL(os.path.join(str(d), "t.so"))


def _call(f, x, out_dtype):
    import torch
    a = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    b = torch.from_numpy(np.zeros(len(x), out_dtype)).cuda()
    assert f(ctypes.c_void_p(a.data_ptr()), ctypes.c_void_p(b.data_ptr()), len(x)) == 0
    return b.cpu().numpy()


def test_reciprocal(lib):
    """Every exponent field (the guard's ends, subnormals, infinities and NaN
    among them), mantissas at the ends of their range and random ones, both
    signs: within one unit in the last place of IEEE division, and equal to it
    where the argument or the result is not normal."""
    rng = np.random.default_rng(0)
    ends = np.array([0, 1, 2, (1 << 29) - 1, 1 << 29, (1 << 51) - 1, 1 << 51, (1 << 52) - 2, (1 << 52) - 1])
    man = np.concatenate([np.broadcast_to(ends, (2048, len(ends))), rng.integers(0, 1 << 52, (2048, 500))], 1)
    bits = (np.arange(2048, dtype=np.uint64)[:, None] << np.uint64(52)) | man.astype(np.uint64)
    x = np.concatenate([bits.ravel(), bits.ravel() | np.uint64(1 << 63)]).view(np.float64)
    x = np.concatenate([x, 1.0 + rng.random(100000), np.float64(1.0) + np.arange(-2000, 2000) * 2.0 ** -52])
    got = _call(lib.rcp, x, np.float64)
    with np.errstate(all="ignore"):
        exp = 1.0 / x
        plain = ~np.isfinite(x) | ~np.isfinite(exp) | (np.abs(x) < 2.0 ** -1022) | (np.abs(exp) < 2.0 ** -1022)
    assert np.array_equal(got[plain], exp[plain], equal_nan=True)
    assert np.array_equal(np.signbit(got[plain & ~np.isnan(x)]), np.signbit(exp[plain & ~np.isnan(x)]))
    ulp = np.abs(got[~plain].view(np.int64) - exp[~plain].view(np.int64))
    assert ulp.max() <= 1


def test_widen(lib):
    """FP32 to FP64 by moving the bits: every exponent field (subnormals and
    infinities among them) with mantissas at the ends of their range, single
    bits and random ones, both signs: the same bits as a conversion; NaN stays
    NaN."""
    rng = np.random.default_rng(0)
    ends = np.concatenate([1 << np.arange(23), (1 << 23) - 1 - (1 << np.arange(23)), [0, (1 << 23) - 1]])
    man = np.concatenate([np.broadcast_to(ends, (256, len(ends))), rng.integers(0, 1 << 23, (256, 2000))], 1)
    bits = ((np.arange(256, dtype=np.uint32)[:, None] << np.uint32(23)) | man.astype(np.uint32)).ravel()
    x = np.concatenate([bits, bits | np.uint32(1 << 31)]).view(np.float32)
    got = _call(lib.widen, x, np.float64)
    nan = np.isnan(x)
    assert np.all(np.isnan(got[nan]))
    assert np.array_equal(got[~nan].view(np.int64), x[~nan].astype(np.float64).view(np.int64))
