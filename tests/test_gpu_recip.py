"""The float64 reciprocal of the kernels (csrc/common.cuh): within two units in the last place of
1 / x over every exponent, random and extreme mantissas and both signs, and the division's own
result where the quick form does not apply (zeros, subnormals, infinities, NaN, results near
the subnormal range). A kernel of its own is compiled against the header.
"""
import ctypes
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

KERNEL = r"""
#include "common.cuh"
__global__ void k(long long n, const double* x, double* y) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) y[i] = deer::recip(x[i]);
}
extern "C" int run(long long n, const void* x, void* y) {
  if (n > 0) k<<<(unsigned)((n + 255) / 256), 256>>>(n, (const double*)x, (double*)y);
  const cudaError_t e = cudaDeviceSynchronize();
  return e != cudaSuccess ? (int)e : (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def recip(tmp_path_factory):
    from paper_2603_16850_gb300 import _build
    d = tmp_path_factory.mktemp("recip")
    (d / "recip.cu").write_text(KERNEL)
    subprocess.run([_build._nvcc(), *_build.NVCC_FLAGS, "-shared", "-o", str(d / "librecip.so"),
                    str(d / "recip.cu")], check=True, capture_output=True)
    lib = ctypes.CDLL(str(d / "librecip.so"))
    lib.run.argtypes = [ctypes.c_longlong, ctypes.c_void_p, ctypes.c_void_p]

    def f(bits):
        x = torch.tensor(bits.astype(np.int64), device="cuda").view(torch.float64)
        y = torch.empty_like(x)
        torch.cuda.synchronize()
        assert lib.run(x.numel(), x.data_ptr(), y.data_ptr()) == 0
        return x.cpu().numpy(), y.cpu().numpy()

    return f


def test_within_two_ulp(recip):
    rng = np.random.default_rng(0)
    m = np.concatenate([rng.integers(0, 1 << 52, 2000, dtype=np.uint64),
                        np.array([0, 1, 2, 3, (1 << 29) - 1, 1 << 29, (1 << 51), (1 << 51) - 1,
                                  (1 << 52) - 2, (1 << 52) - 1], dtype=np.uint64)])
    e = np.arange(1, 2044, dtype=np.uint64)  # normal x with the quick form
    for sign in (0, 1):
        bits = ((e[:, None] << np.uint64(52)) | m[None, :] | np.uint64(sign << 63)).reshape(-1)
        x, y = recip(bits.view(np.int64))
        ref = 1.0 / x
        ulps = np.abs(y.view(np.int64) - ref.view(np.int64))
        assert ulps.max() <= 2


def test_values_that_take_the_division(recip):
    rng = np.random.default_rng(1)
    m = np.concatenate([rng.integers(0, 1 << 52, 200, dtype=np.uint64),
                        np.array([0, 1, (1 << 52) - 1], dtype=np.uint64)])
    e = np.array([0, 2044, 2045, 2046, 2047], dtype=np.uint64)
    bits = ((e[:, None] << np.uint64(52)) | m[None, :]).reshape(-1)
    bits = np.concatenate([bits, bits | np.uint64(1 << 63)])
    x, y = recip(bits.view(np.int64))
    with np.errstate(all="ignore"):
        ref = 1.0 / x
    same = (y.view(np.int64) == ref.view(np.int64)) | (np.isnan(y) & np.isnan(ref))
    assert same.all()
