"""The double-word building blocks of the FP64-accurate path, alone: a kernel compiled here from the
library's headers runs them on given operands, against exactly rounded sums."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SRC = r"""
#include "fe_reduce.cuh"
// sums of k products a[j, t] b[j, t] per thread t of T
__global__ void k_sums(const float* a, const float* b, int k, int T, double* out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= T) return;
  Acc<float> s;
  for (int j = 0; j < k; ++j) s.add_prod(a[(size_t)j * T + t], b[(size_t)j * T + t]);
  out[t] = s.value();
}
extern "C" int sums(const float* a, const float* b, int k, int T, double* out) {
  k_sums<<<(T + 127) / 128, 128>>>(a, b, k, T, out);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2607_02335_gb300 import build as B
    d = tmp_path_factory.mktemp("arith")
    src, so = os.path.join(d, "arith.cu"), os.path.join(d, "arith.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([B.NVCC, *B.ARCH, *B.FLAGS, "-shared", "-o", so, src], check=True)
    return ctypes.CDLL(so)


def ptr(t):
    return ctypes.c_void_p(t.data_ptr())


@pytest.mark.parametrize("k", [1, 16, 2560])
@pytest.mark.parametrize("positive", [True, False])
def test_thread_sum_of_products(lib, k, positive):
    """A normalised double-word sum adds an error of the order of 2^-48 of the running sum per term, of
    either sign: on average over the threads at most 2^-48 sqrt(k / 3) of the sum of |terms| (a random walk
    whose steps grow with the running sum), plus the rounding of the result."""
    T = 512
    rng = np.random.default_rng(k)
    a = rng.standard_normal((k, T)).astype(np.float32)
    b = a if positive else rng.standard_normal((k, T)).astype(np.float32)
    da, db, out = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), torch.empty(T, dtype=torch.float64, device="cuda")
    assert lib.sums(ptr(da), ptr(db), k, T, ptr(out)) == 0
    prod = a.astype(np.float64) * b.astype(np.float64)  # exact: 24-bit factors
    ref = np.array([math.fsum(prod[:, t]) for t in range(T)])
    err = np.abs(out.cpu().numpy() - ref) / np.abs(prod).sum(0)
    assert err.mean() <= 2.0 ** -48 * math.sqrt(k / 3.0) + 2.0 ** -52, err.mean()
