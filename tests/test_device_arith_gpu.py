"""The double-word building blocks of the FP64-accurate path, alone: kernels compiled here from the library's
headers run them on given operands, against exactly rounded sums and against the scalar operations."""
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
// per lane pair t: out[0..1] fl(fl(a b) + c); out[2..5] dw2_prod and out[6..9] dw2_mac with a table
// coefficient (high parts, low parts); out[10..17] the same with a run-time factor; the scalar forms after them
__global__ void k_packed(const float* in, int T, float* out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= T) return;
  float v[6][2];  // coefficient, value, accumulator: high, low
  for (int k = 0; k < 6; ++k)
    for (int l = 0; l < 2; ++l) v[k][l] = in[((size_t)k * T + t) * 2 + l];
  f2 p[6];
  for (int k = 0; k < 6; ++k) p[k] = f2_pack(v[k][0], v[k][1]);
  const dw2 x = {p[2], p[3]}, acc = {p[4], p[5]}, r = {p[0], p[1]};
  const dw2c c = {p[0], f2_neg(p[0]), f2_neg(p[1])};
  float* o = out + (size_t)t * 36;
  auto put = [&](int k, f2 w) { const float2 u = f2_unpack(w); o[2 * k] = u.x; o[2 * k + 1] = u.y; };
  put(0, f2_add(f2_mul(p[0], p[2]), p[4]));
  const dw2n a = dw2_prod(c, x), b = dw2_mac(dw2n{p[4], f2_neg(p[5])}, c, x);
  put(1, a.h), put(2, f2_neg(a.nl)), put(3, b.h), put(4, f2_neg(b.nl));
  const dw2 d = dw2_prod(r, x), e = dw2_mac(acc, r, x);
  put(5, d.h), put(6, d.l), put(7, e.h), put(8, e.l);
  for (int l = 0; l < 2; ++l) {
    const dw cs = {v[0][l], v[1][l]}, xs = {v[2][l], v[3][l]};
    const dw ps = dw_prod(cs, xs), ms = dw_mac({v[4][l], v[5][l]}, cs, xs);
    float* s = o + 18 + l;
    s[0] = __fadd_rn(__fmul_rn(cs.h, xs.h), v[4][l]);
    s[2] = s[10] = ps.h, s[4] = s[12] = ps.l, s[6] = s[14] = ms.h, s[8] = s[16] = ms.l;
  }
}
extern "C" int packed(const float* in, int T, float* out) {
  k_packed<<<(T + 127) / 128, 128>>>(in, T, out);
  return (int)cudaDeviceSynchronize();
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


def test_packed_operations_are_the_scalar_ones(lib):
    """Every half of a packed product, product and sum, and multiply-add has the bits of the scalar
    operations.  The product is where a compiler could go wrong: were it contracted with the sum after it,
    the error-free sums would lose the product's rounding error."""
    T = 4096
    rng = np.random.default_rng(1)
    hi = rng.standard_normal((3, T, 2)).astype(np.float32)
    lo = (hi * rng.uniform(-1, 1, hi.shape) * 2.0 ** -25).astype(np.float32)
    v = np.stack([hi[0], lo[0], hi[1], lo[1], hi[2], lo[2]])
    v[4, : T // 2] = -(v[0] * v[2])[: T // 2]  # sums that cancel: a contracted product would show in every bit
    out = torch.empty((T, 36), dtype=torch.float32, device="cuda")
    d = torch.from_numpy(v).cuda()
    assert lib.packed(ptr(d), T, ptr(out)) == 0
    o = out.cpu().numpy()
    ref = (v[0] * v[2]) + v[4]  # numpy rounds the product and the sum
    assert np.array_equal(o[:, 0:2], ref) and np.array_equal(o[:, 18:20], ref)
    assert np.array_equal(o[:, :18], o[:, 18:])
