"""The reciprocals of recip.cuh against division, compiled here from the header."""
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SOURCE = r"""
#include "recip.cuh"
using namespace dnnmg;
// count of floats with bits [first, first + n) whose recip_ge1 is not 1.0f / x
__global__ void f32_kernel(unsigned first, unsigned n, unsigned long long* bad) {
  for (unsigned long long i = blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (unsigned long long)gridDim.x * blockDim.x) {
    const float x = __uint_as_float(first + (unsigned)i);
    if (__float_as_uint(recip_ge1(x)) != __float_as_uint(1.0f / x)) atomicAdd(bad, 1ull);
  }
}
__global__ void f64_kernel(const double* x, double* y, int n, int any) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = any ? recip64_any(x[i]) : recip64(x[i]);
}
extern "C" int compare_f32(unsigned first, unsigned n, unsigned long long* bad) {
  f32_kernel<<<1216, 256>>>(first, n, bad);
  return cudaDeviceSynchronize() != cudaSuccess;
}
extern "C" int recip_f64(const double* x, double* y, int n, int any) {
  f64_kernel<<<(n + 255) / 256, 256>>>(x, y, n, any);
  return cudaDeviceSynchronize() != cudaSuccess;
}
"""


@pytest.fixture(scope="module")
def native(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_07687_gb300 import build
    work = tmp_path_factory.mktemp("recip")
    src, so = work / "recip.cu", work / "librecip.so"
    src.write_text(SOURCE)
    subprocess.run([build._nvcc()] + build.ARCH + build.FLAGS +
                   ["-I", build.CSRC, "-shared", "-o", str(so), str(src)], check=True)
    assert os.path.exists(so)
    return ctypes.CDLL(str(so))


def test_fp32_reciprocal_equals_division(native):
    """Every float in [1, 2^125)."""
    bad = torch.zeros(1, dtype=torch.int64, device="cuda")
    first, end = 127 << 23, (127 + 125) << 23
    assert native.compare_f32(ctypes.c_uint(first), ctypes.c_uint(end - first),
                              ctypes.c_void_p(bad.data_ptr())) == 0
    assert bad.item() == 0
    # infinity: 0, as by division
    assert native.compare_f32(ctypes.c_uint(0x7F800000), ctypes.c_uint(1),
                              ctypes.c_void_p(bad.data_ptr())) == 0
    assert bad.item() == 0


@pytest.mark.parametrize("any_value", [0, 1])
def test_fp64_reciprocal_is_the_quotient_or_its_neighbour(native, any_value):
    """Random significands over all exponents whose reciprocals are normal, near
    powers of two, and the values that have none."""
    g = torch.Generator().manual_seed(4)
    n = 1 << 22
    m = 1 + torch.rand(n, generator=g, dtype=torch.float64)
    m[: n // 8] = 1 + torch.randint(0, 4096, (n // 8,), generator=g) * 2.0 ** -52
    m[n // 8: n // 4] = 2 - torch.randint(1, 4096, (n // 8,), generator=g) * 2.0 ** -52
    e = torch.randint(-1021, 1021, (n,), generator=g)
    sign = torch.randint(0, 2, (n,), generator=g) * 2.0 - 1
    x = (sign * torch.ldexp(m, e)).cuda()
    x[:6] = torch.tensor([float("inf"), -float("inf"), 0.0, -0.0, float("nan"), 1.0],
                         dtype=torch.float64)
    y = torch.empty_like(x)
    assert native.recip_f64(ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(y.data_ptr()), n,
                            any_value) == 0
    ref = 1.0 / x
    if any_value:
        assert torch.equal(y[:4], ref[:4])
    assert torch.isnan(y[4]) and y[5] == 1.0
    off = (y[6:].view(torch.int64) - ref[6:].view(torch.int64)).abs()
    assert off.max().item() <= 1
    # the error before the last rounding is 2^-80: next to no quotient is missed
    assert (off > 0).sum().item() <= 8
