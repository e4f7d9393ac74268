"""GPU: the branch-free inner minimisation against relu_argmin, bit for bit.

Duals, slopes and bounds are multiples of 1/64 up to 4, so that every product
of the two forms is exact however it is fused; exact ties, zeros of both signs,
empty intervals, infinite bounds and NaN included.
"""
import ctypes
import os
import subprocess

import pytest
import torch

pytestmark = pytest.mark.gpu

SRC = r"""
#include "ld_common.cuh"
using namespace ld;
__device__ float pick(uint32_t h, int wild) {
  if (wild && h % 13 == 0) {
    const float s[6] = {INFINITY, -INFINITY, NAN, -0.f, 0.f, 1e-45f};
    return s[h / 13 % 6];
  }
  return (float)((int)(h % 513) - 256) / 64.f;
}
__global__ void compare(unsigned long long* bad, int total, int wild) {
  unsigned long long n = 0;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
    uint32_t h = t * 2654435761u + 77u;
    float a[4];
    for (int i = 0; i < 4; ++i) {
      h = h * 1664525u + 1013904223u;
      a[i] = pick((h ^ h >> 13) >> 3, wild);
    }
    if (t % 4 == 0) a[1] = a[0];                 // r = c: the ties of a passing ReLU
    if (t % 4 == 1 && a[2] > a[3]) { const float x = a[2]; a[2] = a[3]; a[3] = x; }
    if (t % 8 == 2) { a[2] = -fabsf(a[2]); a[3] = fabsf(a[3]); a[1] = a[3] != 0.f && a[3] == 1.f ? a[0] - a[0] * a[2] : a[1]; }
    float xb, x, yb, y;
    int code;
    relu_argmin<float>(a[0], a[1], a[2], a[3], xb, x, code);
    relu_argmin_flat(a[0], a[1], a[2], a[3], yb, y);
    n += __float_as_uint(xb) != __float_as_uint(yb) && !(xb != xb && yb != yb);
    n += __float_as_uint(x) != __float_as_uint(y) && !(x != x && y != y);
  }
  if (n) atomicAdd(bad, n);
}
extern "C" int run(int wild, unsigned long long* bad) {
  compare<<<1024, 256>>>(bad, 1 << 24, wild);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2104_06718_gb300 import build
    d = tmp_path_factory.mktemp("argmin")
    src, out = d / "argmin.cu", d / "argmin.so"
    src.write_text(SRC)
    csrc = os.path.join(os.path.dirname(build.__file__), "csrc")
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-I", csrc, str(src), "-o", str(out)], check=True)
    lib = ctypes.CDLL(str(out))
    lib.run.argtypes = [ctypes.c_int, ctypes.c_void_p]
    return lib


@pytest.mark.parametrize("wild", [0, 1])
def test_same_vertex(lib, wild):
    bad = torch.zeros(1, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    assert lib.run(wild, bad.data_ptr()) == 0
    assert bad.item() == 0
