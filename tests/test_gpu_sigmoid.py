"""The encoder's sigmoid and Swish (csrc/tc_common.cuh), compiled by
themselves: the bits of 1.f / (1.f + expf(-x)) and x / (1.f + expf(-x)) for every
fp32 x, alone in its block and beside a value that takes the block out of the
range of the reciprocal."""
import ctypes
import subprocess

import pytest

from paper_2609_14991_gb300 import _build

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SOURCE = r"""
#include "tc_common.cuh"
using namespace tsd::tc;
__device__ bool same(float a, float b) { return (isnan(a) && isnan(b)) || __float_as_uint(a) == __float_as_uint(b); }
__global__ void k_compare(float beside, unsigned long long* bad) {
  const unsigned long long step = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < 1ull << 32; i += step) {
    const float x = __uint_as_float((unsigned)i);
    const uint64_t v[2] = {pair_of(x, beside), pair_of(beside, x)};
    const float d = 1.f + expf(-x), db = 1.f + expf(-beside);
    uint64_t y[2];
    float p, q, r, s;
    sigmoid2(v, y);
    unpair(y[0], p, q);
    unpair(y[1], r, s);
    if (!same(p, 1.f / d) || !same(s, 1.f / d) || !same(q, 1.f / db) || !same(r, 1.f / db)) atomicAdd(bad, 1ull);
    swish2(v, y);
    unpair(y[0], p, q);
    unpair(y[1], r, s);
    if (!same(p, x / d) || !same(s, x / d) || !same(q, beside / db) || !same(r, beside / db)) atomicAdd(bad + 1, 1ull);
  }
}
extern "C" __attribute__((visibility("default"))) int compare(float beside, unsigned long long* bad) {
  k_compare<<<1216, 256>>>(beside, bad);
  const cudaError_t e = cudaGetLastError();
  return (int)(e == cudaSuccess ? cudaDeviceSynchronize() : e);
}
"""


def test_every_value(tmp_path):
    src, lib = tmp_path / "sigmoid.cu", tmp_path / "sigmoid.so"
    src.write_text(SOURCE)
    subprocess.run([_build.nvcc()] + _build._flags() + ["-shared", "-cudart", "static", "-o", str(lib), str(src)], check=True)
    fn = ctypes.CDLL(str(lib)).compare
    fn.argtypes = [ctypes.c_float, ctypes.c_void_p]
    for beside in (0.0, 1.5, 88.0, -87.0, -200.0):
        bad = torch.zeros(2, dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        assert fn(beside, bad.data_ptr()) == 0
        assert bad.tolist() == [0, 0], (beside, bad.tolist())
