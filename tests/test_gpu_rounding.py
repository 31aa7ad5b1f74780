"""The short forms of csrc/rounding.cuh against the operations they stand for, over every float of the
range that each is used in: the same bits."""
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SRC = r"""
#include "rounding.cuh"
using namespace tnmc;
__device__ bool same(float a, float b) { return __float_as_uint(a) == __float_as_uint(b); }
__device__ bool ok(int op, float x) {
  if (op == 0) return same(inverse(x), 1.0f / x);
  return same(tf32_rna_finite(x), tf32_rna(x)) && same(tf32_rna_finite(-x), tf32_rna(-x));
}
__global__ void count(int op, unsigned lo, unsigned hi, unsigned long long* bad) {
  unsigned long long n = 0;
  for (unsigned long long b = lo + blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; b <= hi;
       b += (unsigned long long)gridDim.x * blockDim.x)
    n += !ok(op, __uint_as_float((unsigned)b));
  if (n) atomicAdd(bad, n);
}
extern "C" int run(int op, unsigned lo, unsigned hi, void* bad) {
  count<<<1024, 256>>>(op, lo, hi, (unsigned long long*)bad);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2409_06538_gb300 import buildlib
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("rounding")
    (d / "t.cu").write_text(SRC)
    so = str(d / "t.so")
    subprocess.run([buildlib.nvcc()] + buildlib.ARCH + buildlib.NVCC_FLAGS + ["-shared", "-o", so, str(d / "t.cu")],
                   check=True, capture_output=True)
    lib = ctypes.CDLL(so)
    lib.run.argtypes = [ctypes.c_int, ctypes.c_uint, ctypes.c_uint, ctypes.c_void_p]
    return lib


def _bits(x):
    return int(torch.tensor(x, dtype=torch.float32).view(torch.int32).item())


@pytest.mark.parametrize("op,lo,hi", [
    (0, _bits(1e-37), _bits(8e37)),
    # below the largest binade, zero and subnormal numbers among them
    (1, 0, _bits(2.0 ** 127) - 1)], ids=["inverse", "tf32"])
def test_same_bits_over_the_range(lib, op, lo, hi):
    bad = torch.zeros(1, dtype=torch.int64, device="cuda")
    assert lib.run(op, lo, hi, bad.data_ptr()) == 0
    assert int(bad.item()) == 0
