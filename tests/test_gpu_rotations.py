"""The environment build's norms and Jacobi rotations (csrc/rounding.cuh) against their definitions, and its
log Z to the digits that it has."""
import ctypes
import subprocess

import pytest

from oracle import boundary_mps as bm
from oracle import lattice

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SRC = r"""
#include "rounding.cuh"
using namespace tnmc;
template <typename T> __global__ void rotations(const T* a, const T* b, const T* g, double* unit, double* off, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  T c, s;
  rotation_from_gram(a[i], b[i], g[i], c, s);
  const double C = c, S = s, G = g[i], d = (double)(T)(b[i] - a[i]);
  unit[i] = fabs(fma(C, C, -1.0) + S * S);
  // y_p' . y_q' over the scale of the 2 x 2 Gram matrix's differences
  off[i] = fabs(fma(C * C - S * S, G, -(C * S) * d)) / hypot(d, 2.0 * G);
}
__global__ void norms(const double* x, double* y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = norm_of(x[i]);
}
extern "C" int run(int what, const void* a, const void* b, const void* g, double* p, double* q, int n) {
  const int k = (n + 255) / 256;
  if (what == 0) rotations<<<k, 256>>>((const double*)a, (const double*)b, (const double*)g, p, q, n);
  if (what == 1) rotations<<<k, 256>>>((const float*)a, (const float*)b, (const float*)g, p, q, n);
  if (what == 2) norms<<<k, 256>>>((const double*)a, p, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2409_06538_gb300 import buildlib
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("rotations")
    (d / "t.cu").write_text(SRC)
    so = str(d / "t.so")
    subprocess.run([buildlib.nvcc()] + buildlib.ARCH + buildlib.NVCC_FLAGS + ["-shared", "-o", so, str(d / "t.cu")],
                   check=True, capture_output=True)
    lib = ctypes.CDLL(so)
    lib.run.argtypes = [ctypes.c_int] + [ctypes.c_void_p] * 5 + [ctypes.c_int]
    return lib


# The two roots carry two units in the last place each, the sums and products around them half of one: below
# ten of 2^-53 (2^-24) in c and s, twice that in their squares; 24 with the check's own roundings.
@pytest.mark.parametrize("dtype,what,unit", [(torch.float64, 0, 2.0 ** -53), (torch.float32, 1, 2.0 ** -24)])
def test_rotations(lib, dtype, what, unit):
    n = 1 << 20
    gen = torch.Generator(device="cuda").manual_seed(1)
    rnd = lambda: torch.rand(n, generator=gen, device="cuda", dtype=torch.float64)  # noqa: E731
    a, b = 10.0 ** (8 * rnd() - 4), 10.0 ** (8 * rnd() - 4)
    b[: n // 4] = a[: n // 4] * (1 + 1e-3 * rnd()[: n // 4])              # norms close to one another
    b[:64] = a[:64]
    g = torch.sqrt(a * b) * 10.0 ** (-8 * rnd()) * torch.sign(rnd() - 0.5)   # |cosine| from 1e-8 to 1
    a, b, g = (t.to(dtype).contiguous() for t in (a, b, g))
    p, q = (torch.empty(n, device="cuda", dtype=torch.float64) for _ in range(2))
    assert lib.run(what, a.data_ptr(), b.data_ptr(), g.data_ptr(), p.data_ptr(), q.data_ptr(), n) == 0
    assert float(p.max()) <= 24 * unit
    assert float(q.max()) <= 24 * unit


def test_fp64_norms(lib):
    """Newton's step on a root of a few units leaves one unit in the last place at most."""
    n = 1 << 20
    gen = torch.Generator(device="cuda").manual_seed(2)
    x = 10.0 ** (600 * torch.rand(n, generator=gen, device="cuda", dtype=torch.float64) - 299)
    y = torch.empty_like(x)
    assert lib.run(2, x.data_ptr(), None, None, y.data_ptr(), None, n) == 0
    r = torch.sqrt(x)
    assert float(((y - r).abs() / r).max()) <= 2.0 ** -52
    for v in (0.0, float("inf")):
        x[:1] = v
        assert lib.run(2, x.data_ptr(), None, None, y.data_ptr(), None, 1) == 0
        assert float(y[0]) == v


# log Z is the sum of the logarithms of N = L^2 removed scales, each from sums of 2 chi <= 128 terms, whose
# roundings add up as sqrt(128) eps; over the sites these average out, so that log Z >= log(2) N is right to
# 11 / (log 2 sqrt(N)) <= 4 eps from L = 4 on.  32 times that for truncated bonds and the sweeps between.
@pytest.mark.parametrize("precision,eps", [("fp64", 2.0 ** -52), ("fp32", 2.0 ** -23)])
@pytest.mark.parametrize("compression", ["canonical", "zipup"])
@pytest.mark.parametrize("L,chi", [(5, 2), (9, 4), (12, 8), (13, 9), (14, 16), (15, 31), (14, 32), (14, 64)])
def test_log_z_digits(precision, eps, compression, L, chi):
    import paper_2409_06538_gb300 as tn
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if precision == "fp64" and chi > 32:
        pytest.skip("FP64 is built up to chi = 32")
    tn.build()
    p, seeds = 0.2, [3, 4, 5]
    beta = lattice.nishimori_beta(p)
    ctx = tn.TNMC(L, tn.couplings_pmj(L, seeds, p), beta, seeds, chi, precision=precision, compression=compression)
    lz = ctx.build_env()
    ctx.close()
    for k, s in enumerate(seeds):
        Jh, Jv = lattice.split_couplings(lattice.couplings_pmj(s, L, p), L)
        ref = bm.build_envs(Jh, Jv, beta, chi, method=compression).log_z
        assert abs(lz[k] - ref) <= 128 * eps * abs(ref), (k, lz[k], ref)
