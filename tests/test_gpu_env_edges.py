"""Environment build on the GPU at the edges of its tiles: bond dimensions around every padded size,
the smallest lattices, rows whose bond dimensions are cut on one side only, both compressions."""
import numpy as np
import pytest

from oracle import boundary_mps as bm
from oracle import lattice

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def tn():
    import paper_2409_06538_gb300 as pkg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.build()
    return pkg


# log Z is the sum of the logarithms of L^2 removed scales, each from sums of at most 2 chi <= 128 terms
# of one sign pattern: a relative error of a few 128 eps per scale, against log Z >= log(2) L^2.  That is
# 128 eps * few / log 2 < 1e3 eps in all: 1e-4 in FP32 and 1e-12 in FP64 leave another factor of ten for
# what the truncated weights amplify.
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-11), ("fp32", 1e-4)])
@pytest.mark.parametrize("compression", ["canonical", "zipup"])
@pytest.mark.parametrize("L,chi", [(2, 1), (2, 4), (3, 2), (5, 1), (7, 3), (9, 4), (9, 5), (12, 8), (13, 9), (14, 15),
                                   (14, 16), (15, 17), (15, 31), (14, 32), (16, 33), (14, 64)])
def test_log_z_at_tile_edges(tn, precision, tol, compression, L, chi):
    if precision == "fp64" and chi > 32:
        pytest.skip("FP64 is built up to chi = 32")
    p, seeds = 0.2, [3, 4, 5]
    beta = lattice.nishimori_beta(p)
    ctx = tn.TNMC(L, tn.couplings_pmj(L, seeds, p), beta, seeds, chi, precision=precision, compression=compression)
    lz = ctx.build_env()
    for k, s in enumerate(seeds):
        Jh, Jv = lattice.split_couplings(lattice.couplings_pmj(s, L, p), L)
        env = bm.build_envs(Jh, Jv, beta, chi, method=compression)
        assert abs(lz[k] - env.log_z) <= tol * abs(env.log_z), (k, lz[k], env.log_z)
        dims = ctx.copy_env(k, 0)[1]
        assert list(dims) == env.bond_dims(0)
    ctx.close()


@pytest.mark.parametrize("chi,compression", [(13, "canonical"), (16, "canonical"), (16, "zipup")])
def test_same_bits_alone_and_in_a_crowd(tn, chi, compression):
    """chi = 16 has a second build for calls whose realizations fill the GPU; a realization's
    environments do not depend on which one it went through."""
    L, p = 9, 0.109
    per_sm, sms = tn.env_build_occupancy(L, chi, "fp32")
    many = list(range(100, 100 + (per_sm + 1) * sms))       # one wave more than the other build holds
    out = []
    for seeds in (many, many[:3]):
        ctx = tn.TNMC(L, tn.couplings_pmj(L, seeds, p), lattice.nishimori_beta(p), seeds, chi, precision="fp32",
                      compression=compression)
        lz = ctx.build_env()
        out.append((lz[:3], [ctx.copy_env(k, r)[0] for k in range(3) for r in (0, L // 2)]))
        ctx.close()
    assert np.array_equal(out[0][0], out[1][0])
    for a, b in zip(out[0][1], out[1][1]):
        assert np.array_equal(a, b)
