"""Tensor-core sampler at the edges of its tiles: proposal counts around 128, the smallest and odd
lattices, every width between the padded bond dimensions, and a lattice large enough that fewer
environment tiles are kept in flight.  The FP32 FMA sampler over the same environments (the builds
are the same) is the reference."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# each path's conditionals are within 1e-3 of the FP64 ones, so the two are within twice that
TOL = 2e-3


@pytest.fixture(scope="module")
def tn():
    import paper_2409_06538_gb300 as pkg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.build()
    return pkg


def _pair(tn, L, chi, seeds, fields):
    beta, J = tn.nishimori_beta(0.109), tn.couplings_pmj(L, seeds, 0.109)
    out = []
    for precision in ("tf32", "fp32"):
        c = tn.TNMC(L, J, beta, seeds, chi, precision=precision)
        if fields:
            c.set_fields(np.random.default_rng(L).integers(-1, 2, (len(seeds), L, L)).astype(np.int8))
        c.build_env(return_logz=False)
        out.append(c)
    return out


@pytest.mark.parametrize("L,chi,R,n,fields", [
    (2, 16, 3, 1, False), (3, 9, 2, 63, True), (5, 16, 1, 64, False), (8, 12, 5, 65, False), (31, 16, 2, 129, True),
    (32, 32, 2, 64, False), (33, 17, 3, 40, True), (9, 32, 1, 200, False), (64, 16, 400, 64, False),
    (40, 32, 320, 64, False), (224, 20, 1, 3, False)])
def test_same_conditionals_as_fma_sampler(tn, L, chi, R, n, fields):
    seeds = list(range(7, 7 + R))
    tc, fma = _pair(tn, L, chi, seeds, fields)
    out = tc.propose(n, 11)
    spins = tc.spins().reshape(R, 2 * n, L, L)
    pick = spins[:, :: max(1, (2 * n) // 5)].contiguous()
    lq, qp = tc.eval_conditionals(pick)
    lq_ref, qp_ref = fma.eval_conditionals(pick)
    assert float((qp - qp_ref).abs().max()) <= TOL
    # the proposal carries exactly the q it was drawn with
    drawn = out["logq"].reshape(R, 2 * n)[:, :: max(1, (2 * n) // 5)]
    assert float(((drawn - lq).abs() / lq.abs().clamp(min=1.0)).max()) <= 1e-9
    # energies and magnetisations are those of the returned spins
    s = pick.to(torch.int32)
    J = tn.couplings_pmj(L, seeds, 0.109).to(torch.int32)
    jh = J[:, :L * (L - 1)].reshape(R, 1, L, L - 1)
    jv = J[:, L * (L - 1):].reshape(R, 1, L - 1, L)
    E = -(jh * s[..., :-1] * s[..., 1:]).sum((-2, -1)) - (jv * s[..., :-1, :] * s[..., 1:, :]).sum((-2, -1))
    assert torch.equal(E, out["energy"].reshape(R, 2 * n)[:, :: max(1, (2 * n) // 5)].to(E.dtype))
    assert torch.equal(s.sum((-2, -1)), out["magnet"].reshape(R, 2 * n)[:, :: max(1, (2 * n) // 5)].to(torch.int64))
    tc.close()
    fma.close()
