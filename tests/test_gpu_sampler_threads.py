"""One-thread-per-proposal sampler against the warp-per-proposal one: the dispatch chooses by the number
of proposals in FP64, so the two have to give the same bits; FP32 against the oracle at the edges of
its tiles (a warp's 32 proposals, odd lattices, bond dimensions between the padded sizes, fields)."""
import numpy as np
import pytest

from oracle import boundary_mps as bm
from oracle import lattice, sampler

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def tn():
    import paper_2409_06538_gb300 as pkg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.build()
    return pkg


def _run(tn, L, chi, seeds, n, precision, fields=None):
    ctx = tn.TNMC(L, tn.couplings_pmj(L, seeds, 0.109), tn.nishimori_beta(0.109), seeds, chi, precision=precision)
    if fields is not None:
        ctx.set_fields(fields)
    ctx.build_env(return_logz=False)
    out = ctx.propose(n, 3)
    spins = ctx.spins()
    lq, qp = ctx.eval_conditionals(spins.reshape(len(seeds), 2 * n, L, L)[:, :3].contiguous())
    res = out["logq"].cpu(), out["energy"].cpu(), spins.cpu(), lq.cpu(), qp.cpu()
    ctx.close()
    return res


@pytest.mark.parametrize("L,chi", [(3, 2), (8, 4), (9, 7), (12, 8), (11, 13), (16, 16)])
@pytest.mark.parametrize("with_fields", [False, True])
def test_fp64_same_bits_alone_and_in_a_crowd(tn, L, chi, with_fields):
    crowd = list(range(40, 40 + 160))
    f = np.random.default_rng(L).integers(-1, 2, (len(crowd), L, L)).astype(np.int8) if with_fields else None
    many = _run(tn, L, chi, crowd, 33, "fp64", f)        # 10560 proposals
    few = _run(tn, L, chi, crowd[:2], 33, "fp64", None if f is None else f[:2])
    for a, b in zip(many, few):
        assert torch.equal(a[:2], b)


@pytest.mark.parametrize("L,chi,n", [(2, 1, 1), (5, 4, 15), (7, 3, 16), (8, 8, 17), (13, 5, 33), (17, 16, 40), (33, 8, 5)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_conditionals_against_oracle(tn, L, chi, n, precision):
    seeds = [11, 12] if precision == "fp32" else list(range(11, 11 + max(2, 5200 // (2 * n) + 1)))
    logq, energy, spins, lq, qp = _run(tn, L, chi, seeds, n, precision)
    for k in (0, 1):
        Jh, Jv = lattice.split_couplings(lattice.couplings_pmj(seeds[k], L, 0.109), L)
        env = bm.build_envs(Jh, Jv, lattice.nishimori_beta(0.109), chi)
        s = spins[k].reshape(2 * n, L, L)[:3].numpy()
        ev = sampler.evaluate(env, s)
        # the project's tolerances on conditionals: 1e-9 relative in FP64, 1e-3 absolute in FP32
        d = np.abs(qp[k].numpy() - ev["qplus"])
        if precision == "fp64":
            assert np.all(d <= 1e-9 * np.minimum(ev["qplus"], 1 - ev["qplus"]) + 4e-16)
        else:
            assert d.max() <= 1e-3
        assert np.array_equal(energy[k].reshape(2 * n)[:3].numpy(), lattice.energy(s, Jh, Jv))
        m = min(3, n)                                    # the first chain's proposals among them
        assert torch.equal(lq[k][:m], logq[k].reshape(2 * n)[:m])


# The same in FP32 and BF16: more than four CTAs of eight proposals per SM take the thread's path, in
# whole tiles of 32 and in tiles that a realization's proposals do not fill.
@pytest.mark.parametrize("L,chi,crowd,n", [(3, 2, 700, 5), (8, 4, 160, 33), (9, 7, 700, 5), (12, 8, 160, 33),
                                           (11, 13, 160, 33), (16, 16, 1300, 1)])
@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_fp32_same_bits_alone_and_in_a_crowd(tn, L, chi, crowd, n, precision):
    seeds = list(range(40, 40 + crowd))
    many = _run(tn, L, chi, seeds, n, precision)
    few = _run(tn, L, chi, seeds[:2], n, precision)
    for a, b in zip(many, few):
        assert torch.equal(a[:2], b)
