"""The two FMA samplers (one thread and one warp per proposal) give the same bits on environments that
no neighbouring test takes through both: zip-up ones (rows swept from either side), those of periodic
chains (one proposal per region, the chain given per region) and those of overflowed builds."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def tn():
    import paper_2409_06538_gb300 as pkg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.build()
    return pkg


def _run(tn, L, chi, seeds, n, precision, beta, p, compression):
    ctx = tn.TNMC(L, tn.couplings_pmj(L, seeds, p), beta, seeds, chi, precision=precision, compression=compression)
    ctx.build_env(return_logz=False)
    out = ctx.propose(n, 3)
    spins = ctx.spins()
    lq, qp = ctx.eval_conditionals(spins.reshape(len(seeds), 2 * n, L, L)[:, :3].contiguous())
    res = out["logq"].cpu(), out["energy"].cpu(), spins.cpu(), lq.cpu(), qp.cpu(), torch.from_numpy(ctx.realization_status())
    ctx.close()
    return res


# 700 realizations of five proposals in two chains are two CTAs of eight each: 1400 and more than four on
# every SM, the thread's side of the line for all types and bond dimensions; two realizations are on the other.
@pytest.mark.parametrize("L,chi,precision", [(9, 7, "fp32"), (10, 8, "fp64"), (11, 13, "bf16"), (12, 16, "fp32")])
def test_zipup_environments(tn, L, chi, precision):
    seeds = list(range(40, 740))
    args = (5, precision, tn.nishimori_beta(0.109), 0.109, "zipup")
    for a, b in zip(_run(tn, L, chi, seeds, *args), _run(tn, L, chi, seeds[:2], *args)):
        assert torch.equal(a[:2], b)


@pytest.mark.parametrize("compression", ["canonical", "zipup"])
@pytest.mark.parametrize("beta", [24.0, 44.0, 100.0])          # exp(2 beta): squares overflow, a weight overflows
def test_overflowed_environments(tn, beta, compression):
    seeds = list(range(40, 740))
    args = (10, 8, seeds, 5, "fp32", beta, 0.3, compression)
    many = _run(tn, *args)
    few = _run(tn, *args[:2], seeds[:4], *args[3:])
    for a, b in zip(many, few):
        assert torch.equal(a[:4], b)
    assert np.isfinite(many[0].numpy()).all()


@pytest.mark.parametrize("L,chi,precision", [(7, 5, "fp64"), (9, 16, "fp32")])
def test_periodic_chains(tn, L, chi, precision):
    beta, seeds = tn.nishimori_beta(0.109), list(range(70, 420))
    out = []
    for s in (seeds, seeds[:3]):
        ctx = tn.TNMCPeriodic(L, tn.torus_couplings_pmj(L, s, 0.109), beta, s, chi, precision=precision, n_chains=2)
        ctx.step(4, 0)
        out.append((ctx.spins().cpu(), [o["n_acc"] for o in ctx.observables()][:3]))
        ctx.close()
    assert torch.equal(out[0][0][:3], out[1][0]) and out[0][1] == out[1][1]
