"""FP32 builds whose weights come near the end of the format's range: a uniform field of k (in units of
beta = 1) makes entries of exp(k) and coefficients of the reflectors of exp(2k), subnormal reciprocals of
which are the first thing to be lost.  The FP64 build of the same realizations is the reference."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


# Up to k = 42 the squares of the entries are within the format; beyond, a build is right or flagged.
@pytest.mark.parametrize("k", [20, 40, 41, 42, 43, 45, 60, 88])
@pytest.mark.parametrize("precision,chi", [("fp32", 4), ("fp32", 8), ("bf16", 8), ("tf32", 16), ("fp32", 32), ("tf32", 32),
                                           ("fp32", 64)])
def test_strong_fields(k, precision, chi):
    import paper_2409_06538_gb300 as tn
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    tn.build()
    L, seeds = 8, list(range(60, 68))
    J = tn.couplings_pmj(L, seeds, 0.109)
    spins = torch.from_numpy(np.where(np.random.default_rng(k).random((len(seeds), 5, L, L)) < 0.3, -1, 1)
                             .astype(np.int8)).cuda()
    res = []
    for prec, c in (("fp64", min(chi, 32)), (precision, chi)):
        ctx = tn.TNMC(L, J, 1.0, seeds, c, precision=prec)
        ctx.set_fields(np.full((len(seeds), L, L), k, np.int8))
        lz = ctx.build_env()
        ctx.propose(20, 0)
        ctx.accept()
        ctx.observables(allow_numeric=True)
        st = ctx.realization_status()
        qp = ctx.eval_conditionals(spins)[1].cpu().numpy()
        res.append((lz, qp, st == 0))
        ctx.close()
    (lz64, qp64, ok64), (lz, qp, ok) = res
    assert ok64.all()
    if k <= 42:
        assert ok.all()
    # log Z: L^2 scales, each from sums of at most 2 chi terms, 2 chi eps <= 1.6e-5 in all of FP32; conditionals:
    # the project's tolerance on FP32 ones
    assert np.abs(lz - lz64)[ok].max(initial=0.0) <= 64 * 128 * 1.2e-7
    assert np.abs(qp - qp64)[ok].max(initial=0.0) <= 1e-3
