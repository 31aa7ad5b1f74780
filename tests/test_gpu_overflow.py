"""Weights that overflow the build's number format: the environments hold infinities and NaN, the
build ends, the realizations are flagged when they are sampled, and the context stays usable."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision,chi,compression", [("fp32", 8, "canonical"), ("tf32", 16, "canonical"),
                                                       ("tf32", 32, "zipup"), ("fp32", 64, "canonical")])
def test_overflowing_weights_are_flagged(precision, chi, compression):
    import paper_2409_06538_gb300 as tn
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    tn.build()
    L, seeds = 10, [50, 51, 52]
    J = tn.couplings_pmj(L, seeds, 0.3)
    ctx = tn.TNMC(L, J, 100.0, seeds, chi, precision=precision, compression=compression)   # exp(100) > FLT_MAX
    ctx.build_env(return_logz=False)
    ctx.propose(20, 0)
    ctx.accept()
    ctx.observables(allow_numeric=True)
    assert np.all(ctx.realization_status() == 4)
    ctx.set_couplings(J, tn.nishimori_beta(0.109), seeds)
    assert np.all(np.isfinite(ctx.build_env()))
    ctx.propose(20, 0)
    ctx.accept()
    ctx.observables()
    assert np.all(ctx.realization_status() == 0)
    ctx.close()
