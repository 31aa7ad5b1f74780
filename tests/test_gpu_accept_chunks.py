"""Metropolis decisions at the edges of the accept kernel's chunks of steps, over several calls and
one to eight chains, against the oracle's chain on the GPU's own energies and log q."""
import numpy as np
import pytest

from oracle import metropolis

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,chains", [(1, 1), (2, 8), (127, 2), (128, 3), (129, 2), (300, 1)])
def test_decisions_across_chunks(n, chains):
    import paper_2409_06538_gb300 as tn
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    tn.build()
    L, chi, seeds = 6, 1, [2, 3]                 # chi = 1: about a fifth of the proposals is rejected
    beta = tn.nishimori_beta(0.109)
    ctx = tn.TNMC(L, tn.couplings_pmj(L, seeds, 0.109), beta, seeds, chi, precision="fp64", n_chains=chains)
    ctx.build_env(return_logz=False)
    E, lq, fl = [], [], []
    for call in range(2):
        out = ctx.propose(n, call * n)
        fl.append(ctx.accept(flags=True)["flags"].cpu().numpy())
        E.append(out["energy"].cpu().numpy())
        lq.append(out["logq"].cpu().numpy())
    E, lq, fl = (np.concatenate(x, axis=2) for x in (E, lq, fl))
    obs = ctx.observables()
    for k, s in enumerate(seeds):
        for ch in range(chains):
            acc, cur, _ = metropolis.metropolis_chain(E[k, ch], lq[k, ch], beta, s, ch, np.arange(2 * n))
            assert np.array_equal(acc, fl[k, ch].astype(bool))
        assert obs[k]["n_acc"] == int(fl[k].sum()) - chains and obs[k]["n_prop"] == 2 * n * chains
    ctx.close()
