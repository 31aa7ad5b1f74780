"""FP32 builds at low temperature, where the weights exp(2 beta) come near the end of the format's range, on
lattices without frustration (J_ij = t_i t_j with random signs t), whose answer is known: two ground states,
every other configuration suppressed by exp(-4 beta) at least.  A realization is right or flagged."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


# up to beta = 22 the squares exp(4 beta) of the weights are within the format
@pytest.mark.parametrize("beta", [10.0, 16.0, 18.0, 20.0, 20.5, 21.0, 21.5, 21.8, 22.0, 22.5, 23.0, 26.0, 30.0, 44.0, 60.0])
@pytest.mark.parametrize("precision,chi", [("fp32", 8), ("tf32", 16), ("tf32", 32)])
@pytest.mark.parametrize("compression", ["canonical", "zipup"])
def test_unfrustrated(beta, precision, chi, compression):
    import paper_2409_06538_gb300 as tn
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    tn.build()
    L, R, n = 10, 6, 20
    t = np.random.default_rng(7).choice(np.array([-1, 1], np.int8), (R, L, L))
    J = np.concatenate([(t[:, :, 1:] * t[:, :, :-1]).reshape(R, -1), (t[:, 1:] * t[:, :-1]).reshape(R, -1)], axis=1)
    ctx = tn.TNMC(L, torch.from_numpy(np.ascontiguousarray(J)).cuda(), beta, list(range(R)), chi, precision=precision,
                  compression=compression)
    lz = ctx.build_env()
    out = ctx.propose(n, 0)
    ok = ctx.realization_status() == 0
    energy, logq = out["energy"].cpu().numpy().reshape(R, -1), out["logq"].cpu().numpy().reshape(R, -1)
    ctx.close()
    if beta <= 22:
        assert ok.all()
    bonds = 2 * L * (L - 1)
    # log Z = beta bonds + log 2 from L^2 scales, each right to 2 chi eps at most, and weights exp(+-beta) right to
    # half an eps each, one a bond
    tol = (L * L * 2 * chi + bonds) * 2.0 ** -23
    assert np.abs(lz - (beta * bonds + math.log(2.0)))[ok].max(initial=0.0) <= tol
    assert (energy[ok] == -bonds).all()
    # the two ground states have a half each: one draw that is free, every other conditional within 1e-3 of 1
    assert np.abs(logq[ok] + math.log(2.0)).max(initial=0.0) <= L * L * 1e-3
