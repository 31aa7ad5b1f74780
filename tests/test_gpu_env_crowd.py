"""The second build of chi = 16 in FP32, for calls whose realizations fill the GPU (seven per SM; the first
one holds five): what the occupancy query reports, and equal bits at a full wave of the second build."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_full_wave_of_the_second_build():
    import paper_2409_06538_gb300 as tn
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    tn.build()
    L, chi = 9, 16
    # the query is about the first build; from its number the dispatch sends 6 per SM (two of its waves, one of
    # the second's) and 7 per SM to the second one
    per_sm, sms = tn.env_build_occupancy(L, chi, "fp32")
    assert per_sm == 5
    many, out = list(range(100, 100 + 7 * sms)), []
    some = [0, 5 * sms, 7 * sms - 1]
    for seeds, at in ((many, some), ([many[k] for k in some], [0, 1, 2])):
        ctx = tn.TNMC(L, tn.couplings_pmj(L, seeds, 0.109), tn.nishimori_beta(0.109), seeds, chi, precision="fp32")
        lz = ctx.build_env()
        out.append(([lz[k] for k in at], [ctx.copy_env(k, r)[0] for k in at for r in (0, L // 2)]))
        ctx.close()
    assert out[0][0] == out[1][0]
    for a, b in zip(out[0][1], out[1][1]):
        assert np.array_equal(a, b)
