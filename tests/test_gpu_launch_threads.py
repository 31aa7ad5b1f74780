"""Contexts of different lattice sizes used from several host threads at once: the same kernels, each
launch with its own amount of shared memory.  No launch fails, and every context gives what it gives alone."""
import threading

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("chi,precision", [(32, "tf32"), (16, "tf32"), (16, "fp32"), (8, "fp64"), (64, "bf16")])
def test_threads_of_different_sizes(chi, precision):
    import paper_2409_06538_gb300 as tn
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    tn.build()

    def work(L, rounds):
        with torch.cuda.stream(torch.cuda.Stream()):
            seeds = [1, 2]
            ctx = tn.TNMC(L, tn.couplings_pmj(L, seeds, 0.109), 1.0, seeds, chi, precision=precision)
            for i in range(rounds):
                if L < 32:
                    ctx.build_env(return_logz=False)
                elif i == 0:
                    ctx.build_env()
                out = ctx.propose(8, 0)
            res = out["logq"].cpu(), out["energy"].cpu()
            ctx.close()
            return res

    sizes = {4: 250, 6: 250, 9: 200, 64: 60}
    got, errors = {}, []

    def thread(L, rounds):
        try:
            got[L] = work(L, rounds)
        except Exception as e:  # reported below, by the main thread
            errors.append((L, str(e)))

    threads = [threading.Thread(target=thread, args=a) for a in sizes.items()]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for L in sizes:
        for a, b in zip(got[L], work(L, 1)):
            assert torch.equal(a, b)
