"""Workspace of the samplers for chi <= 16: contexts hold one sized for few proposals; the first call for many
takes the rest, or does without it (no memory, stream being captured) with the same results."""
import ctypes

import pytest

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def estimate():
    from paper_2409_06538_gb300 import _capi, build
    build()
    lib = _capi.load()

    def est(precision, L, R, chi, n):
        opts = _capi.Opts(_capi.PRECISIONS[precision], 2, 0, None)
        return lib.tnmc_estimate_device_bytes(L, R, chi, ctypes.byref(opts), n)
    return est


def _props(L, R, n):
    return 2 * n * R * (4 * ((L * L + 31) // 32) + 8 + 4 + 4 + 4)


# bytes of the environments, the build's scratch and a workspace of 32 proposals per SM (FMA samplers, 152 SMs) or
# 256 (tensor cores), rounded up
@pytest.mark.parametrize("precision,L,chi,limit,many", [("fp64", 24, 16, 36e6, 1000), ("fp32", 16, 8, 7e6, 1000),
                                                        ("bf16", 24, 4, 5e6, 1000), ("tf32", 64, 16, 330e6, 200)])
def test_estimate(estimate, precision, L, chi, limit, many):
    none = estimate(precision, L, 1, chi, 0)
    assert none <= limit
    assert estimate(precision, L, 1, chi, 10) == none + _props(L, 1, 10)
    R = 304
    more = estimate(precision, L, R, chi, many) - estimate(precision, L, R, chi, 0) - _props(L, R, many)
    assert 0 < more <= 256 << 20


@pytest.mark.gpu
@pytest.mark.parametrize("precision,L,chi,R,few,many", [("fp64", 10, 16, 40, 1, 150), ("fp32", 12, 8, 40, 3, 300),
                                                        ("tf32", 12, 16, 310, 3, 100)])
def test_calls_for_many_proposals(estimate, monkeypatch, precision, L, chi, R, few, many):
    import paper_2409_06538_gb300 as tn
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    seeds, beta = list(range(5, 5 + R)), tn.nishimori_beta(0.109)
    J = tn.couplings_pmj(L, seeds, 0.109)
    make = lambda: tn.TNMC(L, J, beta, seeds, chi, precision=precision)  # noqa: E731
    more = estimate(precision, L, R, chi, many) - estimate(precision, L, R, chi, 0) - _props(L, R, many)
    assert more > 0

    ctx = make()
    ctx.build_env(return_logz=False)
    ctx.propose(few, 0)
    assert ctx.device_bytes() == estimate(precision, L, R, chi, few)
    want = ctx.propose(many, 0)["logq"].cpu()
    assert ctx.device_bytes() == estimate(precision, L, R, chi, many)
    spins = ctx.spins().reshape(R, 2 * many, L, L)
    lq = ctx.eval_conditionals(spins, want_qplus=False)[0].cpu()
    ctx.close()

    # no memory for more
    alloc = torch.cuda.caching_allocator_alloc

    def refuse(nbytes, device=None, stream=None):
        if nbytes == more:
            raise RuntimeError("out of memory")
        return alloc(nbytes, device=device, stream=stream)

    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", refuse)
    ctx = make()
    ctx.build_env(return_logz=False)
    assert torch.equal(ctx.propose(many, 0)["logq"].cpu(), want)
    assert ctx.device_bytes() == estimate(precision, L, R, chi, many) - more
    monkeypatch.undo()
    assert torch.equal(ctx.propose(many, 0)["logq"].cpu(), want)
    assert ctx.device_bytes() == estimate(precision, L, R, chi, many)
    ctx.close()

    # captured before any call for many
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = make()
        ctx.build_env()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            out = ctx.eval_conditionals(spins, want_qplus=False)[0]
        held = ctx.device_bytes()
        graph.replay()
        assert torch.equal(out.cpu(), lq)
        assert torch.equal(ctx.eval_conditionals(spins, want_qplus=False)[0].cpu(), lq)
        assert ctx.device_bytes() == held + more
        out.zero_()
        graph.replay()
        assert torch.equal(out.cpu(), lq)
        ctx.close()
