"""The capacity estimate covers every call of at most the given number of realizations and proposals: what a
smaller call takes is counted although a larger one goes without (its proposals need several passes over the
sampler's slots, and the other kernel serves it)."""
import ctypes

import pytest

pytest.importorskip("torch")


def _held(precision, L, R, chi, n):
    """What the estimate for n proposals adds beside their own buffers."""
    from paper_2409_06538_gb300 import _capi, build
    build()
    opts = _capi.Opts(_capi.PRECISIONS[precision], 2, 0, None)
    est = lambda n: _capi.load().tnmc_estimate_device_bytes(L, R, chi, ctypes.byref(opts), n)  # noqa: E731
    return est(n) - est(0) - 2 * n * R * (4 * ((L * L + 31) // 32) + 8 + 4 + 4 + 4)


# FP64, chi = 16: 32768 / L slots of 32 proposals, 152 of them in every context (152 SMs)
@pytest.mark.parametrize("L,few,many", [
    (163, (1, 3200), (1, 3300)),       # 200 and 207 tiles for 201 slots
    (100, (300, 8), (340, 8)),         # fewer realizations of a context that holds more
    (100, (320, 5), (330, 5))])
def test_never_below_a_smaller_call(L, few, many):
    a, b = _held("fp64", L, few[0], 16, few[1]), _held("fp64", L, many[0], 16, many[1])
    assert a > 0
    assert b >= a
