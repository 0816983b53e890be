"""The training loss where its squares leave FP32's range: residuals of 1e20, a residual of 1e30 under a
weight of zero, and weights of 2^-118 (batches trained in pairs of thread blocks and without).

A residual y - t is rounded once to FP32 and the loss is summed to 48 bits or more: with |t| = 1e20 and y of
order one every residual is -t exactly, so the loss is known to 1e-13; scaling all weights by 2^-118 scales
it exactly, each loss within 2^-45 of its sum."""
import numpy as np
import pytest

from paper_2301_04259_gb300 import synth

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
LO, HI = synth.SURROGATE_LO, synth.SURROGATE_HI


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2301_04259_gb300 import soap
    return soap


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


@pytest.mark.parametrize("B", [128, 10240])
def test_loss_outside_the_range_of_fp32_squares(S, B):
    rng = np.random.default_rng(B)
    x = _t(synth.surrogate_params(B, B))
    t = rng.normal(0, 1, (B, 129)).astype(np.float32)
    w = rng.uniform(0.5, 1.5, 129).astype(np.float32)
    s = S.soap_surrogate_create(LO, HI, B)
    try:
        S.soap_surrogate_set_params(s, synth.surrogate_init(1))
        plain, _ = S.soap_surrogate_gradients(s, x, _t(t), w)
        tiny, _ = S.soap_surrogate_gradients(s, x, _t(t), w * np.float32(2.0 ** -118))
        big = np.where(rng.random((B, 129)) < 0.5, 1e20, -1e20).astype(np.float32)
        huge, _ = S.soap_surrogate_gradients(s, x, _t(big), w)
        w0 = w.copy()
        w0[5] = 0
        masked = t.copy()
        masked[:, 5] = 1e30
        without, _ = S.soap_surrogate_gradients(s, x, _t(t), w0)
        over, _ = S.soap_surrogate_gradients(s, x, _t(masked), w0)
    finally:
        S.soap_surrogate_free(s)
    assert abs(tiny * 2.0 ** 118 / plain - 1) <= 1e-13
    exact = w.astype(np.float64).sum() * float(np.float32(1e20)) ** 2
    assert abs(huge / exact - 1) <= 1e-13
    assert abs(over / without - 1) <= 1e-13
