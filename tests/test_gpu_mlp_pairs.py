"""A training step's chained network in pairs of CTAs (few rows) and in single CTAs (rows for every
SM): the gradients of the smallest batch and of batches on each side of the switch agree with the FP64
oracle (tolerances as in test_gpu_mlp) and repeat to the bit."""
import numpy as np
import pytest

from oracle import surrogate as SO
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


@pytest.mark.parametrize("B", [128, 9216, 9344])               # 72 tiles in pairs, 73 without
def test_gradients(S, B):
    flat = synth.surrogate_init(1)
    rng = np.random.default_rng(B)
    x = synth.surrogate_params(2, B)
    t = rng.normal(0, 1, (B, 129)).astype(np.float32)
    w = np.full(129, 1.0 / 128, np.float32)
    s = S.soap_surrogate_create(LO, HI, B)
    try:
        S.soap_surrogate_set_params(s, flat)
        loss, g = S.soap_surrogate_gradients(s, _t(x), _t(t), w)
        again, h = S.soap_surrogate_gradients(s, _t(x), _t(t), w)
    finally:
        S.soap_surrogate_free(s)
    assert np.array_equal(g, h)
    layers = SO.unflatten(flat.astype(np.float64), SO.layer_shapes())
    scaled = 2.0 * (x.astype(np.float64) - LO) / (HI - LO) - 1.0
    ref_loss, ref = SO.loss_and_grad(layers, scaled, t.astype(np.float64), w.astype(np.float64))
    assert abs(loss - ref_loss) <= 1e-4 * abs(ref_loss)
    off = 0
    for gw, gb in ref:
        for r in (gw.ravel(), gb):
            got = g[off:off + r.size]
            off += r.size
            assert np.abs(got - r).max() <= 1e-2 * np.abs(r).max() + 1e-7
            assert np.median(np.abs(got - r)) <= 1e-3 * np.abs(r).max() + 1e-8
