"""The surrogate network's chained kernels at the edges of their 128-row tiles: queries of ragged
counts against the network in float64 (BF16 operands as the library rounds them) and against each
other, with and without an error network, and gradients of the smallest batch and of several tiles.

Tolerances: gradients as in test_gpu_surrogate (1e-2 of a layer's largest for operands that round
to the other side of a BF16 tie, 1e-3 in the median).  Query outputs pass five layers of BF16
operands (2^-8 per rounding): 3e-2 of the largest output, 3e-3 in the median."""
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


def _forward(flat, x):
    a = 2.0 * (x.astype(np.float64) - LO) / (HI - LO) - 1.0
    layers = SO.unflatten(flat.astype(np.float64), SO.layer_shapes())
    for l, (w, b) in enumerate(layers):
        z = SO.bf16(a) @ SO.bf16(w).T + b
        a = SO.gelu(z) if l + 1 < len(layers) else z
    return a


def _predict(S, s, x):
    n = len(x)
    coef = torch.full((n + 1, 128), -7.0, device=DEV)           # a canary row past the end
    err = torch.full((n + 1,), -7.0, device=DEV)
    acc = torch.full((n + 1,), 77, dtype=torch.uint8, device=DEV)
    S.soap_surrogate_predict(s, _t(x), 10.0, coef=coef[:n], pred_err=err[:n], accepted=acc[:n])
    torch.cuda.synchronize()
    assert bool((coef[n] == -7.0).all()) and float(err[n]) == -7.0 and int(acc[n]) == 77
    return coef[:n].cpu().numpy(), err[:n].cpu().numpy(), acc[:n].cpu().numpy()


@pytest.mark.parametrize("with_error_net", [False, True])
def test_ragged_queries(S, with_error_net):
    flat, flat_e = synth.surrogate_init(3), synth.surrogate_init(4)
    x = synth.surrogate_params(5, 4500)
    x[131, 2] = 0.5                                             # out of range
    s, e = S.soap_surrogate_create(LO, HI, 128), S.soap_surrogate_create(LO, HI, 256)
    try:
        S.soap_surrogate_set_params(s, flat)
        S.soap_surrogate_set_params(e, flat_e)
        if with_error_net:
            S.soap_surrogate_set_error_net(s, e)
        full = _predict(S, s, x)
        y = _forward(flat, x)
        ye = _forward(flat_e, x)[:, 128] if with_error_net else y[:, 128]
        for got, ref in ((full[0], y[:, :128]), (np.log10(full[1]), ye)):
            d = np.abs(got - ref)
            assert d.max() <= 3e-2 * np.abs(ref).max() and np.median(d) <= 3e-3 * np.abs(ref).max()
        ok = np.all((x >= LO.astype(np.float32)) & (x <= HI.astype(np.float32)), axis=1)
        np.testing.assert_array_equal(full[2], (ok & (full[1] <= 10.0)).astype(np.uint8))
        for n in (1, 31, 127, 128, 129, 257):
            for got, ref in zip(_predict(S, s, x[:n]), full):
                np.testing.assert_array_equal(got, ref[:n])
    finally:
        S.soap_surrogate_free(s)
        S.soap_surrogate_free(e)


@pytest.mark.parametrize("B", [128, 1152])
def test_gradients(S, B):
    rng = np.random.default_rng(B)
    x = synth.surrogate_params(B, B)
    t = rng.normal(0, 1, (B, 129)).astype(np.float32)
    w = np.full(129, 1.0 / 128, np.float32)
    flat = synth.surrogate_init(1)
    s = S.soap_surrogate_create(LO, HI, B)
    try:
        S.soap_surrogate_set_params(s, flat)
        loss, got = S.soap_surrogate_gradients(s, _t(x), _t(t), w)
    finally:
        S.soap_surrogate_free(s)
    layers = SO.unflatten(flat.astype(np.float64), SO.layer_shapes())
    scaled = 2.0 * (x.astype(np.float64) - LO) / (HI - LO) - 1.0
    loss_o, grads = SO.loss_and_grad(layers, scaled, t.astype(np.float64), w.astype(np.float64))
    assert abs(loss - loss_o) <= 1e-4 * abs(loss_o)
    off = 0
    for gW, gb in grads:
        for ref in (gW.ravel(), gb):
            d = np.abs(got[off:off + ref.size] - ref)
            off += ref.size
            assert d.max() <= 1e-2 * np.abs(ref).max() + 1e-7
            assert np.median(d) <= 1e-3 * np.abs(ref).max() + 1e-8
    assert off == got.size
