"""The windowed CCF (wide boxes, FP64 spectra) where its lines per chunk and its pixels per box
change: few and many lines, dense and sparse, boxes of 0.8 to 13 pixels, one and several blocks of
spectra, against the FP64 oracle's CCF of the same spectra.

Tolerances, of the largest CCF value.  FP64: 1e-12 as everywhere.  FP32: every product is positive
(flux times weight times overlap), a chunk adds at most 32 lines x 16 pixels one after another,
each addition rounding by 2^-24 (3.1e-5), and a box edge at a coordinate below 16 pixels is off by
at most 2 x 16 x 2^-24 = 1.9e-6 pixels of a box of at least 0.8 pixels (2.4e-6): 3.4e-5 in all."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2301_04259_gb300 import synth

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2301_04259_gb300 import soap
    return soap


@pytest.mark.parametrize("n_spec", [1, 17])
@pytest.mark.parametrize("width", [0.1, 0.82, 1.6])
@pytest.mark.parametrize("n_lines", [1, 30, 700])
def test_windowed_ccf_matches_oracle(S, n_lines, width, n_spec):
    c = synth.config1(0)
    st = c.star
    rng = np.random.default_rng(n_lines)
    ml = np.sort(rng.uniform(6000.5, 6009.5, n_lines))
    mw = rng.uniform(0.1, 0.9, n_lines)
    lo, step, nv = synth.velocity_grid(st.vsini_kms)
    F = c.quiet[rng.integers(0, st.n_mu, n_spec)] * rng.uniform(0.5, 2.0, (n_spec, 1))
    for dtype, tol in ((np.float64, 1e-12), (np.float32, 3.4e-5)):
        X = np.ascontiguousarray(F.astype(dtype))
        ref = O.ccf(X.astype(np.float64), st, ml, mw, width, lo, step, nv)
        rv = torch.empty(n_spec, dtype=torch.float64, device=DEV)
        ccf = torch.empty((n_spec, nv), dtype=torch.float64, device=DEV)
        with S.Disk(st, torch.from_numpy(c.quiet).to(DEV)) as d:
            S.soap_rv_ccf(d.ctx, torch.from_numpy(X).to(DEV), ml, mw, width, lo, step, nv, rv, None, ccf)
            torch.cuda.synchronize()
        assert np.abs(ccf.cpu().numpy() - ref).max() <= tol * np.abs(ref).max()
