"""The tensor-core CCF of spectra whose rows are not 16-byte aligned (loaded through registers, pixel
pairs or single pixels) and the reduction of few chunks of many outputs: odd and even pixel counts,
offset pointers, few spectra and several tiles, against the FP64 oracle.  Tolerance as in
test_gpu_ccf_tc: 1.7e-4 of the largest CCF value."""
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


@pytest.mark.parametrize("n_px,offset", [(2049, 0), (4102, 0), (4102, 1), (4096, 1), (2115, 0)])
@pytest.mark.parametrize("n_spec", [1, 9, 130, 2000])
def test_unaligned_rows(S, n_px, offset, n_spec):
    c = synth.config2(0, grid_n=8, n_px=n_px, lambda_start=5000.0,
                      lambda_end=5000.0 * np.exp((n_px - 1) / 345000.0))
    rng = np.random.default_rng(n_px)
    F = (c.quiet[rng.integers(0, 20, n_spec)] * rng.uniform(0.5, 2.0, (n_spec, 1))).astype(np.float32)
    flat = torch.full((n_spec * n_px + 8,), float("nan"), device=DEV)      # neighbours must not be read into sums
    spectra = flat[offset:offset + n_spec * n_px].view(n_spec, n_px)
    spectra.copy_(torch.from_numpy(F))
    lo, step, nv = synth.velocity_grid(2.0)
    rv = torch.empty(n_spec, dtype=torch.float64, device=DEV)
    ccf = torch.empty((n_spec, nv), dtype=torch.float64, device=DEV)
    with S.Disk(c.star, torch.from_numpy(c.quiet).to(DEV)) as d:
        S.soap_rv_ccf(d.ctx, spectra, c.mask_lambda, c.mask_weight, 0.82, lo, step, nv, rv, None, ccf,
                      tensor_cores=True)
        torch.cuda.synchronize()
    rows = np.unique(np.concatenate([[0, n_spec - 1], rng.integers(0, n_spec, 20)]))
    ref = O.ccf(F[rows].astype(np.float64), c.star, c.mask_lambda, c.mask_weight, 0.82, lo, step, nv)
    assert np.abs(ccf.cpu().numpy()[rows] - ref).max() <= 1.7e-4 * np.abs(ref).max()
