"""The windowed CCF where its windows hold few lines or none: velocity sweeps near and above the pixels a
block stages, many spectra.  The partial sums stay at one per 32 lines (or what fills the GPU), and the CCF
agrees with the FP64 oracle within the tolerances of the windowed kernel (1e-12 of the largest value in
FP64; in FP32 a chunk adds at most 32 lines x 16 pixels, 3.4e-5)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2301_04259_gb300 import synth

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
PX_KMS, LAM0 = 0.122, 5000.0


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2301_04259_gb300 import soap
    return soap


@pytest.mark.parametrize("dtype,tol", [(np.float64, 1e-12), (np.float32, 3.4e-5)])
@pytest.mark.parametrize("n_lines,n_px,grid", [
    (2000, 20000, (-50.0, 0.5, 201)),            # a sweep of 820 pixels: no window holds a line
    (350, 40000, (-30.0, 0.25, 241)),            # 492 pixels, lines 110 apart: two lines a window
])
def test_wide_sweeps(S, n_lines, n_px, grid, dtype, tol):
    lam1 = LAM0 * np.exp((n_px - 1) * PX_KMS / synth.C_KMS)
    star = synth.Star(grid_n=8, vsini_kms=2.0, incl_deg=90.0, u1=0.3, u2=0.3, lambda_start_A=LAM0,
                      lambda_end_A=lam1, n_px=n_px, mu_values=np.array([0.5, 1.0]))
    rng = np.random.default_rng(n_lines)
    ml = LAM0 * np.exp(np.sort(rng.uniform(500, n_px - 500, n_lines)) * PX_KMS / synth.C_KMS)
    mw = rng.uniform(0.1, 0.9, n_lines)
    n_spec, checked = 300, [0, 7, 299]
    lam = synth.wavelength_grid(LAM0, lam1, n_px)
    base = synth.local_spectra(lam, rng.uniform(LAM0, lam1, 200), rng.uniform(0.1, 0.8, 200),
                               rng.uniform(0.03, 0.08, 200), np.array([0.5, 1.0]))
    X = np.ascontiguousarray((base[rng.integers(0, 2, n_spec)] * rng.uniform(0.5, 2.0, (n_spec, 1))).astype(dtype))
    ref = O.ccf(X[checked].astype(np.float64), star, ml, mw, 0.82, *grid)
    F = torch.from_numpy(X).to(DEV)
    rv = torch.empty(n_spec, dtype=torch.float64, device=DEV)
    ccf = torch.empty((n_spec, grid[2]), dtype=torch.float64, device=DEV)
    with S.Disk(star, torch.from_numpy(base).to(DEV)) as d:
        S.soap_rv_ccf(d.ctx, F[:1], ml[:1], mw[:1], 0.82, *grid, rv[:1])
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        S.soap_rv_ccf(d.ctx, F, ml, mw, 0.82, *grid, rv, None, ccf)
        torch.cuda.synchronize()
        used = before - torch.cuda.mem_get_info()[0]
    assert np.abs(ccf.cpu().numpy()[checked] - ref).max() <= tol * np.abs(ref).max()
    # partial sums, CCF and its scaled copy; four blocks of at most 16 spectra on each SM write partial sums
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rows = (n_lines / 32 + 1 + 2) * n_spec + 4 * sms * 16
    assert used <= rows * grid[2] * 8 + (16 << 20), used
