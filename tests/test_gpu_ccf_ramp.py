"""The FP64 CCF of boxes no wider than a pixel (one multiply-add pair per line and pixel offset)
against the FP64 oracle: box widths from a twentieth of a pixel to all but one, one line to many
(sparse, dense, repeated, beyond the grid), few and many velocities, one and several blocks of
spectra.  Tolerance 1e-12 of the largest CCF value, as everywhere in FP64; where the lines overlap so
little of the grid that the oracle's CCF is zero, so is the library's."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2301_04259_gb300 import synth

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
N_PX = 8191
LAM0 = 5000.0
PX_KMS = 0.8692                                                # a pixel in km/s
LAM1 = LAM0 * np.exp((N_PX - 1) * PX_KMS / synth.C_KMS)


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2301_04259_gb300 import soap
    return soap


def _lines(kind, rng):
    if kind == "one":
        return np.array([0.5 * (LAM0 + LAM1)])
    if kind == "sparse":
        return np.sort(rng.uniform(LAM0, LAM1, 40))
    if kind == "dense":
        return np.sort(rng.uniform(LAM0, LAM1, 3000))
    # repeated lines, lines on pixel centres and edges, lines whose boxes leave the grid, lines far off it
    u = np.concatenate([np.full(9, 1234.3), np.arange(300, 340), np.arange(500, 540) + 0.5, [3.0, N_PX - 2.5]])
    lam = LAM0 * np.exp(u * PX_KMS / synth.C_KMS)
    return np.sort(np.concatenate([lam, [0.1 * LAM0, 10 * LAM0]]))


@pytest.mark.parametrize("grid", [(-22.0, 0.25, 177), (-3.0, 1.5, 5), (-30.0, 0.2, 300), (5.0, 0.01, 64)])
@pytest.mark.parametrize("width", [0.05, 0.5, 0.82, 0.869])
@pytest.mark.parametrize("kind", ["one", "sparse", "dense", "odd"])
def test_narrow_box_ccf(S, kind, width, grid):
    rng = np.random.default_rng(len(kind))
    ml = _lines(kind, rng)
    mw = rng.uniform(0.1, 0.9, ml.size)
    mus = np.array([0.5, 1.0])
    star = synth.Star(grid_n=8, vsini_kms=2.0, incl_deg=90.0, u1=0.3, u2=0.3, lambda_start_A=LAM0,
                      lambda_end_A=LAM1, n_px=N_PX, mu_values=mus)
    lam = synth.wavelength_grid(LAM0, LAM1, N_PX)
    base = synth.local_spectra(lam, rng.uniform(LAM0, LAM1, 700), rng.uniform(0.1, 0.8, 700),
                               rng.uniform(0.03, 0.08, 700), mus)
    with S.Disk(star, torch.from_numpy(base).to(DEV)) as d:
        for n_spec in (1, 9):
            F = base[rng.integers(0, 2, n_spec)] * rng.uniform(0.5, 2.0, (n_spec, 1)) + rng.normal(0, 1e-3, (n_spec, N_PX))
            ref = O.ccf(F, star, ml, mw, width, *grid)
            rv = torch.empty(n_spec, dtype=torch.float64, device=DEV)
            ccf = torch.empty((n_spec, grid[2]), dtype=torch.float64, device=DEV)
            S.soap_rv_ccf(d.ctx, torch.from_numpy(F).to(DEV), ml, mw, width, *grid, rv, None, ccf)
            torch.cuda.synchronize()
            assert np.abs(ccf.cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()
