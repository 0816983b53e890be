"""The FP32 contraction over aligned tap groups against the FP64 one (which reads the same kernels
tap by tap): pixel counts around a block's 512 and a thread's 8 (direct and staged stores), more
groups than a block stages at once, every phase-block size, all effects, a contrast row per class and
per (class, mu bin), and in batches contrasts taken by a line and pixel by pixel.

Tolerance: the mixed path's 2e-6 of the largest quiet flux."""
import dataclasses

import numpy as np
import pytest

from paper_2301_04259_gb300 import synth
from paper_2301_04259_gb300.synth import FACULA, SPOT, Region

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"
TOL32 = 2e-6


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2301_04259_gb300 import soap
    return soap


def _disk(S, n_px, n_mu, vsini, px_kms, grid_n=40):
    """Smooth local spectra on a log grid of px_kms km/s pixels."""
    lam = 5000.0 * np.exp(np.arange(n_px) * px_kms / 299792.458)
    mus = (np.arange(n_mu) + 0.5) / n_mu
    star = dataclasses.replace(synth.config1(0).star, n_px=n_px, lambda_start_A=lam[0], lambda_end_A=lam[-1],
                               mu_values=mus, vsini_kms=vsini, incl_deg=80.0, grid_n=grid_n)
    x = np.arange(n_px)
    q = np.stack([(0.5 + 0.5 * m) * (1 - 0.4 * np.cos(x / 9.0 + m)) for m in mus])
    rows = {SPOT: torch.from_numpy(0.8 * q + 0.1).to(DEV), FACULA: torch.from_numpy(0.9 * q + 0.05).to(DEV)}
    return S.Disk(star, torch.from_numpy(q).to(DEV), rows)


REGIONS = [Region(FACULA, 10.0, 0.0, 0.35, 6100.0), Region(SPOT, 10.0, 5.0, 0.15, 4500.0),
           Region(SPOT, -30.0, 90.0, 0.2, 4900.0), Region(FACULA, 40.0, 180.0, 0.3, 6000.0)]


# n_mu, vsini and pixel size set the groups of a phase block: 3 in the first case, over 100 in the last two
@pytest.mark.parametrize("n_px,n_mu,vsini,px_kms,n_phases", [
    (7, 3, 2.0, 2.0, 1), (512, 5, 3.0, 1.0, 5), (513, 5, 3.0, 1.0, 4), (1016, 8, 4.0, 0.9, 3), (1020, 8, 4.0, 0.9, 7),
    (1537, 20, 30.0, 0.9, 9), (4096, 40, 20.0, 0.5, 6)])
@pytest.mark.parametrize("limb", [False, True])
def test_star(S, n_px, n_mu, vsini, px_kms, n_phases, limb):
    phases = np.arange(n_phases) / n_phases
    got = {}
    with _disk(S, n_px, n_mu, vsini, px_kms) as d:
        S.soap_set_facula_limb_brightening(d.ctx, limb)
        for prec, dt in ((S.SOAP_FP64, torch.float64), (S.SOAP_FP32, torch.float32)):
            out = torch.full((3, n_phases, n_px), float("nan"), dtype=dt, device=DEV)
            S.soap_active_phases(d.ctx, REGIONS, phases, 7, prec, out)
            S.soap_synchronize(d.ctx)
            got[prec] = out.double().cpu().numpy()
    ref = got[S.SOAP_FP64]
    assert np.abs(got[S.SOAP_FP32] - ref).max() <= TOL32 * np.abs(ref).max()


# pixels of 0.9 km/s take the contrast by a line, those of 20 km/s pixel by pixel; the kernels of the last
# case's phase blocks (4 classes, 40 bins, 242 taps) do not fit in shared memory, those of the one before
# with few phases a block only
@pytest.mark.parametrize("n_px,px_kms,vsini,n_mu", [(1025, 0.9, 12.0, 12), (1024, 0.9, 12.0, 12), (515, 20.0, 12.0, 12),
                                                    (600, 0.9, 30.0, 20), (700, 0.5, 60.0, 40)])
@pytest.mark.parametrize("residual", [False, True])
def test_batch(S, n_px, px_kms, vsini, n_mu, residual):
    phases = np.concatenate([np.arange(9) / 9.0, [0.1, 0.3], [0.7]])
    items = [(vsini, 80.0, 0, 4, 0, 9), (0.5 * vsini, 60.0, 1, 2, 9, 2), (-vsini, 30.0, 0, 0, 11, 1)]
    with _disk(S, n_px, n_mu, vsini, px_kms) as d:
        outs = []
        for v in range(S.soap_batch_num_variants()):
            S.soap_batch_set_variant(d.ctx, v)
            out = torch.full((12, n_px), float("nan"), dtype=torch.float32, device=DEV)
            S.soap_active_batch(d.ctx, items, REGIONS, phases, out,
                                output=S.SOAP_BATCH_RESIDUAL if residual else S.SOAP_BATCH_SPECTRUM)
            S.soap_synchronize(d.ctx)
            outs.append(out.cpu())
    for o in outs[1:]:
        assert torch.equal(o, outs[0])
    # the first item alone as a star in FP64
    with _disk(S, n_px, n_mu, vsini, px_kms) as d:
        ref = torch.empty((1, 9, n_px), dtype=torch.float64, device=DEV)
        quiet = torch.empty(n_px, dtype=torch.float64, device=DEV)
        S.soap_active_phases(d.ctx, REGIONS, phases[:9], S.SOAP_EFFECT_TOT, S.SOAP_FP64, ref)
        S.soap_quiet_spectrum(d.ctx, S.SOAP_FORM_TOEPLITZ, S.SOAP_FP64, quiet)
        S.soap_synchronize(d.ctx)
    ref, quiet = ref[0].cpu().numpy(), quiet.cpu().numpy()
    want = ref - quiet if residual else ref
    assert np.abs(outs[0][:9].double().numpy() - want).max() <= TOL32 * quiet.max()
    assert not outs[0][11].any() if residual else np.isfinite(outs[0][11].numpy()).all()
