"""More phase blocks than a grid holds in y (65,535): FP64 and FP32 spectra of a small star at 131,079 phases
against the FP64 oracle at the first, the last and those around the limit of either block size.  Tolerances
as everywhere: 1e-12 of the largest flux in FP64, 1e-5 in FP32."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2301_04259_gb300 import synth

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("limb", [False, True])
@pytest.mark.parametrize("f64", [True, False])
def test_many_phases(f64, limb):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2301_04259_gb300 import soap as S
    n = 2 * 65535 + 9
    case = synth.make_case(5, name="many phases", grid_n=12, lambda_start=6000.0, lambda_end=6000.5, n_px=200,
                           mu_values=(0.3, 0.6, 0.9), n_lines=4, depth_law="uniform", sigma_law="angstrom",
                           vsini_kms=3.0, incl_deg=75.0, n_phases=5,
                           regions=[synth.Region(synth.FACULA, 10.0, -20.0, 0.5, 6100.0),
                                    synth.Region(synth.SPOT, -10.0, 40.0, 0.3, 4800.0)])
    phases = np.linspace(0.0, 1.0, n, endpoint=False)
    checked = np.array([0, 65534, 65535, 131068, 131069, 131070, 131071, n - 1])
    out = torch.empty((1, n, case.star.n_px), dtype=torch.float64 if f64 else torch.float32, device=DEV)
    active = {t: torch.from_numpy(a).to(DEV) for t, a in case.active.items()}
    with S.Disk(case.star, torch.from_numpy(case.quiet).to(DEV), active) as d:
        if limb:
            S.soap_set_facula_limb_brightening(d.ctx, True)
        S.soap_active_phases(d.ctx, case.regions, phases, S.SOAP_EFFECT_TOT, S.SOAP_FP64 if f64 else S.SOAP_FP32, out)
        torch.cuda.synchronize()
        few = torch.empty((1, checked.size, case.star.n_px), dtype=out.dtype, device=DEV)
        S.soap_active_phases(d.ctx, case.regions, phases[checked], S.SOAP_EFFECT_TOT,
                             S.SOAP_FP64 if f64 else S.SOAP_FP32, few)
        torch.cuda.synchronize()
    got = out[0].cpu().numpy()[checked].astype(np.float64)
    tol = 1e-12 if f64 else 1e-5
    assert np.abs(got - few[0].cpu().numpy()).max() <= tol * np.abs(got).max()
    if not limb:
        ref = O.active(case.star, case.quiet, case.active, case.regions, phases[checked])[0]
        assert np.abs(got - ref).max() <= tol * np.abs(ref).max()
