"""An RV call that fails for want of memory leaves the next one, with the mask of the one before it, as it
was: the failed call's tables are not taken for that mask's."""
import numpy as np
import pytest

from paper_2301_04259_gb300 import synth

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
N_PX = 8191
LAM0 = 5000.0
PX_KMS = 0.8692
LAM1 = LAM0 * np.exp((N_PX - 1) * PX_KMS / synth.C_KMS)
GRID = (-22.0, 0.25, 177)


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2301_04259_gb300 import soap
    return soap


def test_failed_call_leaves_no_tables(S):
    rng = np.random.default_rng(0)

    def lam(u):
        return LAM0 * np.exp(np.sort(u) * PX_KMS / synth.C_KMS)
    mask = lam(rng.uniform(60, N_PX - 60, 2500))
    # 1,300 lines on the grid with a gap that no unit of 16 lines bridges, and so many beyond it that
    # the partial sums of 100,000 spectra take more memory than there is (443 GB)
    other = np.concatenate([lam(rng.uniform(60, 2000, 1289)), lam(rng.uniform(7500, N_PX - 60, 11)),
                            LAM1 * np.linspace(2, 3, 98700)])
    star = synth.Star(grid_n=8, vsini_kms=2.0, incl_deg=90.0, u1=0.3, u2=0.3, lambda_start_A=LAM0,
                      lambda_end_A=LAM1, n_px=N_PX, mu_values=np.array([0.5, 1.0]))
    F = torch.from_numpy(rng.uniform(0.2, 1.0, (9, N_PX))).to(DEV)
    many = torch.empty((100000, N_PX), dtype=torch.float64, device=DEV)
    rv = torch.empty(100000, dtype=torch.float64, device=DEV)
    with S.Disk(star, torch.ones((2, N_PX), dtype=torch.float64, device=DEV)) as d:
        def ccf():
            out = torch.empty((9, GRID[2]), dtype=torch.float64, device=DEV)
            S.soap_rv_ccf(d.ctx, F, mask, np.ones(mask.size), 0.82, *GRID, rv[:9], None, out)
            torch.cuda.synchronize()
            return out
        before = ccf()
        with pytest.raises(S.SoapError):
            S.soap_rv_ccf(d.ctx, many, other, np.ones(other.size), 0.82, *GRID, rv)
        assert torch.equal(ccf(), before)
