"""Pixels that a CCF value does not weigh leave it alone, in FP64 with boxes no wider than a pixel: not a
number, infinite or huge ones under lines of weight zero, outside the lines' boxes at the spectrum's ends,
and between the boxes of neighbouring velocities.  (Lines enough for the kernel of running sums, whose
sums hold such pixels; the windowed kernel, which takes few lines, spreads a bad pixel to boxes that end at
its edge, but not to lines of weight zero.)

Tolerance 1e-12 of the largest CCF value that weighs no such pixel, as everywhere in FP64.  Values that
do weigh a huge one carry its overlap, whose edges are known to 1e-11 pixels: 1e-10 of the largest."""
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
MUS = np.array([0.5, 1.0])
STAR = synth.Star(grid_n=8, vsini_kms=2.0, incl_deg=90.0, u1=0.3, u2=0.3, lambda_start_A=LAM0, lambda_end_A=LAM1,
                  n_px=N_PX, mu_values=MUS)
BAD = [np.nan, np.inf, -np.inf, 1e30]


@pytest.fixture(scope="module")
def ccf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2301_04259_gb300 import soap as S

    def run(F, ml, mw, width, grid):
        out = torch.empty((len(F), grid[2]), dtype=torch.float64, device=DEV)
        rv = torch.empty(len(F), dtype=torch.float64, device=DEV)
        with S.Disk(STAR, torch.ones((2, N_PX), dtype=torch.float64, device=DEV)) as d:
            S.soap_rv_ccf(d.ctx, torch.from_numpy(F).to(DEV), ml, mw, width, *grid, rv, None, out)
            torch.cuda.synchronize()
        return out.cpu().numpy()
    return run


def _case(n_lines, n_spec):
    rng = np.random.default_rng(n_lines)
    u = np.sort(rng.uniform(60, N_PX - 60, n_lines))
    return rng, u, rng.uniform(0.1, 0.9, n_lines), rng.uniform(0.2, 1.0, (n_spec, N_PX))


def _lam(u):
    return LAM0 * np.exp(np.asarray(u) * PX_KMS / synth.C_KMS)


@pytest.mark.parametrize("bad", BAD)
@pytest.mark.parametrize("n_lines", [40, 1500])
def test_lines_of_weight_zero(ccf, n_lines, bad):
    grid = (-22.0, 0.25, 177)
    rng, u, mw, F = _case(n_lines, 9)
    # lines of weight zero, each over a bad pixel that no other line reaches
    ends = np.abs(grid[0]) / PX_KMS + 4
    gaps = [k for k in range(n_lines - 1) if u[k + 1] - u[k] > 2 * ends + 2][:5] if n_lines == 40 else []
    if gaps:
        at = [round(0.5 * (u[k] + u[k + 1])) for k in gaps]
        keep = np.ones(n_lines, bool)
    else:                                                      # dense: the lines around the bad pixels go
        at = [1000, 2345, 7000]
        keep = np.all(np.abs(u[:, None] - np.array(at)) > ends, axis=1)
    u2 = np.concatenate([u[keep], at])
    w2 = np.concatenate([mw[keep], np.zeros(len(at))])
    order = np.argsort(u2)
    F[:, at] = bad
    got = ccf(F, _lam(u2[order]), w2[order], 0.82, grid)
    ref = O.ccf(F, STAR, _lam(u[keep]), mw[keep], 0.82, *grid)
    assert np.isfinite(ref).all() and np.abs(ref).max() < 1e6
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("bad", BAD)
def test_ends_of_the_spectrum(ccf, bad):
    grid = (-22.0, 0.25, 177)
    rng, u, mw, F = _case(2500, 3)
    F[:, [0, N_PX - 1]] = bad
    # boxes that just leave the grid at one end of the velocities, and one that stays
    s = np.arctanh(22.0 / synth.C_KMS) / (PX_KMS / synth.C_KMS)
    u2 = np.sort(np.concatenate([u, [s - 1.2, s - 0.4, N_PX - 1 - s + 0.4, N_PX - 1 - s + 1.2]]))
    w2 = rng.uniform(0.1, 0.9, u2.size)
    got = ccf(F, _lam(u2), w2, 0.82, grid)
    ref = O.ccf(F, STAR, _lam(u2), w2, 0.82, *grid)
    assert np.isfinite(ref).all() and np.abs(ref).max() < 1e6
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("bad", BAD)
@pytest.mark.parametrize("width", [0.3, 0.82])
def test_between_the_boxes(ccf, width, bad):
    # steps of 2.3 pixels: many pixels lie in no velocity's box
    grid = (-20.0, 2.0, 21)
    rng, u, mw, F = _case(2500, 9)
    F[2, [1000, 6001]] = bad
    F[5, 4000] = bad
    got = ccf(F, _lam(u), mw, width, grid)
    ref = O.ccf(F, STAR, _lam(u), mw, width, *grid)
    clean = np.isfinite(ref) & (np.abs(ref) < 1e6)
    assert clean[[2, 5]].any() and not clean[2].all()
    assert np.abs(got - ref)[clean].max() <= 1e-12 * np.abs(ref[clean]).max()
    if np.isfinite(bad):
        hit = ~clean
        assert np.abs(got - ref)[hit].max() <= 1e-10 * np.abs(ref[hit]).max()
    else:
        assert not np.isfinite(got[~clean]).any()
