"""The FP64 bisector kernel of small shifts at the edges it can go wrong at: pixel counts around a
block's 256, several rows a block, table sizes from two depths up, depths exactly on the table's
nodes, fluxes above one, below zero and not finite, and shifts at the edge of the kernel's range,
where the general kernel takes over.

The tolerance, 1e-12 of the largest flux: positions are rounded to 2^-53 of the pixel index in the
kernel and in the oracle, which the steepest flux (below one a pixel) turns into less than
2 x 2^-53 x 4,096 = 9e-13."""
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


def _star(n_px, delta):
    st = synth.config1(0).star
    st.n_px = n_px
    st.lambda_start_A, st.lambda_end_A = 5000.0, 5000.0 * np.exp(delta * (n_px - 1))
    return st


def _inject(S, st, F, bis, orig):
    quiet = torch.ones((len(st.mu_values), st.n_px), dtype=torch.float64, device=DEV)
    with S.Disk(st, quiet) as d:
        out = torch.empty(F.shape, dtype=torch.float64, device=DEV)
        S.soap_inject_bisectors(d.ctx, torch.from_numpy(F).to(DEV), out, bis, orig)
        torch.cuda.synchronize()
        return out.cpu().numpy()


# the last one's velocities are above the small form's 1e-5 c
@pytest.mark.parametrize("n_px,rows,n_d,delta,scale", [
    (255, 1, 2, 2e-6, 0.2), (256, 3, 11, 2e-6, 0.2), (257, 2, 3, 4e-6, 0.3), (769, 5, 101, 3e-7, 0.4),
    (4096, 2411, 11, 2e-6, 0.2), (3000, 20, 20001, 2e-6, 0.2), (2049, 4, 21, 9e-8, 0.9), (1000, 4, 21, 9e-8, 1.2)])
def test_small_shifts_match_the_oracle(S, n_px, rows, n_d, delta, scale):
    rng = np.random.default_rng(n_px)
    st = _star(n_px, delta)
    dl = O.delta(st.lambda_start_A, st.lambda_end_A, n_px)
    x = np.arange(n_px)
    # smooth fluxes from -0.1 to 1.1: a shift's gradient stays far below one pixel a pixel
    F = 0.5 + 0.6 * np.sin(2 * np.pi * x / 400.0 + rng.uniform(0, 6, (rows, 1)))
    on = np.round(F * (n_d - 1)) / (n_d - 1)                # stretches exactly on the table's nodes
    if n_d > 1000:
        F = np.where((x // 50) % 2 == 0, on, F)
    d = np.linspace(0, 1, n_d)
    a, b = rng.uniform(-1, 1, (2, rows, 1))
    s = min(scale, 20.0 * dl * 2.99792458e5)                # the gradient of the shift below 0.6 pixel a pixel
    bis = s * (0.5 * a + 0.5 * b * d * (1 - d) * 4)
    ref = O.inject_bisectors(F, bis, np.zeros(n_d), dl)
    got = _inject(S, st, F, bis, np.zeros(n_d))
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()


def test_fluxes_that_are_not_finite_stay_where_they_are(S):
    """A NaN or an infinity has depth zero (or one) and spoils the two output pixels it brackets;
    every other pixel is as without it."""
    n_px, st = 1024, _star(1024, 2e-6)
    F = np.full((2, n_px), 0.8)
    bad = {100: np.nan, 255: np.inf, 256: 0.8, 600: -np.inf}
    for k, v in bad.items():
        F[:, k] = v
    bis = np.zeros((2, 11))
    bis[1] = 0.2
    got = _inject(S, st, F, bis, np.zeros(11))
    k0 = 0.2 / 2.99792458e5 / 2e-6
    assert 0.2 < k0 < 0.5
    spoiled = np.zeros(n_px, bool)
    for k in (100, 255, 600):
        spoiled[k - 1: k + 2] = True
    assert np.all(np.abs(got[:, ~spoiled] - 0.8) <= 1e-15)
    assert not np.isfinite(got[:, [101, 256, 601]][1]).any()  # row 1: moved by k0 pixels to the right
    assert not np.isfinite(got[0, [100, 255, 600]]).any()


def test_neighbours_moved_onto_each_other_are_refused(S):
    n_px, st = 512, _star(512, 2e-6)
    dl = O.delta(st.lambda_start_A, st.lambda_end_A, n_px)
    for at in (255, 256, 510):                              # across a block's edge, and the last pair
        F = np.ones((1, n_px))
        F[0, at + 1:] = 0.0
        bis = np.zeros((1, 2))
        bis[0, 0] = 1.5 * dl * 2.99792458e5                 # depth zero moves past its right neighbour
        with pytest.raises(S.SoapError):
            _inject(S, st, F, bis, np.zeros(2))
