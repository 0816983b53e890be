"""Projection onto the PCA basis on the tensor cores: ragged spectra, pixels and components, one
and several tiles, tiles computed by two CTAs, repeated calls bit for bit, and non-finite inputs.

Tolerance: the split drops products below 3 x 2^-24 of a product, subtracting the mean rounds by
2^-24, and at most 512 pixels x 5 products are added to an accumulator between two FP32 sums; with
FP32 rounding at every addition the plain product's worst case, p x 2^-24 of sum |x - mean| |v|,
bounds all of it for p >= 512 (and 520 x 2^-24 below)."""
import pytest

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


def _inputs(n, p, k):
    g = torch.Generator(device=DEV).manual_seed(n + p + k)
    mean = torch.randn(p, generator=g, device=DEV)
    return torch.randn((n, p), generator=g, device=DEV) + mean, mean, torch.randn((k, p), generator=g, device=DEV)


@pytest.mark.parametrize("n,p,k", [(1, 1, 1), (5, 63, 128), (129, 1000, 128), (300, 4097, 128), (1000, 777, 200),
                                   (128, 16834, 3), (9800, 640, 128), (20011, 130, 128), (9729, 65, 257)])
def test_projection(S, n, p, k):
    X, mean, basis = _inputs(n, p, k)
    out = torch.full((n + 1, k), 5.0, device=DEV)
    S.soap_pca_project(X, mean, basis, out[:n])
    ref = (X.double() - mean.double()) @ basis.double().T
    mag = (X.double() - mean.double()).abs() @ basis.double().abs().T
    assert bool(((out[:n].double() - ref).abs() <= max(p, 520) * 2.0 ** -24 * mag).all())
    assert bool((out[n] == 5.0).all())
    again = torch.empty((n, k), device=DEV)
    S.soap_pca_project(X, mean, basis, again)
    assert torch.equal(out[:n], again)


def test_error_is_not_that_of_a_long_float_sum(S):
    """Over 16,834 pixels the error stays below that of a float32 product summed in order."""
    X, mean, basis = _inputs(512, 16834, 128)
    out = torch.empty((512, 128), device=DEV)
    S.soap_pca_project(X, mean, basis, out)
    ref = (X.double() - mean.double()) @ basis.double().T
    # rounding of the order of 2^-24 sqrt(p) / 2 of the result for a sequential sum: 3.9e-6
    assert float((out.double() - ref).norm() / ref.norm()) < 2.0e-6


def test_non_finite_inputs(S):
    X, mean, basis = _inputs(300, 500, 128)
    X[3, 7] = float("inf")
    X[140, 400] = float("nan")
    X[299, 499] = -3.4e38                                       # rounds to -inf in BF16
    out = torch.empty((300, 128), device=DEV)
    S.soap_pca_project(X, mean, basis, out)
    ref = X.double() @ basis.double().T - mean.double() @ basis.double().T
    ok = [r for r in range(300) if r not in (3, 140, 299)]
    assert bool(torch.isfinite(out[ok]).all()) and bool(torch.isnan(out[140]).all())
    assert torch.equal(out[3], torch.sign(basis[:, 7]) * float("inf"))
    # overflow where the sum exceeds the largest float, and nowhere else
    assert torch.equal(torch.isinf(out[299]), ref[299].abs() > torch.finfo(torch.float32).max)
