"""The projection's error as a norm, where the elementwise bound of test_gpu_pca_project is loose: odd row
lengths (loads of single pixels), tiles cut between thread blocks, several tiles of components.  Three BF16
parts and six products keep it below that of one FP32 rounding per value and per running sum: 2e-6, as over
16,834 pixels."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("n,p,k", [(129, 1000, 128), (300, 4097, 128), (1000, 777, 200), (128, 16834, 3),
                                   (9800, 641, 128), (20011, 131, 128), (9729, 65, 257)])
def test_error(n, p, k):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2301_04259_gb300 import soap as S
    g = torch.Generator(device=DEV).manual_seed(n + p + k)
    mean = torch.randn(p, generator=g, device=DEV)
    X, basis = torch.randn((n, p), generator=g, device=DEV) + mean, torch.randn((k, p), generator=g, device=DEV)
    out = torch.empty((n, k), device=DEV)
    S.soap_pca_project(X, mean, basis, out)
    ref = (X.double() - mean.double()) @ basis.double().T
    assert float((out.double() - ref).norm() / ref.norm()) < 2.0e-6
