"""The persistent tensor-core GEMM with more output tiles than SMs: ragged rows and columns, even
and odd output strides (two ways of storing), with and without bias, columns past N left alone.

Tolerance: BF16 products are exact in FP32; K additions each round by at most 2^-23 of the largest
partial sum, which sum |a b| + |bias| bounds."""
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


@pytest.mark.parametrize("bias", [False, True])
@pytest.mark.parametrize("M,N,K,ldc", [(2600, 5003, 136, 5004), (2600, 5003, 72, 5003), (20011, 128, 64, 131),
                                       (20011, 60, 200, 60), (1, 40000, 384, 40002)])
def test_many_tiles(S, M, N, K, ldc, bias):
    g = torch.Generator(device=DEV).manual_seed(M + N + K)
    A = torch.randn((M, K), generator=g, device=DEV).bfloat16()
    B = torch.randn((N, K), generator=g, device=DEV).bfloat16()
    b = torch.randn(N, generator=g, device=DEV) if bias else None
    C = torch.full((M, ldc), -3.0, device=DEV)
    S.soap_gemm_bf16_tn(A, B, C, bias=b)
    ref, mag = A.double() @ B.double().T, A.double().abs() @ B.double().abs().T
    if bias:
        ref, mag = ref + b.double(), mag + b.double().abs()
    assert bool(((C[:, :N].double() - ref).abs() <= K * 2.0 ** -23 * mag).all())
    assert bool((C[:, N:] == -3.0).all()) if ldc > N else True
