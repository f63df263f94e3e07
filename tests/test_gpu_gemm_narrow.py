"""Narrow GEMMs (N <= 32) on both sides of the ring's dispatch: up to 152 tiles
of 128 rows, one CTA an SM, and more, two CTAs an SM; K shorter and longer than
the rings.  Products of BF16 values are exact in FP32; K additions of FP32 values
of up to about 4 K^(1/2) err by at most K 2^-24 of that, within 1e-4 K^(1/2) for
K <= 512 (an output of FP32 rounds by 6e-8 of itself)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gm():
    if not torch.cuda.is_available():
        pytest.fail("CUDA GPU required for -m gpu tests")
    from paper_2007_12273_gb300 import build, gm as gm_
    build.build()
    gm_.load()
    return gm_


@pytest.mark.parametrize("M", [128, 152 * 128, 152 * 128 + 1, 40001])
@pytest.mark.parametrize("N", [1, 16, 31, 32])
@pytest.mark.parametrize("K", [8, 64, 200, 512])
def test_narrow_gemm(gm, M, N, K):
    g = torch.Generator(device="cuda").manual_seed(M + 7 * N + K)
    A = torch.randn(M, K, generator=g, device="cuda").to(torch.bfloat16)
    B = torch.randn(N, K, generator=g, device="cuda").to(torch.bfloat16)
    bias = torch.randn(N, generator=g, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    C = gm.gm_gemm_bf16(A, B, bias=bias, relu=True, err=err)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    ref = torch.relu(A.double() @ B.double().T + bias.double())
    assert C.shape == (M, N)
    assert float((C.double() - ref).abs().max()) <= 1e-4 * K ** 0.5
