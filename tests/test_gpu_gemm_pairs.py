"""The GEMM on CTA pairs (whole 256 x 256 tiles, at least one per pair of
SMs) against FP64, at fewer K blocks than its six stages, exactly as many,
one more, and tile counts that leave pairs unevenly loaded; the 1-CTA kernel
on both sides of the rule; an output that is not 32-byte aligned."""
import pytest
import torch

from paper_1904_06680_gb300 import npp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K,shift", [(2304, 2304, 64, 0), (2304, 2304, 384, 0), (2560, 2048, 448, 0),
                                         (4864, 1024, 320, 4), (2304, 2432, 128, 0), (2432, 2304, 128, 0),
                                         (256, 256, 1024, 0), (20480, 256, 192, 0), (1024, 19456, 64, 0)])
def test_gemm_against_fp64(M, N, K, shift):
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn(M, K, generator=g, device="cuda").to(torch.bfloat16)
    B = torch.randn(N, K, generator=g, device="cuda").to(torch.bfloat16)
    buf = torch.full((M * N + 8,), float("nan"), device="cuda")
    C = buf[shift:shift + M * N].view(M, N)
    npp.npp_gemm_bf16(A, B, C, M, N, K)
    torch.cuda.synchronize()
    npp.npp_gemm_status()
    want = A.double() @ B.double().T
    bound = K * 2.0 ** -22 * (A.double().abs() @ B.double().abs().T)
    assert bool(((C.double() - want).abs() <= bound).all())
    rest = torch.cat([buf[:shift], buf[shift + M * N:]])
    assert bool(torch.isnan(rest).all())
