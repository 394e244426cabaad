"""The tensor-core GEMM on TF32 halves (operands whose columns of A and rows of B are scaled
inversely over 12 decades) at the edges of its split's tiles of 32 x 32: rows and inner lengths
around multiples of 32, odd row strides (no vector loads), both layouts of both operands, more
tiles than the launch takes at once.

Tolerance 1e-6 relative Frobenius as for the library's other FP32 products: 22-bit operands leave
~2e-7 and FP32 accumulation ~3e-7, while a lost half leaves ~5e-4.
"""
import pytest
import torch

from paper_1403_6968_gb300 import gemm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ta,tb", [(False, False), (True, True), (True, False), (False, True)])
@pytest.mark.parametrize("M,N,K", [(128, 8, 128), (129, 33, 129), (160, 31, 191), (255, 64, 1001),
                                   (1500, 1300, 160), (4100, 70, 2052)])
def test_tf32_split(M, N, K, ta, tb):
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    s = torch.pow(10.0, 12 * torch.rand(K, generator=g, device="cuda") - 6)
    a = torch.randn(M, K, generator=g, device="cuda") * s
    b = torch.randn(K, N, generator=g, device="cuda") / s[:, None]
    w = a.double() @ b.double()
    c = torch.empty(M, N, device="cuda")
    gemm(a.T.contiguous() if ta else a, b.T.contiguous() if tb else b, c, ta=ta, tb=tb)
    assert ((c.double() - w).norm() / w.norm()).item() <= 1e-6
