"""Sums of the tensor-core GEMM where few tiles leave CTA pairs idle: no further from FP64 than
three TF32 products per operand pair over chunks of 32 values.

The tensor cores truncate as they accumulate, which takes a fraction off every product of
random factors that repeated squaring multiplies by 15 from A to A^16.  For TF32 halves it is
8.7e-8 (measured at all sizes, spread below 2e-9 from 10^4 entries on); it is the part of the
error that lies along the result, <c - w, w> / <w, w>.  The other bound is the relative
Frobenius error of those products, split along K as they were for idle SMs.
"""
import pytest
import torch

from paper_1403_6968_gb300 import gemm

pytestmark = pytest.mark.gpu


def _product(M, N, K):
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    a, b = torch.randn(M, K, generator=g, device="cuda"), torch.randn(K, N, generator=g, device="cuda")
    c = torch.empty(M, N, device="cuda")
    gemm(a, b, c)
    w = a.double() @ b.double()
    return c.double() - w, w


@pytest.mark.parametrize("M,N,K", [(128, 128, 128), (200, 200, 200), (700, 700, 700), (893, 642, 893),
                                   (1000, 1000, 1000), (1300, 1300, 1300), (1654, 113, 1654)])
def test_bias_of_small_products(M, N, K):
    d, w = _product(M, N, K)
    assert abs(((d * w).sum() / (w * w).sum()).item()) <= 8.7e-8


@pytest.mark.parametrize("M,N,K,bound", [(314, 3654, 2299, 1.62e-7), (731, 1533, 1692, 1.55e-7),
                                         (231, 4229, 1691, 1.55e-7), (1718, 819, 2243, 1.72e-7),
                                         (333, 4345, 1430, 1.59e-7)])
def test_long_sums_of_few_tiles(M, N, K, bound):
    d, w = _product(M, N, K)
    assert (d.norm() / w.norm()).item() <= bound
