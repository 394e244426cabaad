"""The tensor-core GEMM on operands with isolated entries far below their neighbours (fewer than
eight of 32 along a row and along a column) that meet zeros and small entries of the other
operand, where FP16 halves would leave such a product with a few bits; and the inner lengths
whose last run of FP16 values is short.

Bound per entry: |C - W| <= 4e-6 sum_k |a||b|, W in FP64.  22-bit operands and the dropped
product of the low halves leave 3 x 2^-22 = 7e-7, truncation over a chunk of 64 values (24
tensor-core steps at 2^-24 each) 1.4e-6 at most, FP32 sums of up to 16 chunks 1e-6; an entry
2^-20 below its neighbours in FP16 halves is off by 2^-20 = 9.5e-7 of itself and one 2^-24
below by 1.5e-5.
"""
import numpy as np
import pytest
import torch

from paper_1403_6968_gb300 import gemm

pytestmark = pytest.mark.gpu
TOL = 4e-6


def _check(a, b, ta=False, tb=False):
    A, B = a.double(), b.double()
    w, scale = A @ B, A.abs() @ B.abs()
    c = torch.empty(a.shape[0], b.shape[1], device="cuda")
    gemm(a.T.contiguous() if ta else a, b.T.contiguous() if tb else b, c, ta=ta, tb=tb)
    assert ((c.double() - w).abs() <= TOL * scale).all()


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


@pytest.mark.parametrize("small_right", [False, True])
@pytest.mark.parametrize("n", [129, 143, 200, 256, 333])
@pytest.mark.parametrize("size", [1e-7, 1e-9, 1e-11])
def test_dense_times_permutation(size, n, small_right):
    """One entry in 40 of a dense operand is small; the other operand picks every entry alone."""
    g = torch.Generator(device="cuda").manual_seed(n)
    a = _normal(g, n, n)
    a = torch.where(torch.rand(n, n, generator=g, device="cuda") < 1 / 40, a * size, a)
    p = torch.eye(n, device="cuda")[torch.randperm(n, generator=g, device="cuda")]
    _check(p, a) if small_right else _check(a, p)


@pytest.mark.parametrize("ta,tb", [(False, False), (True, True)])
@pytest.mark.parametrize("per32", [1, 3, 7])
@pytest.mark.parametrize("M,N,K", [(192, 96, 256), (130, 70, 333), (300, 40, 135)])
def test_isolated_entries_meet_only_rows(M, N, K, per32, ta, tb):
    """per32 entries of 32 in some rows of A are 1e-10 beside entries of about 1, in columns that
    are zero elsewhere; B has rows of 1e10 there and zeros in the others."""
    g = torch.Generator(device="cuda").manual_seed(per32 + K)
    a, b = _normal(g, M, K), torch.zeros(K, N, device="cuda")
    cols = torch.cat([torch.arange(k, min(k + per32, K), device="cuda") for k in range(5, K, 32)])
    rows = torch.arange(3, M, 32 // per32 if per32 < 7 else 5, device="cuda")
    a[:, cols] = 0
    a[rows[:, None], cols] = 1e-10 * _normal(g, len(rows), len(cols))
    b[cols] = 1e10 * _normal(g, len(cols), N)
    _check(a, b, ta, tb)


@pytest.mark.parametrize("ta,tb", [(False, False), (True, True), (True, False), (False, True)])
@pytest.mark.parametrize("K", [128, 129, 130, 136, 143, 144, 191, 192, 193, 199, 207, 208, 321])
def test_short_last_runs(K, ta, tb):
    """Dense operands, and operands that are large in the last values of K alone."""
    g = torch.Generator(device="cuda").manual_seed(K)
    a, b = _normal(g, 150, K), _normal(g, K, 72)
    _check(a, b, ta, tb)
    a[:, : K - 20] *= 1e-3
    b[K - 3:] *= 1e4
    _check(a, b, ta, tb)


@pytest.mark.parametrize("ta,tb", [(False, False), (True, True)])
@pytest.mark.parametrize("scale", [30, 300, 3e3, 1e5])
@pytest.mark.parametrize("n", [256, 400, 529])
def test_outlier_rows(n, scale, ta, tb):
    """Rows far larger than the others, a diagonal far larger than the rest: small entries beside
    a large one in the runs of one side, dense runs in those of the other."""
    g = torch.Generator(device="cuda").manual_seed(n)
    a, b = _normal(g, n, n), _normal(g, n, n)
    a[7::61] *= scale
    _check(a, a, ta, tb)
    b.diagonal().mul_(scale)
    _check(a, b, ta, tb)
    _check(b, b, ta, tb)


@pytest.mark.parametrize("n,p", [(256, 33), (300, 64), (1024, 17), (327, 40)])
def test_chain(n, p):
    """G <- A^T G with a diagonal A: the product that is split for the next one by the kernel
    that finishes it has isolated entries of 2^-27 (k + c a multiple of 16, k one of 5)."""
    from paper_1403_6968_gb300 import Program
    k = 2
    rng = np.random.default_rng(n)
    d = rng.uniform(1, 2, n) * np.where(np.arange(n) % 5, 1, 2.0 ** -11)
    x = rng.uniform(1, 2, (n, p))
    x[(np.arange(n)[:, None] + np.arange(p)) % 16 == 0] *= 2.0 ** -16
    a, seed, d64 = np.diag(d).astype(np.float32), x.astype(np.float32), d.astype(np.float32)
    zero = torch.zeros(n, p, device="cuda")
    prog = Program("iteration", [torch.from_numpy(a).cuda(), zero, zero], k=k, r_max=1)
    dT0 = torch.empty(n, p, device="cuda")
    prog.adjoint_iteration_seed(torch.from_numpy(seed).cuda(), dA=torch.empty(n, n, device="cuda"),
                                dB=torch.empty(n, p, device="cuda"), dT0=dT0)
    prog.sync()
    ref = d64.astype(np.float64)[:, None] ** k * seed
    assert (np.abs(dT0.cpu().numpy() - ref) <= k * TOL * np.abs(ref)).all()
    prog.close()
