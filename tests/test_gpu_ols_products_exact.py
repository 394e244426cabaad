"""G = W U of a wide row-block replacement (17 to 32 factor columns) keeps all 24 bits of W's
entries, whatever the size.

X is diagonal (s_j, so W_jj = 1 / s_j^2 =: w_j) above k zero rows, whose responses are 1 and
which are replaced by distinct unit rows e_j.  Then X^T Y goes from 0 to e_j's and beta_j from 0
to w_j / (1 + w_j) = (W U)_j (1 - w_j + ..): w_j of about 1e-6 is rounded to FP32 once, its
product with the unit row is exact, and beta is rounded once more: 2^-24 each, 1.3e-7 in all with
what terms of 1e-6 leave.  The w_j chosen have mantissas below 1.25 whose lowest 13 bits begin and
end in ones, of which two 11-bit halves hold 11: a product through those is off by 3 2^-23 / 1.25,
2.8e-7.
"""
import numpy as np
import pytest
import torch

from paper_1403_6968_gb300 import Program

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k,p", [(2048, 9, 1), (2048, 16, 3), (2500, 12, 1), (1000, 16, 1)])
def test_beta_of_unit_rows(n, k, p):
    g = np.random.default_rng(n + k)
    s = (1024 * (1 + g.random(20000))).astype(np.float32)
    w = (1 / s.astype(np.float64) ** 2).astype(np.float32).view(np.uint32)
    fit = ((w & 0x600000) == 0) & ((w & 0x1000) != 0) & ((w & 3) == 3)
    d = s[~fit][:n]
    at = np.sort(g.permutation(n)[:k])
    d[at] = s[fit][:k]
    x = torch.zeros(n + k, n, device="cuda")
    x[:n] = torch.diag(torch.from_numpy(d).cuda())
    y = torch.zeros(n + k, p, device="cuda")
    y[n:] = 1
    new = torch.zeros(k, n, device="cuda")
    new[torch.arange(k), torch.from_numpy(at).cuda()] = 1
    prog = Program("ols", [x, y], k=k)
    prog.apply_row_block(np.arange(n, n + k), new)
    prog.sync()
    got = prog.read_view_host(1).astype(np.float64)
    wj = 1 / d[at].astype(np.float64) ** 2
    want = np.zeros(n)
    want[at] = wj / (1 + wj)
    assert np.abs(got - want[:, None])[np.setdiff1d(np.arange(n), at)].max() == 0
    assert (np.abs(got[at] - want[at, None]) / want[at, None]).max() <= 1.3e-7
    prog.close()
