"""Level products of 9 to 16 columns keep all 24 bits of the view's entries, whatever the
view's size: sums of two entries whose low bits cancel are exact in FP32, and not where an
entry is held in two 11-bit halves.

A = [[0, B], [0, 0]] has A^2 = 0.  With U's column q the two unit rows 2q, 2q + 1 of the lower
half and V's column q another unit row of it, (A + U V^T)^2 = (A U) V^T: column V_q of A^2 is
B[:, 2q] + B[:, 2q + 1].  B's columns alternate between 1 + 4099 2^-23 and 1 + 4101 2^-23,
whose sum 2 + 8200 2^-23 is a float with 11 significant bits below its leading ones, so that
the later update of A^2 (split operands, for 17 to 32 columns) holds it.  Every entry is
compared for equality.
"""
import pytest
import torch

from paper_1403_6968_gb300 import Program

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,r", [(3501, 9), (3584, 12), (3617, 16), (4096, 16), (1000, 12)])
def test_two_term_sums_are_exact(n, r):
    h = n // 2
    a = torch.zeros(n, n, device="cuda")
    a[:h, h:] = 1 + 4099 * 2.0 ** -23
    a[:h, h + 1::2] = 1 + 4101 * 2.0 ** -23
    u, v = torch.zeros(n, r, device="cuda"), torch.zeros(n, r, device="cuda")
    q = torch.arange(r, device="cuda")
    u[h + 2 * q, q] = 1
    u[h + 2 * q + 1, q] = 1
    v[h + 2 * r + q, q] = 1
    prog = Program("power", [a], k=2, r_max=r)
    prog.apply_delta(u, v)
    prog.sync()
    want = torch.zeros(n, n, device="cuda")
    want[:h, h + 2 * r:h + 3 * r] = 2 + 8200 * 2.0 ** -23
    assert torch.equal(prog.read_view(1), want)
    prog.close()
