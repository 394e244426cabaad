"""The tensor-core products pass at 9 to 16 factor columns (its narrowest tile) and
around the size from which such levels take it, through a program's update: A^8 at rank
r has levels of 1, 2, 4 r columns, so r = 3, 4 reach 12 and 16 columns at P_4.

Tolerance 1e-5 relative Frobenius per view against FP64 products of the updated
matrix (three FP32 levels; measured about 1e-6 in the FP32 programs).
"""
import numpy as np
import pytest

from oracle.metrics import rel_frob

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,r", [(3499, 3), (3501, 3), (3584, 4), (3617, 4)])
def test_products_of_9_to_16_columns(n, r):
    from paper_1403_6968_gb300 import Program
    g = torch.Generator(device="cuda").manual_seed(n + r)
    a = torch.randn(n, n, generator=g, device="cuda") * (0.5 / n ** 0.5)
    u = torch.randn(n, r, generator=g, device="cuda") * 0.01
    v = torch.randn(n, r, generator=g, device="cuda") * 0.01
    prog = Program("power", [a], k=8, r_max=r)
    prog.apply_delta(u, v)
    prog.sync()
    p = a.double() + u.double() @ v.double().T
    for j in range(4):
        got = prog.read_view(j)
        assert rel_frob(got.cpu().numpy(), p.cpu().numpy()) < 1e-5, f"view {j}"
        p = p @ p
    prog.close()
