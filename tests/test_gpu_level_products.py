"""Wide levels on the tensor cores with their splits in one launch: views whose two products
passes run side by side (fewer CTAs than SMs, up to n = 2688 on 152 SMs) and just past that,
one tile and one row past it, 17 to 64 columns, two updates in a row.

Tolerance 1e-5 relative Frobenius per view against FP64 products of the updated matrix.
"""
import pytest
import torch

from paper_1403_6968_gb300 import Program

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("program", ["power", "power_sum"])
@pytest.mark.parametrize("n,k,r", [(33, 8, 8), (128, 16, 3), (129, 16, 8), (1000, 16, 5),
                                   (2688, 8, 5), (2689, 8, 8)])
def test_wide_levels(program, n, k, r):
    g = torch.Generator(device="cuda").manual_seed(n + r)
    a = torch.randn(n, n, generator=g, device="cuda") * (0.5 / n ** 0.5)
    prog = Program(program, [a], k=k, r_max=r)
    a = a.double()
    for _ in range(2):
        u = torch.randn(n, r, generator=g, device="cuda") * 0.01
        v = torch.randn(n, r, generator=g, device="cuda") * 0.01
        prog.apply_delta(u, v)
        a = a + u.double() @ v.double().T
    prog.sync()
    powers, sums, h = [a], [a], 1
    while h < k:
        sums.append(powers[-1] @ sums[-1] + sums[-1])
        powers.append(powers[-1] @ powers[-1])
        h *= 2
    want = powers + (sums[1:] if program == "power_sum" else [])
    for i, w in enumerate(want):
        err = ((prog.read_view(i).double() - w).norm() / w.norm()).item()
        assert err < 1e-5, f"view {i}: {err:.2e}"
    prog.close()
