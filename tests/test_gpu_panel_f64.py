"""Panel kernels of FP64 programs where their tiles change: 45 and 46 tiles of 64 x 64 (rows of 16
or 64 a tile), panels whose row blocks are chosen by their FMAs (few rows, one column tile, a row
past a block), factors of 1 and 8 columns, all strategies.  1e-12 relative Frobenius per view: at
most 8 steps of FP64 sums over 2900 rows (8 x 2900^0.5 x 1.1e-16 = 5e-14)."""
import pytest
import torch

from paper_1403_6968_gb300 import Program

pytestmark = pytest.mark.gpu
K = 8


@pytest.mark.parametrize("strategy", ["factored", "hybrid"])
@pytest.mark.parametrize("n,p,r", [(2880, 64, 1), (2881, 64, 2), (15, 1, 1), (17, 3, 8), (161, 16, 2),
                                   (300, 200, 8), (777, 129, 8), (1025, 33, 1)])
def test_panels(n, p, r, strategy):
    g = torch.Generator(device="cuda").manual_seed(n + p)

    def normal(*shape, scale=1.0):
        return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64) * scale

    a, b, t = normal(n, n, scale=0.5 / n ** 0.5), normal(n, p), normal(n, p)
    prog = Program("iteration", [a, b, t], k=K, r_max=r, precision="f64", strategy=strategy)
    u, v, ub, vb = normal(n, r, scale=0.1), normal(n, r, scale=0.1), normal(n, r), normal(p, r)
    prog.apply_delta(u, v)
    prog.apply_delta(ub, vb, input_id=1)
    prog.sync()
    a, b = a + u @ v.T, b + ub @ vb.T
    for i in range(1, K + 1):
        t = a @ t + b
        got = torch.from_numpy(prog.read_view_host(i)).cuda()
        assert ((got - t).norm() / t.norm()).item() < 1e-12, f"T_{i}"
    prog.close()
