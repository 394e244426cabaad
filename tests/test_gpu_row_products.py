"""X = P F over whole rows (the Krylov chain of the iteration): columns around one 1024-wide
chunk, row remainders, views of a few rows, every compiled factor width and the widths and
sizes just past them (which take the strip passes), against the definition in FP64.

Tolerance: relative Frobenius per view; one update in FP32 leaves a few roundings of 6e-8 per
step over four steps, 1e-5 in all.
"""
import pytest
import torch

from paper_1403_6968_gb300 import Program

pytestmark = pytest.mark.gpu

K = 4
SIZES = [(5, 1), (31, 2), (127, 4), (1021, 2), (1024, 1), (1025, 3), (2051, 4), (4096, 3),
         (4097, 4), (1300, 5), (8191, 2), (8193, 2), (8193, 1)]


@pytest.mark.parametrize("n,r", SIZES)
@pytest.mark.parametrize("model", ["linear", "exp"])
def test_row_products(n, r, model):
    g = torch.Generator(device="cuda").manual_seed(100 * n + r)

    def normal(*shape, scale=1.0):
        return torch.randn(*shape, generator=g, device="cuda") * scale

    p = 3
    a, b, t0 = normal(n, n, scale=0.5 / n ** 0.5), normal(n, p), normal(n, p)
    prog = Program("iteration", [a, b, t0], k=K, r_max=r, model=model)
    u, v = normal(n, r, scale=0.05), normal(n, r, scale=0.05)
    ub, vb = normal(n, r, scale=0.05), normal(p, r, scale=0.05)
    prog.apply_delta(u, v)
    prog.apply_delta(ub, vb, input_id=1)
    prog.sync()
    a, b, t = a.double() + u.double() @ v.double().T, b.double() + ub.double() @ vb.double().T, t0.double()
    kept = range(1, K + 1) if model == "linear" else (1, 2, 4)
    at = 1
    for i in range(1, K + 1):
        t = a @ t + b
        if i in kept:
            got = torch.from_numpy(prog.read_view_host(at)).cuda().double()
            err = ((got - t).norm() / t.norm()).item()
            assert err < 1e-5, f"T_{i}: {err:.2e}"
            at += 1
    prog.close()
