"""Updates of B wider than one products pass takes (16 columns in FP32, 8 in FP64) in the
exponential and skip models, whose product S' U_b then runs in several passes: the widths
around the pass's limit and the largest a program accepts (r_max k = 128), on row remainders,
twice in a row (eager capture, then the replayed graph).

Tolerance: relative Frobenius per view against the FP64 recurrence, 1e-5 in FP32 and 1e-10 in
FP64 (an update leaves a few roundings per step over at most 8 steps).
"""
import pytest
import torch

from paper_1403_6968_gb300 import Program

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [129, 700])
@pytest.mark.parametrize("precision,model,k,skip,r", [
    ("f32", "exp", 4, 0, 17), ("f32", "exp", 4, 0, 20), ("f32", "exp", 4, 0, 32),
    ("f32", "skip", 4, 2, 32), ("f32", "exp", 8, 0, 16), ("f64", "exp", 4, 0, 9),
    ("f64", "exp", 4, 0, 32), ("f64", "exp", 8, 0, 12), ("f64", "skip", 8, 4, 16)])
def test_wide_updates_of_b(n, precision, model, k, skip, r):
    dt = torch.float64 if precision == "f64" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(n + r)

    def normal(*shape, scale=1.0):
        return torch.randn(*shape, generator=g, device="cuda", dtype=dt) * scale

    p = 21
    a, b, t0 = normal(n, n, scale=0.4 / n ** 0.5), normal(n, p), normal(n, p)
    prog = Program("iteration", [a, b, t0], k=k, r_max=r, precision=precision, model=model, skip=skip)
    kept = [1, 2, 4, 8][: k.bit_length()]
    a, b = a.double(), b.double()
    for _ in range(2):
        ub, vb = normal(n, r, scale=0.1), normal(p, r, scale=0.1)
        prog.apply_delta(ub, vb, input_id=1)
        prog.sync()
        b = b + ub.double() @ vb.double().T
        t, at = t0.double(), 1
        for i in range(1, k + 1):
            t = a @ t + b
            if i in kept:
                err = ((prog.read_view(at).double() - t).norm() / t.norm()).item()
                assert err < (1e-10 if precision == "f64" else 1e-5), f"T_{i}: {err:.2e}"
                at += 1
    prog.close()
