"""The assembly of a level's new factors where its form changes: 256-row CTAs x columns around 76
with many partial sets, few sets, and remainders of 256 and 32 rows, against FP64.

Tolerance 1e-5 relative Frobenius per view (FP32, one update over two squarings or three linear
steps: a few roundings of 6e-8 per step), 1e-12 for FP64.
"""
import pytest
import torch

from paper_1403_6968_gb300 import Program

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,n,r,model", [
    ("f32", 2304, 8, "linear"), ("f32", 2305, 8, "linear"), ("f32", 1024, 16, "linear"),
    ("f32", 1025, 16, "linear"), ("f32", 1281, 16, "linear"), ("f32", 33, 8, "linear"),
    ("f32", 2433, 8, "exp"), ("f64", 1025, 16, "linear"), ("f64", 769, 16, "linear")])
def test_assembly(precision, n, r, model):
    dt = torch.float32 if precision == "f32" else torch.float64
    g = torch.Generator(device="cuda").manual_seed(n + r)

    def normal(*shape, scale=1.0):
        return torch.randn(*shape, generator=g, device="cuda", dtype=dt) * scale

    a = normal(n, n, scale=0.5 / n ** 0.5)
    prog = Program("power", [a], k=4, r_max=r, precision=precision, model=model)
    u, v = normal(n, r, scale=0.1), normal(n, r, scale=0.1)
    prog.apply_delta(u, v)
    prog.sync()
    w = a.double() + u.double() @ v.double().T
    powers = [w, w @ w, w @ w @ w, w @ w @ w @ w]
    want = powers if model == "linear" else [powers[0], powers[1], powers[3]]
    for i, ref in enumerate(want):
        got = torch.from_numpy(prog.read_view_host(i)).cuda().double()
        err = ((got - ref).norm() / ref.norm()).item()
        assert err < (1e-5 if precision == "f32" else 1e-12), f"view {i}: {err:.2e}"
    prog.close()
