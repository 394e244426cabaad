"""Writes of the hybrid iteration stay inside the program's own blocks: every block that the
caller's allocator hands out is followed by a guard, which must be untouched after updates of
A and of B.  Its products T_{i-1}^T V go over one panel of p columns, which is cut into more
row blocks than the k panels that the other strategy takes at once; the sizes are those where
the partial sums of one panel are the larger ones (n = 4096, k = 16: p = 1024 has 37 blocks of
1024 columns, the k panels 2 blocks of 16384).

Tolerance: relative Frobenius per view, 1e-5 in FP32 and 1e-10 in FP64 (one update each leaves
a few roundings per step over at most 16 steps of a contraction).
"""
import pytest
import torch

from paper_1403_6968_gb300 import Program
from paper_1403_6968_gb300 import _lib as L
from paper_1403_6968_gb300 import linview

pytestmark = pytest.mark.gpu

GUARD = 1 << 18


class _Guarded:
    """Allocator callbacks over torch tensors, each with GUARD bytes of a pattern behind it."""

    def __init__(self):
        self.blocks = {}
        self.callbacks = (L.ALLOC_FN(self._alloc), L.FREE_FN(self._free))

    def _alloc(self, nbytes, stream, ctx):
        t = torch.full((int(nbytes) + GUARD,), 0xA5, dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        self.blocks[t.data_ptr()] = (t, int(nbytes))
        return t.data_ptr()

    def _free(self, ptr, nbytes, stream, ctx):
        torch.cuda.synchronize()
        self.blocks.pop(int(ptr))

    def touched(self):
        return [n for t, n in self.blocks.values() if not bool((t[n:] == 0xA5).all())]


@pytest.mark.parametrize("n,p,k,r,precision", [
    (4096, 1024, 16, 1, "f32"), (4096, 1024, 16, 2, "f32"), (3000, 809, 16, 1, "f32"),
    (4096, 609, 16, 1, "f64"), (2500, 1345, 2, 2, "f32"), (4096, 1280, 8, 1, "f32")])
def test_hybrid_writes_stay_inside(n, p, k, r, precision, monkeypatch):
    guarded = _Guarded()
    monkeypatch.setattr(linview, "_torch_allocator", lambda: guarded.callbacks)
    dt = torch.float64 if precision == "f64" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(n + p)

    def normal(*shape, scale=1.0):
        return torch.randn(*shape, generator=g, device="cuda", dtype=dt) * scale

    a, b, t0 = normal(n, n, scale=0.4 / n ** 0.5), normal(n, p), normal(n, p)
    u, v = normal(n, r, scale=0.01), normal(n, r, scale=0.01)
    ub, vb = normal(n, r, scale=0.1), normal(p, r, scale=0.1)
    prog = Program("iteration", [a, b, t0], k=k, r_max=r, precision=precision, strategy="hybrid")
    prog.apply_delta(u, v)
    prog.apply_delta(ub, vb, input_id=1)
    prog.sync()
    assert guarded.blocks and guarded.touched() == []
    a, b, t = (a.double() + u.double() @ v.double().T, b.double() + ub.double() @ vb.double().T,
               t0.double())
    for i in range(1, k + 1):
        t = a @ t + b
        err = ((prog.read_view(i).double() - t).norm() / t.norm()).item()
        assert err < (1e-10 if precision == "f64" else 1e-5), f"T_{i}: {err:.2e}"
    prog.close()
