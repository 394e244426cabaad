"""Panel kernels of the general form (M = T^T V and T += K M^T) at the edges of
their tiles: right-hand sides narrower than one lane's columns, just past one
CTA's 128 columns, unaligned widths, a single row block, updates of A and of B
in every model and strategy, against the FP64 oracle's re-evaluation.

Tolerances: FP64 1e-10 and FP32 1e-5 relative Frobenius per view (one update in
FP32 leaves a few roundings of 6e-8 per step over at most 8 steps).
"""
import numpy as np
import pytest
import torch

import linview_inputs as li
from oracle import iteration as oi
from oracle.metrics import rel_frob
from paper_1403_6968_gb300 import Program

pytestmark = pytest.mark.gpu

SHAPES = [  # n, p, r
    (64, 1, 1),     # one row block, one column
    (65, 3, 8),     # row remainder, columns of an unaligned panel
    (200, 129, 3),  # one column past a 128-column tile
    (333, 64, 2),
    (130, 1000, 4),
]


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("model,strategy", [("linear", "factored"), ("linear", "hybrid"),
                                            ("exp", "factored"), ("skip", "factored")])
@pytest.mark.parametrize("n,p,r", SHAPES)
def test_panel_products(n, p, r, model, strategy, precision):
    k = 8
    dt = np.float32 if precision == "f32" else np.float64
    a, b, t0 = li.iteration_inputs(n, p, seed=n + p, dtype=dt)
    prog = Program("iteration", [torch.from_numpy(x).cuda() for x in (a, b, t0)], k=k, r_max=r,
                   precision=precision, model=model, strategy=strategy,
                   skip=4 if model == "skip" else 0)
    (u, v), = li.lowrank_update_stream(n, r, 1, seed=2, dtype=dt)
    prog.apply_delta(torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda())
    (ub, vb), = li.lowrank_update_stream(n, r, 1, seed=3, sigma=0.1, dtype=dt, n_cols=p)
    prog.apply_delta(torch.from_numpy(ub).cuda(), torch.from_numpy(vb).cuda(), input_id=1)
    prog.sync()
    d = lambda x: x.astype(np.float64)  # noqa: E731
    ref = oi.reeval(d(a) + d(u) @ d(v).T, d(b) + d(ub) @ d(vb).T, d(t0), k)
    kept = {"linear": range(1, k + 1), "exp": (1, 2, 4, 8), "skip": (1, 2, 4, 8)}[model]
    tol = 1e-5 if precision == "f32" else 1e-10
    for j, i in enumerate(kept):
        err = rel_frob(prog.read_view_host(1 + j), ref[i])
        assert err < tol, f"T_{i}: {err:.2e}"
    prog.close()
