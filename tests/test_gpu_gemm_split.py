"""The tensor-core GEMM's operand split at its edges: tile remainders of the CTA
pair (a second CTA without rows, one row or column past a tile, the shortest
inner lengths, split K), and operands whose entries differ so much in size that
FP16 halves would lose them, which must run on TF32 halves.

Tolerance 1e-6 relative Frobenius (per scaled row or column where those differ in
size) as for the library's other FP32 products: 22-bit operands leave ~2e-7 and FP32
accumulation ~3e-7 at K = 8192, while a lost half leaves ~5e-4.
"""
import numpy as np
import pytest

from oracle.metrics import rel_frob

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 1e-6


def _gemm(a, b, ta=False, tb=False):
    from paper_1403_6968_gb300 import gemm
    m, n = a.shape[1 if ta else 0], b.shape[0 if tb else 1]
    c = torch.empty(m, n, device="cuda")
    gemm(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), c, ta=ta, tb=tb)
    return c.cpu().numpy()


@pytest.mark.parametrize("ta,tb", [(False, False), (True, True)])
@pytest.mark.parametrize("M,N,K", [(128, 8, 128), (129, 65, 129), (256, 256, 191), (257, 257, 192),
                                   (384, 129, 2049), (1, 64, 200), (513, 1025, 333), (300, 40, 5000)])
def test_tile_edges(M, N, K, ta, tb):
    g = np.random.default_rng(M + N + K)
    a = g.standard_normal((K, M) if ta else (M, K)).astype(np.float32)
    b = g.standard_normal((N, K) if tb else (K, N)).astype(np.float32)
    ref = (a.T if ta else a).astype(np.float64) @ (b.T if tb else b).astype(np.float64)
    assert rel_frob(_gemm(a, b, ta, tb), ref) <= TOL


@pytest.mark.parametrize("ta", [False, True])
@pytest.mark.parametrize("decades", [3, 6, 12])
def test_scaled_inner_index(decades, ta):
    """Columns of A and rows of B scaled inversely: every term of the sums counts
    alike, however small A's entry is beside its row's largest."""
    g = np.random.default_rng(1)
    M, N, K = 300, 200, 640
    s = 10.0 ** g.integers(-decades, decades + 1, K)
    a = (g.standard_normal((M, K)) * s).astype(np.float32)
    b = (g.standard_normal((K, N)) / s[:, None]).astype(np.float32)
    ref = a.astype(np.float64) @ b.astype(np.float64)
    assert rel_frob(_gemm(np.ascontiguousarray(a.T) if ta else a, b, ta), ref) <= TOL


def test_scaled_rows_and_columns():
    """Rows of A and columns of B of very different size: each keeps its accuracy."""
    g = np.random.default_rng(2)
    M, N, K = 260, 140, 300
    sa, sb = 10.0 ** g.integers(-14, 15, M), 10.0 ** g.integers(-14, 15, N)
    a = (g.standard_normal((M, K)) * sa[:, None]).astype(np.float32)
    b = (g.standard_normal((K, N)) * sb).astype(np.float32)
    ref = a.astype(np.float64) @ b.astype(np.float64)
    got = _gemm(a, b)
    for i in range(0, M, 13):
        cols = np.abs(np.log10(sb)) <= 14
        d = (got[i, cols] - ref[i, cols]) / sb[cols]
        assert np.linalg.norm(d) <= 4 * TOL * np.linalg.norm(ref[i, cols] / sb[cols])


def test_small_block():
    """A block of small entries in the rows of large ones, met by zeros of B."""
    g = np.random.default_rng(3)
    n = 256
    a = g.standard_normal((n, n)).astype(np.float32)
    a[:, : n // 2] *= np.float32(1e-9)
    b = g.standard_normal((n, n)).astype(np.float32)
    b[n // 2:, : n // 2] = 0
    ref = a.astype(np.float64) @ b.astype(np.float64)
    got = _gemm(a, b)
    assert rel_frob(got[:, : n // 2], ref[:, : n // 2]) <= TOL


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_non_finite(value):
    g = np.random.default_rng(4)
    a = g.standard_normal((200, 256)).astype(np.float32)
    b = g.standard_normal((256, 96)).astype(np.float32)
    a[17, 40] = value
    got = _gemm(a, b)
    assert not np.isfinite(got[17]).any()
    rest = np.delete(np.arange(200), 17)
    assert rel_frob(got[rest], a[rest].astype(np.float64) @ b.astype(np.float64)) <= TOL


def test_tf32_split_reused():
    """A split kept for several products (A^T in the adjoint of the iteration) whose
    operands need TF32: A scaled by a similarity over 24 decades."""
    from oracle import iteration as oi
    import linview_inputs as li
    from paper_1403_6968_gb300 import Program
    n, p, k = 256, 24, 6
    a, b, t0 = li.iteration_inputs(n, p, seed=5)
    s = 10.0 ** np.random.default_rng(6).integers(-12, 13, n)
    a, b, t0 = (x.astype(np.float32) for x in (a * s[:, None] / s, b * s[:, None], t0 * s[:, None]))
    prog = Program("iteration", [torch.from_numpy(x).cuda() for x in (a, b, t0)], k=k, r_max=1)
    seed = (np.random.default_rng(7).standard_normal((n, p)) / s[:, None]).astype(np.float32)
    dA, dB = torch.empty(n, n, device="cuda"), torch.empty(n, p, device="cuda")
    prog.adjoint_iteration_seed(torch.from_numpy(seed).cuda(), dA=dA, dB=dB)
    prog.sync()
    A, B, T = (x.astype(np.float64) for x in (a, b, t0))
    ts = oi.reeval(A, B, T, k)
    G, rA, rB = seed.astype(np.float64), 0.0, 0.0
    for i in range(k, 0, -1):
        rA, rB = rA + G @ (ts[i - 1] if i > 1 else T).T, rB + G
        G = A.T @ G
    scale = s[:, None]
    assert rel_frob(dB.cpu().numpy() * scale, rB * scale) <= 5 * TOL
    assert rel_frob(dA.cpu().numpy() * scale / s, rA * scale / s) <= 5 * TOL
    prog.close()


@pytest.mark.parametrize("model", ["linear", "exp"])
@pytest.mark.parametrize("n,p", [(128, 8), (300, 33), (1000, 64), (513, 65), (1537, 17)])
def test_chain_split(n, p, model):
    """Chains T_i = A T_{i-1} + B and G_i = A^T G_{i+1}: the kernel that finishes a
    product (p <= 64: tile remainders, rows past the last run, one row past a tile)
    also splits it for the next one.  k rounds of 3e-7 each: 5 x the tolerance."""
    from oracle import iteration as oi
    import linview_inputs as li
    from paper_1403_6968_gb300 import Program
    k = 4
    a, b, t0 = (x.astype(np.float32) for x in li.iteration_inputs(n, p, seed=n + p))
    prog = Program("iteration", [torch.from_numpy(x).cuda() for x in (a, b, t0)], k=k, r_max=1,
                   model=model)
    A, B, T = (x.astype(np.float64) for x in (a, b, t0))
    ts = oi.reeval(A, B, T, k)
    if model == "linear":
        assert rel_frob(prog.read_view(k).cpu().numpy(), ts[k]) <= 5 * TOL
    seed = np.random.default_rng(8).standard_normal((n, p)).astype(np.float32)
    dA, dB = torch.empty(n, n, device="cuda"), torch.empty(n, p, device="cuda")
    dT0 = torch.empty(n, p, device="cuda")
    prog.adjoint_iteration_seed(torch.from_numpy(seed).cuda(), dA=dA, dB=dB, dT0=dT0)
    prog.sync()
    G, rA, rB = seed.astype(np.float64), 0.0, 0.0
    for i in range(k, 0, -1):
        rA, rB, G = rA + G @ ts[i - 1].T, rB + G, A.T @ G
    for got, ref in ((dA, rA), (dB, rB), (dT0, G)):
        assert rel_frob(got.cpu().numpy(), ref) <= 5 * TOL
    prog.close()


def test_chain_split_turns_to_tf32():
    """The first product of the chain has FP16 halves, its result (rows over eight
    decades) needs TF32: the flag that a product leaves for the next one, while other
    blocks of the same launch still go by its own."""
    from oracle import iteration as oi
    import linview_inputs as li
    from paper_1403_6968_gb300 import Program
    n, p, k = 1000, 48, 4
    a, b, t0 = li.iteration_inputs(n, p, seed=9)
    s = 10.0 ** np.random.default_rng(10).uniform(-4, 4, n)
    a, b, t0 = (x.astype(np.float32) for x in (a * s, 0 * b, t0))
    prog = Program("iteration", [torch.from_numpy(x).cuda() for x in (a, b, t0)], k=k, r_max=1)
    seed = np.random.default_rng(11).standard_normal((n, p)).astype(np.float32)
    dB, dT0 = torch.empty(n, p, device="cuda"), torch.empty(n, p, device="cuda")
    dA = torch.empty(n, n, device="cuda")
    prog.adjoint_iteration_seed(torch.from_numpy(seed).cuda(), dA=dA, dB=dB, dT0=dT0)
    prog.sync()
    G, rB = seed.astype(np.float64), 0.0
    for i in range(k, 0, -1):
        rB, G = rB + G, a.astype(np.float64).T @ G
    assert rel_frob(dT0.cpu().numpy() / s[:, None], G / s[:, None]) <= 5 * TOL
    assert rel_frob(dB.cpu().numpy() / s[:, None], rB / s[:, None]) <= 5 * TOL
    prog.close()
