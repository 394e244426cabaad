"""The workloads this library is timed on, each through its public Python entry points.

A case is one call (or the few calls that belong together) that a user's program makes over
and over on a program it keeps: one update of a maintained program and the refresh of all of
its views, one burst of serving requests, one reverse pass, one re-evaluation, one product.
``prepare`` draws the inputs from a seed and builds the program, ``run`` is one pass and
returns the refreshed state itself (zero-copy tensors over the views), ``exact`` is the same
result from the definition in FP64 with plain torch.

Updates alternate: the first pass adds the update, the second takes it away again (for OLS:
puts the old rows back), so that a state can be refreshed any number of times.
"""
import math

import numpy as np
import torch

from paper_1403_6968_gb300 import Program, Server
from paper_1403_6968_gb300.linview import gemm

SIGMA = 0.01  # scale of the factors of an update (the paper's row updates)


def listed():
    return [
        # A^8 in FP64 at n = 256 under row updates: the smallest maintained program, where the
        # time is launches and latency
        dict(name="power_f64_n256_row", kind="update", program="power", dtype="f64", n=256, k=8,
             r=1, row=True),
        # a small ragged FP32 A^16 view under a coalesced rank-3 delta: one request of a server
        # that keeps many views of different sizes
        dict(name="power_f32_n1000_r3", kind="update", program="power", dtype="f32", n=1000, k=16,
             r=3, row=False),
        # the headline: A^16 and the sums S'_2..S'_16 at n = 8192, one changed row of A
        dict(name="powersum_f32_n8192_row", kind="update", program="power_sum", dtype="f32",
             n=8192, k=16, r=1, row=True),
        # the same program under dense rank-4 updates (level factors of 4 to 64 columns)
        dict(name="powersum_f32_n8192_r4", kind="update", program="power_sum", dtype="f32",
             n=8192, k=16, r=4, row=False),
        # serving: one request each for six resident A^16 views of mixed size, their refreshes
        # overlapping on the GPU; factors in host memory
        dict(name="serve_burst_6_views", kind="serve", sizes="1024,2048,4096,1024,2048,1024",
             ranks="1,8,4,5,2,8", k=16),
        # T_{i+1} = A T_i + B, 16 steps, p = 64, a rank-2 update of A (linear model)
        dict(name="iteration_n8192_p64_r2", kind="iteration", dtype="f32", n=8192, p=64, k=16,
             r=2, model="linear", skip=0, strategy="factored", db=False),
        # gradient descent as the general form: wide right-hand sides, one replaced data row is
        # a rank-2 update of A and then a rank-1 update of B (exponential model)
        dict(name="iteration_exp_n4096_p1024", kind="iteration", dtype="f32", n=4096, p=1024,
             k=16, r=2, model="exp", skip=0, strategy="factored", db=True),
        # reverse pass of the 16-step iteration: dL/dA and dL/dB of L = ||T_16||^2
        dict(name="iteration_adjoint_n8192_p64", kind="adjoint", program="iteration", dtype="f32",
             n=8192, p=64, k=16),
        # OLS: 16 rows of a 65536 x 4096 X replaced; W = (X^T X)^-1 and beta refreshed
        dict(name="ols_m65536_n4096_k16", kind="ols", dtype="f32", m=65536, n=4096, p=16, k=16),
        # OLS of ordinary, odd size, one replaced row
        dict(name="ols_m20001_n1503_k1", kind="ols", dtype="f32", m=20001, n=1503, p=1, k=1),
        # re-evaluation of A^16 and its sums: the correction of drift, and requests past the
        # rank cap
        dict(name="reeval_powersum_n8192", kind="reeval", program="power_sum", dtype="f32",
             n=8192, k=16),
        # the library's product on a ragged shape with a transposed operand
        dict(name="gemm_f32_3001x1025x5003_ta", kind="gemm", dtype="f32", M=3001, N=1025, K=5003,
             ta=True, tb=False, beta=0.0),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["update", "update", "update", "serve", "iteration", "iteration", "adjoint",
                       "ols", "reeval", "gemm"])
    if kind == "update":
        f64 = rng.random() < 0.25
        return dict(kind="update", program=rng.choice(["power", "power_sum"]),
                    dtype="f64" if f64 else "f32", n=_logint(rng, 64, 2048 if f64 else 8192),
                    k=rng.choice([4, 8, 16]), r=rng.choice([1, 1, 2, 3, 4, 5, 8]), row=False)
    if kind == "serve":
        count = rng.randint(2, 6)
        return dict(kind="serve", k=16, sizes=",".join(str(_logint(rng, 512, 4096)) for _ in range(count)),
                    ranks=",".join(str(rng.randint(1, 8)) for _ in range(count)))
    if kind == "iteration":
        model, skip = rng.choice([("linear", 0), ("linear", 0), ("exp", 0), ("skip", 4)])
        hybrid = model == "linear" and rng.random() < 0.2
        return dict(kind="iteration", dtype="f32", n=_logint(rng, 256, 4096 if hybrid else 8192),
                    p=_logint(rng, 1, 128 if hybrid else 1024), k=16, r=rng.choice([1, 2, 2, 4]),
                    model=model, skip=skip, strategy="hybrid" if hybrid else "factored",
                    db=rng.random() < 0.3)
    if kind == "adjoint":
        if rng.random() < 0.3:
            return dict(kind="adjoint", program="power", dtype="f32", n=_logint(rng, 200, 4096), p=0,
                        k=rng.choice([4, 8, 16]))
        return dict(kind="adjoint", program="iteration", dtype="f32", n=_logint(rng, 256, 8192),
                    p=_logint(rng, 1, 256), k=rng.choice([4, 8, 16]))
    if kind == "ols":
        n = _logint(rng, 64, 4096)
        return dict(kind="ols", dtype="f32", m=min(65536, n * rng.randint(4, 24) + 1), n=n,
                    p=rng.choice([1, 1, 4, 16]), k=rng.choice([1, 2, 4, 7, 16]))
    if kind == "reeval":
        return dict(kind="reeval", program=rng.choice(["power", "power_sum"]), dtype="f32",
                    n=_logint(rng, 300, 7000), k=rng.choice([4, 8, 16]))
    f64 = rng.random() < 0.15
    hi = 700 if f64 else 6000
    return dict(kind="gemm", dtype="f64" if f64 else "f32", M=_logint(rng, 100, hi),
                N=_logint(rng, 16, hi), K=_logint(rng, 100, hi), ta=rng.random() < 0.5,
                tb=rng.random() < 0.5, beta=rng.choice([0.0, 0.0, -0.5]))


class _Shared:
    """The memory of a view, which the program owns and the tensor over it keeps alive."""

    def __init__(self, owner, ptr, rows, cols, ld, dtype):
        self.owner = owner
        size = 8 if dtype == "f64" else 4
        self.__cuda_array_interface__ = {"shape": (rows, cols), "strides": (ld * size, size),
                                         "typestr": "<f%d" % size, "data": (ptr, False), "version": 2}


def _views(prog, dtype, owner=None):
    """Zero-copy tensors over all views of a program, in the order of their ids."""
    got = []
    for vid in range(prog.num_views()):
        ptr, ld = prog.view_device_ptr(vid)
        rows, cols = prog.view_shape(vid)
        got.append(torch.as_tensor(_Shared(owner or prog, ptr, rows, cols, ld, dtype), device="cuda"))
    return got


def _inputs(case, seed):
    """The inputs of a case, on the GPU (serving: the factors on the host), from the seed alone."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    dt = torch.float64 if case.get("dtype") == "f64" else torch.float32

    def normal(rows, cols, scale=1.0):
        return torch.randn(rows, cols, generator=g, device="cuda", dtype=dt) * scale

    def matrix(n):  # spectral radius about 1/2
        return normal(n, n, 0.5 / math.sqrt(n))

    kind, d = case["kind"], {}
    if kind == "serve":
        d["a"], d["u"], d["v"] = [], [], []
        for n, r in _served(case):
            d["a"].append(matrix(n))
            d["u"].append(normal(n, r, SIGMA).cpu().numpy())
            d["v"].append(normal(n, r, SIGMA).cpu().numpy())
        return d
    if kind == "ols":
        m, n, p, k = case["m"], case["n"], case["p"], case["k"]
        scale = torch.ones(n, device="cuda", dtype=dt)  # a tenth of the columns is small
        scale[torch.randperm(n, generator=g, device="cuda")[: n // 10]] = 1e-2
        d["x"] = normal(m, n) * scale
        d["y"] = normal(m, p)
        d["rows"] = torch.randperm(m, generator=g, device="cuda")[:k].sort().values
        d["new"] = normal(k, n) * scale
        return d
    if kind == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        d["a"] = normal(K, M) if case["ta"] else normal(M, K)
        d["b"] = normal(N, K) if case["tb"] else normal(K, N)
        d["c"] = normal(M, N)
        return d
    n = case["n"]
    d["a"] = matrix(n)
    if case.get("p"):
        d["b"], d["t0"] = normal(n, case["p"]), normal(n, case["p"])
    if kind == "update" and case["row"]:
        d["i"] = int(torch.randint(n, (1,), generator=g, device="cuda"))
        d["v"] = normal(n, 1, SIGMA)
    elif kind in ("update", "iteration"):
        d["u"], d["v"] = normal(n, case["r"], SIGMA), normal(n, case["r"], SIGMA)
        if case.get("db"):
            d["ub"], d["vb"] = normal(n, 1, SIGMA), normal(case["p"], 1, SIGMA)
    if kind == "adjoint" and case["program"] == "power":
        d["g"] = normal(n, n)
    return d


def _served(case):
    return list(zip((int(x) for x in case["sizes"].split(",")),
                    (int(x) for x in case["ranks"].split(","))))


def prepare(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    s = {"case": case, "pass": 0}
    if kind == "gemm":
        return s | d
    if kind == "serve":
        srv = Server(max_inflight=4, r_cap=8)
        s["server"] = srv
        s["ids"] = [srv.add_view(a, k=case["k"]) for a in d["a"]]
        srv.drain()
        s["views"] = [_views(srv.program(i), "f32", owner=srv) for i in s["ids"]]
        s["u"], s["v"] = [d["u"], [-u for u in d["u"]]], d["v"]
        return s
    if kind == "ols":
        s["prog"] = prog = Program("ols", [d["x"], d["y"]], k=case["k"], precision=case["dtype"])
        s["rows"] = d["rows"].cpu().numpy()
        s["new"] = [d["new"], d["x"][d["rows"]].clone()]
        s["views"] = _views(prog, case["dtype"])
        return s
    ins = [d["a"]] + ([d["b"], d["t0"]] if "t0" in d else [])
    more = {}
    if kind == "iteration":
        more = dict(model=case["model"], skip=case["skip"], strategy=case["strategy"])
    prog = Program(case.get("program", "iteration"), ins, k=case["k"], r_max=case.get("r", 1),
                   precision=case["dtype"], **more)
    s["prog"] = prog
    if kind in ("update", "iteration"):
        prog.prepare_updates()
        if "i" in d:
            s["i"], s["v"] = d["i"], [d["v"], -d["v"]]
        else:
            s["u"], s["v"] = [d["u"], -d["u"]], d["v"]
        if "ub" in d:
            s["ub"], s["vb"] = [d["ub"], -d["ub"]], d["vb"]
    if kind == "adjoint":
        s["dA"] = torch.empty_like(d["a"])
        s["dB"] = torch.empty_like(d["b"]) if "b" in d else None
        s["g"] = d.get("g")
    s["views"] = _views(prog, case["dtype"])
    return s


def run(s):
    case = s["case"]
    kind, turn = case["kind"], s["pass"] & 1
    s["pass"] += 1
    if kind == "gemm":
        gemm(s["a"], s["b"], s["c"], beta=case["beta"], ta=case["ta"], tb=case["tb"])
        return s["c"]
    if kind == "serve":
        for vid, u, v in zip(s["ids"], s["u"][turn], s["v"]):
            s["server"].submit(vid, u, v)
        s["server"].drain()
        return s["views"]
    prog = s["prog"]
    if kind == "ols":
        prog.apply_row_block(s["rows"], s["new"][turn])
    elif kind == "reeval":
        prog.reeval()
    elif kind == "adjoint":
        if case["program"] == "power":
            prog.adjoint_power(s["g"], s["dA"])
            return s["dA"]
        prog.adjoint_iteration(dA=s["dA"], dB=s["dB"])
        return [s["dA"], s["dB"]]
    else:
        if "i" in s:
            prog.apply_row_delta(s["i"], s["v"][turn])
        else:
            prog.apply_delta(s["u"][turn], s["v"])
        if "ub" in s:
            prog.apply_delta(s["ub"][turn], s["vb"], input_id=1)
    return s["views"]


def _powers(case):
    return [1 << j for j in range(case["k"].bit_length())]


def _t_views(case):
    """The i of the maintained T_i of an iteration program, and the h of its auxiliary views."""
    k = case["k"]
    if case.get("model", "linear") == "linear":
        return list(range(1, k + 1)), []
    s = k // 2 if case["model"] == "exp" else case["skip"]
    lead = [1 << j for j in range(s.bit_length())]
    return lead + list(range(2 * s, k + 1, s)), lead[1:]


def work(case):
    kind, size = case["kind"], 8 if case.get("dtype") == "f64" else 4
    if kind == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": size * (M * K + K * N + M * N * (2 if case["beta"] else 1)),
                "flops": 2.0 * M * N * K}
    if kind == "ols":
        # W read and written; the replaced rows of X; beta and X^T Y read and written
        n, p, k = case["n"], case["p"], case["k"]
        return {"bytes": size * (2 * n * n + 2 * 2 * n * p + 3 * k * n),
                "flops": 2.0 * 2 * n * n * 2 * k + 3 * 2.0 * n * p * 2 * k}

    def chain(n, k, r, sums):  # App. A: two products below P_k and one update per view
        levels = k.bit_length()
        flops = sum(2.0 * n * n * r * h * ((3 if h < k else 1) + (1 if sums and h > 1 else 0))
                    for h in (1 << j for j in range(levels)))
        views = levels + (levels - 1 if sums else 0)
        return {"bytes": size * (2.0 * views * n * n + 2 * n * r), "flops": flops}

    if kind == "serve":
        all_ = [chain(n, case["k"], r, False) for n, r in _served(case)]
        return {m: sum(w[m] for w in all_) for m in ("bytes", "flops")}
    n, k = case["n"], case["k"]
    if kind == "update":
        return chain(n, k, case["r"], case["program"] == "power_sum")
    if kind == "reeval":
        levels = k.bit_length() - 1
        sums = case["program"] == "power_sum"
        products = levels + (levels - 1 if sums else 0)
        return {"bytes": size * n * n * (1.0 + levels * (2 if sums else 1)),
                "flops": 2.0 * n ** 3 * products}
    p = case["p"]
    if kind == "adjoint":
        if case["program"] == "power":
            levels = k.bit_length() - 1
            return {"bytes": size * n * n * (2.0 + levels), "flops": 4.0 * n ** 3 * levels}
        return {"bytes": size * (2.0 * n * n + n * p * (k + 2)),
                "flops": 2.0 * n * n * p * (k - 1) + 2.0 * n * n * k * p}
    ts, aux = _t_views(case)
    r = case["r"]
    out = {"bytes": size * (2.0 * n * n * (1 + 2 * len(aux)) + 2.0 * n * p * len(ts) + 2 * n * r),
           "flops": 2.0 * n * n * r * k + 4.0 * n * p * r * sum(ts) + 4.0 * n * n * r * sum(aux)}
    if case["db"]:
        out["bytes"] += size * (n * n * (1.0 + 2 * len(aux)) + 2.0 * n * p * len(ts))
        out["flops"] += 2.0 * n * n * k + 4.0 * n * p * sum(ts)
    return out


def exact(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    f = {key: x.double() for key, x in d.items() if isinstance(x, torch.Tensor) and x.is_floating_point()}

    def powers(a, k, sums):
        p, sm, ps, ss = a, a, [a], []
        h = 1
        while h < k:
            if sums:
                sm = p @ sm + sm
                ss.append(sm)
            p = p @ p
            ps.append(p)
            h *= 2
        return ps, ss

    if kind == "gemm":
        c = (f["a"].T if case["ta"] else f["a"]) @ (f["b"].T if case["tb"] else f["b"])
        return c + case["beta"] * f["c"] if case["beta"] else c
    if kind == "serve":
        got = []
        for a, u, v in zip(d["a"], d["u"], d["v"]):
            u, v = (torch.from_numpy(np.asarray(x, dtype=np.float64)).cuda() for x in (u, v))
            got.append(powers(a.double() + u @ v.T, case["k"], False)[0])
        return got
    if kind == "ols":
        x = f["x"]
        x[d["rows"]] = f["new"]
        z, xty = x.T @ x, x.T @ f["y"]
        w = torch.cholesky_inverse(torch.linalg.cholesky(z))
        return [w, w @ xty, xty, d["x"].index_copy(0, d["rows"], d["new"])]
    a = f["a"]
    if kind == "update":
        if case["row"]:
            a[d["i"]] += f["v"][:, 0]
        else:
            a = a + f["u"] @ f["v"].T
    if kind in ("update", "reeval"):
        ps, ss = powers(a, case["k"], case["program"] == "power_sum")
        return ps + ss
    k = case["k"]
    if kind == "adjoint" and case["program"] == "power":
        ps, g = powers(a, k // 2, False)[0], f["g"]
        for p in reversed(ps):
            g = g @ p.T + p.T @ g
        return g
    b = f["b"]
    if kind == "iteration":
        a = a + f["u"] @ f["v"].T
        if case["db"]:
            b = b + f["ub"] @ f["vb"].T
    ts = [f["t0"]]
    for _ in range(k):
        ts.append(a @ ts[-1] + b)
    if kind == "adjoint":
        g, da, db = 2 * ts[k], torch.zeros_like(a), torch.zeros_like(b)
        for i in range(k, 0, -1):
            da += g @ ts[i - 1].T
            db += g
            g = a.T @ g
        return [da, db]
    kept, aux = _t_views(case)
    out = [a] + [ts[i] for i in kept] + [b, ts[0]]
    if aux:
        ps, ss = powers(a, aux[-1], True)
        out += ps[1:] + ss
    return out
