"""Performance cases: the calls a user of this solver makes, over the range of
sizes and options it is used with, each with its inputs and the values it
should return.

A case is a dict of plain values.  ``prepare`` makes what a program holds
before the call (on the GPU, from a seed), ``run`` makes the call through the
Python binding, ``work`` counts the bytes and flops that any implementation
of the call needs, and ``exact`` gives the call's results from 64-bit torch
arithmetic (or the known solution of the generated problem).

Problems are A = U diag(sigma) V^T with U close to orthonormal, sigma
log-spaced from 1 to 1/kappa, b = A x_* + r with r orthogonal to range(A) and
||r|| = rho ||x_*||.  kappa stays at or below 1e6, where the least-squares
solution of the FP64 data is determined to better than 1e-9.
"""
import math

import numpy as np
import torch

import paper_2603_16644_gb300 as lsq

_KIND = {"gaussian": lsq.GAUSSIAN, "sparse": lsq.SPARSE_SIGN, "srft": lsq.SRFT}
_PREC = {"fp8": lsq.FP8_E4M3, "bf16": lsq.BF16, "fp16": lsq.FP16, "fp32": lsq.FP32, "fp64": lsq.FP64,
         "auto_sketch": lsq.AUTO_SKETCH}
DEV = "cuda"


def listed():
    return [
        # One small solve at a time (the paper's 1000 x 100 experiments): launches and latency.
        {"name": "pne_1000x100", "op": "solve", "method": "pne", "m": 1000, "n": 100, "kappa": 1e5, "rho": 1e-6,
         "kind": "gaussian", "s": 200, "prec": "fp32", "refine": 0},
        # One training step of the learned precision proposer at its training batch size.
        {"name": "mlp_step_4096", "op": "mlp", "batch": 4096},
        # The low-precision preconditioner's first step alone: a BF16 sparse-sign sketch of a tall matrix.
        {"name": "sketch_sparse_bf16", "op": "sketch", "m": 65536, "n": 1024, "s": 4096, "kind": "sparse",
         "prec": "bf16"},
        # The same step where the estimate asks for a double-precision preconditioner (m = 2^17, n = 2000, s = 2n).
        {"name": "sketch_gaussian_fp64", "op": "sketch", "m": 131072, "n": 2000, "s": 4000, "kind": "gaussian",
         "prec": "fp64"},
        # The QR of that sketch.
        {"name": "precond_qr_fp64", "op": "qr", "s": 4000, "n": 2000},
        # A_p = A R_s^{-1}, A_p^T A_p and A_p^T b of the same problem: a program with its own preconditioner.
        {"name": "trsm_gram_131072x2000", "op": "trsm_gram", "m": 131072, "n": 2000, "hpne": False},
        # The normal equations of the largest problem: Cholesky and the triangular solves.
        {"name": "factor_chol_4096", "op": "factor", "n": 4096, "hpne": False},
        # The half-preconditioned equations: LU with partial pivoting and the triangular solves.
        {"name": "factor_lu_2000", "op": "factor", "n": 2000, "hpne": True},
        # The paper's timing experiment's shape with its sketch (SRFT, s = 3n), solved by HPNE.
        {"name": "hpne_srft_100000x400", "op": "solve", "method": "hpne", "m": 100000, "n": 400, "kappa": 1e5,
         "rho": 1e-6, "kind": "srft", "s": 1200, "prec": "fp32", "refine": 0},
        # Many uneven problems in one call, precisions from the estimate on a sketch.
        {"name": "batched_64_uneven", "op": "batched", "count": 64, "m_max": 40000, "n_max": 512, "shape_seed": 3},
        # One tall-skinny solve with a low-precision sketch and one refinement step.
        {"name": "pne_65536x1024", "op": "solve", "method": "pne", "m": 65536, "n": 1024, "kappa": 1e2, "rho": 1e-8,
         "kind": "sparse", "s": 4096, "prec": "bf16", "refine": 1},
        # The largest single problem, precision from the estimate on a sketch.
        {"name": "pne_262144x4096", "op": "solve", "method": "pne", "m": 262144, "n": 4096, "kappa": 1e4, "rho": 1e-6,
         "kind": "gaussian", "s": 8192, "prec": "auto_sketch", "refine": 0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes log-uniform over the listed ranges (odd ones
    among them), options as they are used together."""
    op = rng.choice(["solve", "solve", "solve", "trsm_gram", "trsm_gram", "sketch", "sketch", "qr", "factor",
                     "batched", "mlp"])
    if op == "solve":
        m = _log_int(rng, 1000, 131072)
        n = _log_int(rng, 48, min(m // 4, 2000))
        prec = rng.choice(["bf16", "fp32", "fp32", "fp64", "auto_sketch"])
        kind = rng.choice(["gaussian", "sparse", "srft"])
        return {"op": op, "method": rng.choice(["pne", "pne", "hpne"]), "m": m, "n": n,
                "kappa": 1e2 if prec == "bf16" else 10.0 ** rng.uniform(1, 5), "rho": 10.0 ** rng.uniform(-12, -6),
                "kind": kind, "s": n * {"gaussian": 2, "sparse": 4, "srft": 3}[kind], "prec": prec,
                "refine": rng.choice([0, 1])}
    if op == "trsm_gram":
        m = _log_int(rng, 2000, 262144)
        return {"op": op, "m": m, "n": _log_int(rng, 32, min(m // 4, 2000)), "hpne": rng.random() < 0.4}
    if op == "sketch":
        m = _log_int(rng, 2000, 131072)
        n = _log_int(rng, 32, min(m // 4, 2000))
        kind, prec = rng.choice([("gaussian", "fp8"), ("gaussian", "bf16"), ("gaussian", "fp64"), ("gaussian", "fp64"),
                                 ("sparse", "bf16"), ("sparse", "fp32"), ("sparse", "fp64"), ("srft", "fp32"),
                                 ("srft", "fp64")])
        return {"op": op, "m": m, "n": n, "s": n * {"gaussian": 2, "sparse": 4, "srft": 3}[kind], "kind": kind,
                "prec": prec}
    if op == "qr":
        n = _log_int(rng, 32, 2000)
        return {"op": op, "s": n * rng.choice([2, 3, 4]), "n": n}
    if op == "factor":
        hpne = rng.random() < 0.5
        return {"op": op, "n": _log_int(rng, 32, 2000 if hpne else 4096), "hpne": hpne}
    if op == "batched":
        return {"op": op, "count": rng.randint(8, 64), "m_max": _log_int(rng, 4000, 40000),
                "n_max": _log_int(rng, 64, 512), "shape_seed": rng.randint(0, 1 << 20)}
    return {"op": "mlp", "batch": _log_int(rng, 64, 4096)}


# ---- inputs ------------------------------------------------------------------
def _gen(seed, stream):
    return torch.Generator(device=DEV).manual_seed((int(seed) * 16 + stream) % (1 << 62))


def _x_star(n, seed):
    return torch.randn(n, generator=_gen(seed, 0), dtype=torch.float64, device=DEV)


def _tall(m, n, kappa, seed):
    """A (m x n FP64, column-major) and V, sigma with A close to U diag(sigma) V^T."""
    g = _gen(seed, 1)
    V = torch.linalg.qr(torch.randn((n, n), generator=g, dtype=torch.float32, device=DEV))[0]
    sigma = torch.logspace(0.0, -math.log10(kappa), n, dtype=torch.float32, device=DEV)
    At = torch.empty((n, m), dtype=torch.float64, device=DEV)
    At.copy_((V * sigma) @ (torch.randn((n, m), generator=g, dtype=torch.float32, device=DEV) / math.sqrt(m)))
    for j in range(0, n, 512):  # all 53 bits of the entries in use
        part = At[j:j + 512]
        part.mul_(torch.rand(part.shape, generator=g, dtype=torch.float64, device=DEV).mul_(2.0 ** -26).add_(1.0))
    return At.t(), V.double(), sigma.double()


def _rhs(A, V, sigma, rho, seed):
    """b = A x_* + r, r orthogonal to range(A): the residual of a Gaussian
    vector by conjugate gradients on A V diag(1/sigma), which is well
    conditioned (convergence factor about sqrt(n / m) a step)."""
    m, n = A.shape
    x = _x_star(n, seed)

    def mul(z):
        return A @ (V @ (z / sigma))

    def mul_t(r):
        return (V.t() @ (A.t() @ r)) / sigma

    r = torch.randn(m, generator=_gen(seed, 2), dtype=torch.float64, device=DEV)
    for _ in range(2):  # the second pass takes out the first one's rounding
        s = mul_t(r)
        p, gamma = s.clone(), s @ s
        for _ in range(int(20.0 / math.log(math.sqrt(m / n))) + 3):
            q = mul(p)
            alpha = gamma / (q @ q).clamp_min(1e-300)
            r = r - alpha * q
            s = mul_t(r)
            new = s @ s
            p = s + (new / gamma.clamp_min(1e-300)) * p
            gamma = new
    r = r * (rho * torch.linalg.norm(x) / torch.linalg.norm(r))
    return A @ x + r


def _opts(case, n, seed):
    return lsq.make_opts(kind=_KIND[case["kind"]], s=case["s"], n=n, seed=seed & 0xFFFFFFFF,
                         sketch_prec=_PREC[case["prec"]],
                         qr_prec=lsq.FP64 if case["prec"] == "fp64" else lsq.FP32,
                         refine_steps=case.get("refine", 0))


def _triangular(n, seed, stream, kappa=1e3):
    """An upper triangular R (column-major FP64) like a preconditioner's: the
    factor of a QR with singular values from 1 to 1/kappa."""
    g = _gen(seed, stream)
    V = torch.linalg.qr(torch.randn((n, n), generator=g, dtype=torch.float32, device=DEV))[0]
    sigma = torch.logspace(0.0, -math.log10(kappa), n, dtype=torch.float32, device=DEV)
    R = torch.linalg.qr(sigma[:, None] * V.t())[1]
    R = R * torch.sign(torch.diagonal(R))[:, None]
    return lsq.colmajor(torch.triu(R).double())


def _batch_shapes(case):
    rng = np.random.default_rng(case["shape_seed"])
    out = []
    for _ in range(case["count"]):
        n = int(rng.integers(32, case["n_max"] + 1))
        m = int(rng.integers(max(2000, 4 * n), max(case["m_max"], 4 * n) + 1))
        kappa, rho = 10.0 ** rng.uniform(2, 6), 10.0 ** rng.uniform(-12, -8)
        kind, mult = (lsq.GAUSSIAN, lsq.SPARSE_SIGN)[int(rng.integers(0, 2))], int(rng.integers(1, 3)) * 2
        out.append((m, n, kappa, rho, kind, mult * n))
    return out


def _factor_inputs(case, seed):
    n = case["n"]
    g = _gen(seed, 3)
    X = torch.randn((4 * n, n), generator=g, dtype=torch.float64, device=DEV) if n <= 512 else \
        torch.randn((4 * n, n), generator=g, dtype=torch.float32, device=DEV)
    G = (X.t() @ X).double() / (4 * n)  # condition number about 9, as A_p^T A_p
    c = torch.randn(n, generator=g, dtype=torch.float64, device=DEV)
    R = _triangular(n, seed, 4)
    if case["hpne"]:
        return lsq.colmajor(G.float() @ R.float()), c, None
    G = (G + G.t()) * 0.5
    return lsq.colmajor(G), c, R


def _mlp_inputs(case, seed):
    g = _gen(seed, 5)
    d = lsq.N_FEATURES
    parts = []
    for out, inp in [(64, d), (64, 64), (64, 64), (4, 64)]:
        parts += [torch.randn(out * inp, generator=g, device=DEV) * math.sqrt(2.0 / inp),
                  torch.randn(out, generator=g, device=DEV) * 0.1]
    X = torch.randn((case["batch"], d), generator=g, device=DEV)
    y = torch.randint(0, 4, (case["batch"],), generator=g, device=DEV).to(torch.int32)
    return torch.cat(parts).float(), X, y


def prepare(case, seed):
    op = case["op"]
    if op == "solve":
        A, V, sigma = _tall(case["m"], case["n"], case["kappa"], seed)
        return {"op": op, "A": A, "b": _rhs(A, V, sigma, case["rho"], seed), "opts": _opts(case, case["n"], seed),
                "method": case["method"]}
    if op == "trsm_gram":
        m, n = case["m"], case["n"]
        R = _triangular(n, seed, 4)
        g = _gen(seed, 1)
        At = torch.empty((n, m), dtype=torch.float64, device=DEV)
        At.copy_((R.float().t() @ torch.randn((n, m), generator=g, dtype=torch.float32, device=DEV)) / math.sqrt(m))
        return {"op": op, "A": At.t(), "R": R, "hpne": case["hpne"],
                "b": torch.randn(m, generator=g, dtype=torch.float64, device=DEV)}
    if op == "sketch":
        A = _tall(case["m"], case["n"], 1e4, seed)[0]
        return {"op": op, "A": A, "opts": _opts(case, case["n"], seed)}
    if op == "qr":
        return {"op": op, "As": _tall(case["s"], case["n"], 1e4, seed)[0]}
    if op == "factor":
        G, c, R = _factor_inputs(case, seed)
        return {"op": op, "G": G, "c": c, "R": R, "hpne": case["hpne"]}
    if op == "batched":
        shapes = _batch_shapes(case)
        As, bs, opts = [], [], []
        for i, (m, n, kappa, rho, kind, s) in enumerate(shapes):
            A, V, sigma = _tall(m, n, kappa, seed * 64 + i)
            As.append(A)
            bs.append(_rhs(A, V, sigma, rho, seed * 64 + i))
            opts.append(lsq.make_opts(kind=kind, s=s, n=n, seed=i + 1, sketch_prec=lsq.AUTO_SKETCH, refine_steps=1))
        x = torch.empty(sum(p[1] for p in shapes), dtype=torch.float64, device=DEV)
        info = torch.zeros(len(shapes), dtype=torch.int32, device=DEV)
        xs = list(torch.split(x, [p[1] for p in shapes]))
        desc = lsq.batch_descriptors(As, bs, xs, list(torch.split(info, 1)), opts)
        return {"op": op, "As": As, "bs": bs, "x": x, "info": info, "desc": desc,
                "ws": lsq.batched_workspace(desc)}
    p, X, y = _mlp_inputs(case, seed)
    return {"op": op, "p": p, "X": X, "y": y, "m1": torch.zeros_like(p), "m2": torch.zeros_like(p), "step": 0}


def run(state):
    op = state["op"]
    if op == "solve":
        return lsq.solve(state["A"], state["b"], method=state["method"], opts=state["opts"])
    if op == "trsm_gram":
        return lsq.trsm_gram(state["A"], state["R"], state["b"], hpne=state["hpne"])
    if op == "sketch":
        return lsq.sketch(state["A"], state["opts"])
    if op == "qr":
        return lsq.precond_qr(state["As"], qr_prec=lsq.FP64)
    if op == "factor":
        x, F, piv, info = lsq.factor_solve(state["G"], state["c"], state["R"], hpne=state["hpne"])
        return (x, F, piv, info) if state["hpne"] else (x, torch.tril(F), None, info)  # L is the lower triangle
    if op == "batched":
        lsq.solve_batched(state["desc"], state["ws"])
        return state["x"], state["info"]
    state["step"] += 1
    grad, loss = lsq.mlp_backward(state["p"], state["X"], state["y"])
    lsq.mlp_adam(state["p"], grad, state["m1"], state["m2"], state["step"], lr=2e-3)
    return grad, loss, state["p"], state["m1"], state["m2"]


def _solve_work(m, n, s, kind, hpne):
    sketch = 2.0 * s * n * m if kind == "gaussian" else 8.0 * 2.0 * n * m
    return {"bytes": 8.0 * (m * n + m + n),
            "flops": sketch + 2.0 * s * n * n + m * n * n * (3.0 if hpne else 2.0) + n ** 3 * (2 / 3 if hpne else 1 / 3)}


def work(case):
    op = case["op"]
    if op == "solve":
        return _solve_work(case["m"], case["n"], case["s"], case["kind"], case["method"] == "hpne")
    if op == "trsm_gram":
        m, n = case["m"], case["n"]
        return {"bytes": 8.0 * (2 * m * n + m + 1.5 * n * n + n), "flops": m * n * n * (3.0 if case["hpne"] else 2.0)}
    if op == "sketch":
        m, n, s = case["m"], case["n"], case["s"]
        flops = {"gaussian": 2.0 * s * n * m, "sparse": 16.0 * n * m,
                 "srft": n * 2.0 ** math.ceil(math.log2(m)) * math.ceil(math.log2(m))}[case["kind"]]
        return {"bytes": 8.0 * m * n + (8.0 if case["prec"] == "fp64" else 4.0) * s * n + 4.0 * n, "flops": flops}
    if op == "qr":
        s, n = case["s"], case["n"]
        return {"bytes": 8.0 * (s * n + n * n), "flops": 2.0 * s * n * n - 2.0 / 3.0 * n ** 3}
    if op == "factor":
        n = case["n"]
        return {"bytes": 8.0 * (2.0 * n * n + 2 * n), "flops": n ** 3 * (2 / 3 if case["hpne"] else 1 / 3)}
    if op == "batched":
        each = [_solve_work(m, n, s, "gaussian" if kind == lsq.GAUSSIAN else "sparse", False)
                for m, n, _, _, kind, s in _batch_shapes(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    b, d = case["batch"], lsq.N_FEATURES
    params = 64 * d + 64 + 2 * (64 * 64 + 64) + 4 * 64 + 4
    return {"bytes": 4.0 * (b * (d + 1) + 7 * params), "flops": 6.0 * b * params}


# ---- exact values ------------------------------------------------------------
def _mlp_exact(case, seed):
    p32, X32, y = _mlp_inputs(case, seed)
    p = p32.double().requires_grad_(True)
    h, at, d = X32.double(), 0, lsq.N_FEATURES
    for k, (out, inp) in enumerate([(64, d), (64, 64), (64, 64), (4, 64)]):
        W, bias = p[at:at + out * inp].view(out, inp), p[at + out * inp:at + out * inp + out]
        at += out * inp + out
        h = h @ W.t() + bias
        if k < 3:
            h = torch.relu(h)
    loss = torch.nn.functional.cross_entropy(h, y.long())
    loss.backward()
    g = p.grad
    m1, m2 = 0.1 * g, 0.001 * g * g
    new = p.detach() - 2e-3 * g / (g.abs() + 1e-8)
    return g, loss.detach().reshape(1), new, m1, m2


def exact(case, seed):
    op = case["op"]
    if op == "solve":  # the solution the right-hand side was made from
        return _x_star(case["n"], seed), None
    if op == "batched":
        return torch.cat([_x_star(p[1], seed * 64 + i) for i, p in enumerate(_batch_shapes(case))]), None
    if op == "sketch":  # needs the library's random operator
        return None
    st = prepare(case, seed)
    if op == "mlp":
        return _mlp_exact(case, seed)
    if op == "trsm_gram":
        A, R, b = st["A"], st["R"], st["b"]
        Ap = torch.linalg.solve_triangular(R, A, upper=True, left=False)
        return Ap, Ap.t() @ (A if st["hpne"] else Ap), Ap.t() @ b
    if op == "qr":
        R = torch.linalg.qr(st["As"], mode="r")[1]
        return R * torch.sign(torch.diagonal(R))[:, None], None
    G, c, R = st["G"], st["c"], st["R"]
    if st["hpne"]:
        LU, piv = torch.linalg.lu_factor(G)
        return torch.linalg.lu_solve(LU, piv, c[:, None])[:, 0], LU, None, None
    L = torch.linalg.cholesky(G)
    y = torch.cholesky_solve(c[:, None], L)
    return torch.linalg.solve_triangular(R, y, upper=True)[:, 0], L, None, None
