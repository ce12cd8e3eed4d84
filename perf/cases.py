"""The work a user of this library has it do, as measurable cases.

A case is one call of a public entry point (paper_2405_09233_gb300.Context) on tensors that already
live on the GPU, in the library's layout: a tensor X in R^{n1 x n2 x p} is a contiguous (p, n2, n1)
torch tensor.  Kinds:

  apply    Y = M(X) = A*X - X*B in FP64: sylv_apply (engine "dfma") or sylv_apply_ozaki ("ozaki")
  lowp     Y = M(X) in FP32 storage: sylv_apply_lowp with its four precisions
  tstar    C = A*B, the T-product itself
  solve    restarted tGMRES / tFOM on M(X) = C from X0 = 0 (single instance)
  batched  many uneven instances in one batched_solve
  tbas     Tubal Block Arnoldi on a sparse operator
  direct   t-Bartels-Stewart on a small dense equation

Inputs are the families of paper_2405_09233_gb300.inputs (dense, sparse, batched), drawn on the GPU.
A program keeps one Context and, per equation, the prepared operator; so do the states here.
"""
import math

import numpy as np
import torch

from paper_2405_09233_gb300 import Context

DEV = "cuda"
_ctx = None


def _context():
    """The process's one library context."""
    global _ctx
    if _ctx is None:
        _ctx = Context(torch.cuda.current_device())
    return _ctx


# ---------------------------------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------------------------------
def listed():
    return [
        # The smallest call: one operator application of the 24 x 24 x 4 example, all launch latency.
        {"name": "apply_fp64_tiny", "kind": "apply", "n": 24, "s": 24, "p": 4, "engine": "dfma"},
        # An ordinary FP64 application at sizes that no tile divides and a tube length that is no power of two.
        {"name": "apply_fp64_ragged", "kind": "apply", "n": 500, "s": 130, "p": 12, "engine": "dfma"},
        # One residual of the n = s = 1024, p = 16 workload on the emulated-FP64 engine.
        {"name": "apply_emulated", "kind": "apply", "n": 1024, "s": 1024, "p": 16, "engine": "ozaki"},
        # The inner operator of the largest mixed-precision workload (n = 4096, s = 256, p = 32).
        {"name": "apply_bf16_large", "kind": "lowp", "n": 4096, "s": 256, "p": 32, "precision": "mixed_bf16"},
        # Split TF32 at ragged sizes: the FP32-accurate inner operator on the tensor cores.
        {"name": "apply_tf32x3", "kind": "lowp", "n": 1000, "s": 300, "p": 8, "precision": "mixed_tf32x3"},
        # FP32 on the CUDA cores, the inner operator of a TS_MIXED_FP32 solve.
        {"name": "apply_fp32", "kind": "lowp", "n": 512, "s": 128, "p": 16, "precision": "mixed_fp32"},
        # A rectangular T-product with an odd tube length.
        {"name": "tstar_odd", "kind": "tstar", "n1": 300, "n2": 200, "m": 100, "p": 7},
        # A whole small FP64 solve (24 x 24 x 4): a handful of short dependent kernels per step.
        {"name": "solve_fp64_small", "kind": "solve", "n": 24, "s": 24, "p": 4, "g": 0.1, "method": "tgmres",
         "precision": "fp64", "engine": "dfma", "spectral": False, "restart": 20, "steps": 18},
        # The fast whole solve at n = s = 1024, p = 16: BF16 inner solves, emulated-FP64 residuals.
        {"name": "solve_mixed_1024", "kind": "solve", "n": 1024, "s": 1024, "p": 16, "g": 0.1, "method": "tgmres",
         "precision": "mixed_bf16", "engine": "ozaki", "spectral": False, "restart": 30, "steps": 20},
        # Many uneven equations at once (n in [64, 1024], s in [16, 128], p in {4, 8, 16}).
        {"name": "batched_mixed", "kind": "batched", "count": 64, "n_lo": 64, "n_hi": 1024, "s_lo": 16, "s_hi": 128,
         "shapes": 7, "precision": "mixed_bf16", "engine": "ozaki", "restart": 20, "steps": 20},
        # TBAS(10) on the sparse 128 x 128-grid operator with block width 32.
        {"name": "tbas_sparse", "kind": "tbas", "grid": 128, "s": 32, "p": 8, "precision": "fp64", "restart": 10,
         "steps": 20},
        # The direct solver on a small dense equation.
        {"name": "direct_64", "kind": "direct", "n": 64, "s": 64, "p": 8},
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "lowp", "lowp", "tstar", "solve", "solve", "batched", "tbas", "direct"])
    p = rng.choice([1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 12, 15, 16, 16, 20, 24, 31, 32])
    if kind == "apply":
        return {"kind": kind, "n": _log(rng, 8, 1024), "s": _log(rng, 4, 512), "p": p,
                "engine": rng.choice(["dfma", "ozaki"])}
    if kind == "lowp":
        return {"kind": kind, "n": _log(rng, 24, 2048), "s": _log(rng, 8, 512), "p": p,
                "precision": rng.choice(["mixed_bf16", "mixed_tf32x3", "mixed_tf32", "mixed_fp32"])}
    if kind == "tstar":
        return {"kind": kind, "n1": _log(rng, 4, 600), "n2": _log(rng, 4, 600), "m": _log(rng, 2, 400), "p": p}
    if kind == "solve":
        precision = rng.choice(["fp64", "fp64", "mixed_bf16", "mixed_tf32x3", "mixed_fp32"])
        engine = rng.choice(["dfma", "ozaki"])
        method = rng.choice(["tgmres", "tgmres", "tfom"]) if precision == "fp64" else "tgmres"
        spectral = precision == "fp64" and rng.random() < 0.2
        return {"kind": kind, "n": _log(rng, 12, 640), "s": _log(rng, 8, 320), "p": min(p, 16), "g": 0.1,
                "method": method, "precision": precision, "engine": engine, "spectral": spectral,
                "restart": rng.choice([10, 20, 30]), "steps": 20}
    if kind == "batched":
        precision, engine = rng.choice([("mixed_bf16", "ozaki"), ("mixed_tf32x3", "ozaki"), ("fp64", "ozaki"),
                                        ("mixed_fp32", "dfma"), ("fp64", "dfma")])
        return {"kind": kind, "count": _log(rng, 3, 64), "n_lo": 16, "n_hi": _log(rng, 64, 768), "s_lo": 8, "s_hi": 96,
                "shapes": rng.randrange(1 << 20), "precision": precision, "engine": engine, "restart": 20, "steps": 20}
    if kind == "tbas":
        grid, s = _log(rng, 16, 128), _log(rng, 2, 40)
        return {"kind": kind, "grid": grid, "s": s, "p": rng.choice([1, 2, 3, 4, 6, 8]),
                "precision": rng.choice(["fp64", "fp64", "mixed_fp32"]),
                "restart": max(2, min(10, grid * grid // (2 * s))), "steps": 20}
    return {"kind": kind, "n": _log(rng, 8, 128), "s": _log(rng, 4, 96), "p": rng.choice([1, 2, 3, 4, 5, 8])}


# ---------------------------------------------------------------------------------------------------
# Plain torch in 64 bits: the T-product through the DFT along mode 3, on (p, n2, n1) storage
# ---------------------------------------------------------------------------------------------------
def _product(Ast, Xst):
    """Storage of A*X from storages (p, n2, n1) of A and (p, m, n2) of X."""
    p = Ast.shape[0]
    Ah, Xh = torch.fft.rfft(Ast, dim=0), torch.fft.rfft(Xst, dim=0)
    return torch.fft.irfft(torch.matmul(Xh, Ah), n=p, dim=0)


def _operator(Ast, Bst, Xst):
    """Storage of M(X) = A*X - X*B."""
    p = Ast.shape[0]
    Ah, Bh, Xh = (torch.fft.rfft(t, dim=0) for t in (Ast, Bst, Xst))
    return torch.fft.irfft(torch.matmul(Xh, Ah) - torch.matmul(Bh, Xh), n=p, dim=0).contiguous()


# ---------------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _randn(shape, gen, scale=1.0):
    return torch.randn(shape, dtype=torch.float64, device=DEV, generator=gen).mul_(scale)


def _uniform(shape, gen):
    return torch.rand(shape, dtype=torch.float64, device=DEV, generator=gen).mul_(2.0).sub_(1.0)


def _add_tridiag(M, sign):
    """M += sign * tridiag(-1, 4, -1), in place."""
    M.diagonal().add_(4.0 * sign)
    if M.shape[0] > 1:
        M.diagonal(1).sub_(1.0 * sign)
        M.diagonal(-1).sub_(1.0 * sign)


def _dense(n, s, p, g, gen):
    """The dense family: A, B, X* (storage)."""
    A = _randn((p, n, n), gen, g / math.sqrt(n))
    _add_tridiag(A[0], 1.0)
    B = _randn((p, s, s), gen, g / math.sqrt(s))
    _add_tridiag(B[0], -1.0)
    return A, B, _uniform((p, s, n), gen)


def _batch_shapes(case):
    r = np.random.default_rng(case["shapes"])
    out = []
    for _ in range(case["count"]):
        n = int(round(math.exp(r.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))))
        out.append((n, int(r.integers(case["s_lo"], case["s_hi"] + 1)), int(r.choice([4, 8, 16]))))
    return out


def _sparse(case, seed):
    """The sparse family: p CSR slices (5-point Laplacian; 4 off-diagonal entries per row), B, X*."""
    grid, s, p = case["grid"], case["s"], case["p"]
    n = grid * grid
    r = np.random.default_rng(seed)
    i = np.arange(n)
    x, y = i % grid, i // grid
    cols = np.stack([i - grid, i - 1, i, i + 1, i + grid], 1)
    keep = np.stack([y > 0, x > 0, i >= 0, x < grid - 1, y < grid - 1], 1)
    vals = np.broadcast_to(np.array([-1.0, -1.0, 4.0, -1.0, -1.0]), cols.shape)
    slices = [(np.concatenate([[0], np.cumsum(keep.sum(1))]), cols[keep], vals[keep])]
    for _ in range(1, p):
        # four distinct offsets 1 .. n-1 per row, taken cyclically: distinct off-diagonal columns
        first = r.integers(1, n // 4, size=(n, 1))
        gaps = r.integers(1, n // 4, size=(n, 3))
        off = np.concatenate([first, first + np.cumsum(gaps, 1)], 1)
        c = np.sort((i[:, None] + off) % n, 1)
        slices.append((np.arange(0, 4 * n + 1, 4), c.reshape(-1), 0.05 * r.standard_normal(4 * n)))
    gen = _gen(seed)
    B = _randn((p, s, s), gen, 0.1 / math.sqrt(s))
    B[0].diagonal().sub_(4.0)
    return n, slices, B, _uniform((p, s, n), gen)


def _sparse_operator(n, slices, B, X):
    """Storage of M(X) with sparse A, from the definition: Y_t = sum_k A_((t-k) mod p) X_k - (X*B)_t."""
    p = X.shape[0]
    Y = torch.zeros_like(X)
    Xi = X.transpose(1, 2).contiguous()                       # (p, n, s)
    for t, (ptr, col, val) in enumerate(slices):
        A = torch.sparse_csr_tensor(torch.from_numpy(ptr.astype(np.int64)), torch.from_numpy(col.astype(np.int64)),
                                    torch.from_numpy(np.ascontiguousarray(val)), size=(n, n),
                                    check_invariants=False).to(DEV)
        for k in range(p):
            Y[(t + k) % p] += (A @ Xi[k]).transpose(0, 1)
    return (Y - _product(X, B)).contiguous()


def _problem(case, seed):
    """(A, B, X*) of a dense kind; of `lowp`, X* in FP32."""
    A, B, X = _dense(case["n"], case["s"], case["p"], case.get("g", 0.1), _gen(seed))
    return A, B, X.float() if case["kind"] == "lowp" else X


def prepare(case, seed):
    ctx, kind = _context(), case["kind"]
    st = {"case": case, "ctx": ctx}
    if kind in ("apply", "lowp"):
        A, B, X = _problem(case, seed)
        st.update(op=ctx.op_create_dense(A, B), X=X, Y=torch.empty_like(X))
    elif kind == "tstar":
        gen = _gen(seed)
        st.update(A=_randn((case["p"], case["n2"], case["n1"]), gen), B=_randn((case["p"], case["m"], case["n2"]), gen),
                  Y=torch.empty((case["p"], case["m"], case["n1"]), dtype=torch.float64, device=DEV))
    elif kind == "solve":
        A, B, X = _problem(case, seed)
        st.update(op=ctx.op_create_dense(A, B), C=_operator(A, B, X), X=torch.empty_like(X))
    elif kind == "batched":
        gen, ops, Cs, Xs = _gen(seed), [], [], []
        for n, s, p in _batch_shapes(case):
            A, B, X = _dense(n, s, p, 0.1, gen)
            ops.append(ctx.op_create_dense(A, B))
            Cs.append(_operator(A, B, X))
            Xs.append(torch.empty_like(X))
        st.update(ops=ops, Cs=Cs, Xs=Xs)
    elif kind == "tbas":
        n, slices, B, X = _sparse(case, seed)
        base = np.cumsum([0] + [len(c) for _, c, _ in slices[:-1]])
        op = ctx.op_create_csr(n, case["p"], np.concatenate([ptr + b for (ptr, _, _), b in zip(slices, base)]),
                               np.concatenate([c for _, c, _ in slices]), np.concatenate([v for _, _, v in slices]), B)
        st.update(op=op, C=_sparse_operator(n, slices, B, X), X=torch.empty_like(X))
    else:
        A, B, X = _problem(case, seed)
        st.update(A=A, B=B, C=_operator(A, B, X), X=torch.empty_like(X))
    return st


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind == "apply":
        if case["engine"] == "ozaki":
            return ctx.sylv_apply_ozaki(state["op"], state["X"], state["Y"])
        return ctx.sylv_apply(state["op"], state["X"], state["Y"])
    if kind == "lowp":
        return ctx.sylv_apply_lowp(state["op"], state["X"], case["precision"], state["Y"])
    if kind == "tstar":
        return ctx.tstar(state["A"], state["B"], state["Y"])
    if kind == "solve":
        X = state["X"].zero_()
        if case["method"] == "tfom":
            ctx.tfom_solve(state["op"], state["C"], X, restart=case["restart"], engine=case["engine"],
                           spectral=case["spectral"])
        else:
            ctx.tgmres_solve(state["op"], state["C"], X, restart=case["restart"], precision=case["precision"],
                             engine=case["engine"], spectral=case["spectral"])
        return X
    if kind == "batched":
        Xs = state["Xs"]
        for X in Xs:
            X.zero_()
        ctx.batched_solve(state["ops"], state["Cs"], Xs, restart=case["restart"], precision=case["precision"],
                          engine=case["engine"])
        return Xs
    if kind == "tbas":
        X = state["X"].zero_()
        ctx.tba_solve(state["op"], state["C"], X, restart=case["restart"], precision=case["precision"])
        return X
    return ctx.t_bartels_stewart(state["A"], state["B"], state["C"], state["X"])


# ---------------------------------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------------------------------
def _apply_work(n, s, p, size, x_size):
    """One application: the operator's spectrum at `size` bytes a real read once, X read and Y written;
    8 operations per complex and 2 per real multiply-add of the slice products."""
    K = p // 2 + 1
    real = 2 if p % 2 == 0 and p > 1 else 1
    reals = 2 * (K - real) + real
    return {"bytes": size * reals * (n * n + s * s) + 2 * x_size * n * s * p,
            "flops": n * s * (n + s) * (8 * (K - real) + 2 * real)}


def work(case):
    kind = case["kind"]
    if kind == "apply":
        return _apply_work(case["n"], case["s"], case["p"], 8, 8)
    if kind == "lowp":
        return _apply_work(case["n"], case["s"], case["p"], 2 if case["precision"] == "mixed_bf16" else 4, 4)
    if kind == "tstar":
        n1, n2, m, p = case["n1"], case["n2"], case["m"], case["p"]
        K = p // 2 + 1
        real = 2 if p % 2 == 0 and p > 1 else 1
        return {"bytes": 8 * p * (n1 * n2 + n2 * m + n1 * m), "flops": n1 * n2 * m * (8 * (K - real) + 2 * real)}
    if kind in ("solve", "batched"):
        shapes = _batch_shapes(case) if kind == "batched" else [(case["n"], case["s"], case["p"])]
        w = {"bytes": 0, "flops": 0}
        for n, s, p in shapes:   # operator and C read, X written; about `steps` applications to 1e-10
            one = _apply_work(n, s, p, 8, 8)
            w["bytes"] += one["bytes"]
            w["flops"] += case["steps"] * one["flops"]
        return w
    if kind == "tbas":
        # `steps` block steps: the sparse product, and the block Gram-Schmidt over half the restart on average
        n, s, p = case["grid"] ** 2, case["s"], case["p"]
        K = p // 2 + 1
        nnz = n * (5 + 4 * (p - 1))
        gram = case["restart"] / 2 + 2
        return {"bytes": 12 * nnz + 8 * p * s * (s + 2 * n),
                "flops": case["steps"] * K * 8 * (nnz * s + 2 * gram * n * s * s)}
    n, s, p = case["n"], case["s"], case["p"]
    K = p // 2 + 1
    # complex Schur forms of the s x s slices, s shifted factorisations of the n x n slices, the column sweep
    return {"bytes": 8 * p * (n * n + s * s + 2 * n * s),
            "flops": K * (8 * 25 * s ** 3 // 3 + s * (8 * n ** 3 // 3 + 8 * n * n) + 8 * n * s * s)}


def exact(case, seed):
    """The same outputs by plain torch in 64 bits; for solves, the manufactured solution."""
    kind = case["kind"]
    if kind in ("apply", "lowp"):
        A, B, X = _problem(case, seed)
        return _operator(A, B, X.double())
    if kind == "tstar":
        gen = _gen(seed)
        A = _randn((case["p"], case["n2"], case["n1"]), gen)
        return _product(A, _randn((case["p"], case["m"], case["n2"]), gen))
    if kind == "batched":
        gen = _gen(seed)
        return [_dense(n, s, p, 0.1, gen)[2] for n, s, p in _batch_shapes(case)]
    if kind == "tbas":
        return _sparse(case, seed)[3]
    return _problem(case, seed)[2]
