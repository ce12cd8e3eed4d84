"""FP32 Grams of many rows: how long their FP32 chains are.

A = 4 I, B = -4 I and C with orthogonal columns of +-1 in one frontal slice: V_1 = C / sqrt(n) entry by entry, so the
Gram <V_1, A V_1> adds up n equal FP32 products per diagonal entry, whose rounding errors do not average out.  One
block step solves the equation up to half the relative error of that Gram."""
import numpy as np
import pytest

from paper_2405_09233_gb300 import Context

pytestmark = pytest.mark.gpu


def chain_error(v, terms):
    """Relative error of `terms` products v v added up in FP32."""
    p, s = float(v) ** 2, 0.0
    for _ in range(terms):
        s = float(np.float32(s + p))
    return abs(s / (terms * p) - 1.0)


@pytest.mark.parametrize("s", [48, 64])
def test_rows_per_fp32_sum(s):
    import torch
    n, p = 12544, 8
    # 60 blocks of 210 rows per slice; the 13 blocks of 965 rows a third of a complex slice's share would be err by 1.3e-5
    bound = chain_error(np.float32(1.0 / np.sqrt(n)), 210)
    assert bound < 5e-7 < 1e-5 < chain_error(np.float32(1.0 / np.sqrt(n)), 965)
    ctx = Context(0)
    B = torch.zeros((p, s, s), dtype=torch.float64, device="cuda")
    B[0].diagonal().fill_(-4.0)
    rows = [np.arange(n + 1)] + [np.full(n + 1, n)] * (p - 1)   # A^(1) = 4 I, the other slices empty
    op = ctx.op_create_csr(n, p, np.concatenate(rows), np.arange(n), np.full(n, 4.0), B)
    i, j = np.arange(n)[None, :] % 64, np.arange(s)[:, None]
    walsh = 1.0 - 2.0 * (np.array([bin(q).count("1") for q in range(64)])[i & j] % 2)
    C = torch.zeros((p, s, n), dtype=torch.float64, device="cuda")
    C[0] = torch.from_numpy(walsh).cuda()
    X = torch.zeros_like(C)
    res = ctx.tba_solve(op, C, X, restart=1, tol=1e-12, max_restarts=1, precision="mixed_fp32")
    # half of the Gram's error and of the squared norms V_1 was scaled by, and a few FP32 roundings of V_1
    assert res.info.relres_true <= 0.5 * bound + 8 * 2.0 ** -24, res.info.relres_true
    op.close()
    ctx.workspace_check()
    ctx.close()
