"""TBAS over block widths that change the shape of its Gram, row-product and Cholesky kernels (column groups
of 4, columns per thread, row groups), with few rows, odd p and both precisions."""
import numpy as np
import pytest

from oracle import krylov as kr
from paper_2405_09233_gb300 import Context, inputs
from tests.gpu_helpers import from_dev, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = Context(0)
    yield c
    c.workspace_check()
    c.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed_fp32"])
@pytest.mark.parametrize("dims", [(17, 1, 1), (40, 2, 2), (41, 3, 5), (70, 5, 4), (90, 7, 3), (96, 8, 2), (130, 9, 2),
                                  (150, 13, 4), (200, 17, 2), (250, 25, 3), (300, 31, 2), (300, 33, 2), (330, 40, 1),
                                  (400, 57, 2), (400, 64, 2)], ids=lambda d: "n%d_s%d_p%d" % d)
def test_recovers_the_solution(ctx, dims, precision):
    """Solved to a true relative residual of 1e-10; M's inverse is of norm below 1 on this family (spectra of
    A and -B in [1, 7]) and ||C|| below 10 ||X*||, so X is within 1e-9 of X* relative to its norm."""
    import torch
    n, s, p = dims
    pr = inputs.dense_problem(n, s, p, seed=n + s)
    C = kr.sylv_apply(pr.A, pr.B, pr.Xstar)
    op = ctx.op_create_dense(to_dev(pr.A), to_dev(pr.B))
    X = torch.zeros((p, s, n), dtype=torch.float64, device="cuda")
    res = ctx.tba_solve(op, to_dev(C), X, restart=max(2, min(8, n // (2 * s))), tol=1e-10, precision=precision)
    assert res.status == 0 and res.relres <= 1e-10, res
    assert np.linalg.norm(from_dev(X) - pr.Xstar) <= 1e-9 * np.linalg.norm(pr.Xstar)
