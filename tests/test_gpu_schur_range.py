"""Schur factors of B whose trailing blocks lie so far below its largest entry that their squares leave the FP64
range (B = lower shift + tiny diagonal: eigenvalues that tiny, and Wilkinson shifts formed from them)."""
import numpy as np
import pytest

from oracle import krylov as kr
from paper_2405_09233_gb300 import Context, inputs
from .gpu_helpers import from_dev, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = Context(0)
    yield c
    c.workspace_check()
    c.close()


def tiny_diagonal(s, tiny, coupled):
    """0.5 below the diagonal, multiples of `tiny` on it; `coupled`: `tiny` above it too."""
    B = np.zeros((s, s, 1))
    B[:, :, 0] = 0.5 * np.eye(s, k=-1) + tiny * np.diag(np.arange(s, 0.0, -1.0) - 1.0)
    if coupled:
        B[:, :, 0] += tiny * np.eye(s, k=1)
    return B


# |B| < 1 and the spectrum of A in [2, 6]: the equation's condition number is below about 20 and a backward stable
# solver's relative error below ~ (n + s) u 20 times a modest constant.
RTOL = 1e-12


@pytest.mark.parametrize("coupled", [False, True])
@pytest.mark.parametrize("s", [2, 3, 7])
@pytest.mark.parametrize("tiny", [1e-150, 1e-155, 1e-160, 1e-200, 1e-300, 1e-310])
def test_direct(ctx, s, tiny, coupled):
    n = 9
    A = (4.0 * np.eye(n) - np.eye(n, k=1) - np.eye(n, k=-1))[:, :, None]
    B, X = tiny_diagonal(s, tiny, coupled), inputs.random_tensor((n, s, 1), seed=s)
    C = kr.sylv_apply(A, B, X)
    got = from_dev(ctx.t_bartels_stewart(to_dev(A), to_dev(B), to_dev(C)))
    np.testing.assert_allclose(got, X, rtol=0, atol=RTOL * np.abs(X).max())


def test_block_arnoldi(ctx):
    import torch
    n, s = 40, 2
    A = (4.0 * np.eye(n) - np.eye(n, k=1) - np.eye(n, k=-1))[:, :, None]
    B, X = tiny_diagonal(s, 1e-160, False), inputs.random_tensor((n, s, 1), seed=3)
    C = kr.sylv_apply(A, B, X)
    op = ctx.op_create_dense(to_dev(A), to_dev(B))
    Xd = torch.zeros((1, s, n), dtype=torch.float64, device="cuda")
    res = ctx.tba_solve(op, to_dev(C), Xd, restart=10, tol=1e-10)
    assert res.status == 0, res
    assert np.linalg.norm(from_dev(Xd) - X) <= 1e-9 * np.linalg.norm(X)   # ||M^-1|| < 1, ||C|| < 10 ||X||
