"""One-launch FP64 application of small operators against the three-launch form and against a plain FFT reference."""
import pytest
import torch

from paper_2405_09233_gb300 import Context

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = Context(0)
    yield c
    c.workspace_check()
    c.close()


def _problem(n, s, p, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    r = lambda *shape: torch.randn(shape, dtype=torch.float64, device="cuda", generator=g)
    return r(p, n, n), r(p, s, s), r(p, s, n)


def _reference(A, B, X):
    Ah, Bh, Xh = (torch.fft.rfft(t, dim=0) for t in (A, B, X))
    return torch.fft.irfft(torch.matmul(Xh, Ah) - torch.matmul(Bh, Xh), n=X.shape[0], dim=0)


# tile edges (4 rows, 2 or 4 columns), every transform (powers of two, direct sums of each bound), one slice,
# long thin tiles, and sizes on either side of the rule
@pytest.mark.parametrize("n,s,p", [(1, 1, 1), (1, 1, 2), (1, 3, 4), (3, 2, 2), (4, 4, 4), (5, 3, 3), (7, 9, 5), (6, 5, 8),
                                   (24, 24, 4), (33, 6, 16), (9, 17, 31), (12, 8, 32), (13, 4, 12), (64, 64, 4),
                                   (2, 130, 2), (200, 3, 1), (300, 20, 3), (100, 50, 7)])
def test_small_apply(ctx, n, s, p):
    A, B, X = _problem(n, s, p, 7 * n + s + p)
    op = ctx.op_create_dense(A, B)
    Y = ctx.sylv_apply(op, X)
    split = ctx.tstar(A, X) - ctx.tstar(X, B)   # the general transforms and products, each its own launch
    ref = _reference(A, B, X)
    # sums of at most 2 (n + s) p products of standard normals, each rounding 2^-53: the error grows like the
    # square root of the count, the result like it too; 64 roundings of the largest entry bound both
    tol = 64 * 2.0 ** -53 * max(float(ref.abs().max()), float((n + s) * p) ** 0.5)
    assert float((Y - ref).abs().max()) <= tol
    assert float((Y - split).abs().max()) <= tol


@pytest.mark.parametrize("n,s,p", [(5, 3, 3), (24, 24, 4), (17, 30, 8)])
def test_small_residual(ctx, n, s, p):
    A, B, Xs = _problem(n, s, p, 3)
    A = A * (0.1 / n ** 0.5)
    B = B * (0.1 / s ** 0.5)
    A[0] += 4 * torch.eye(n, dtype=torch.float64, device="cuda")
    B[0] -= 4 * torch.eye(s, dtype=torch.float64, device="cuda")
    op = ctx.op_create_dense(A, B)
    C = _reference(A, B, Xs).contiguous()
    X0 = Xs * 0.5                              # a non-zero start: the first residual is formed by the operator
    want = float((C - _reference(A, B, X0)).norm())
    res = ctx.tgmres_solve(op, C, X0, restart=20, tol=1e-11)
    assert abs(res.true_history[0] - want) <= 1e-12 * want
    assert res.true_history[-1] <= 1e-11 * float(C.norm())
