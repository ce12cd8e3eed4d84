"""The Gram-Schmidt sweep by blocks of eight basis vectors against the oracle's vector-by-vector one.

Restart lengths around one and two blocks, and vector lengths around the line between the one-launch cluster
step (at most 8192 entries) and the chain of launches, with lengths that no 16-byte access divides."""
import numpy as np
import pytest

from oracle import krylov as kr, tproduct as tp
from paper_2405_09233_gb300 import Context, inputs
from tests.gpu_helpers import from_dev, to_dev

pytestmark = pytest.mark.gpu

CASES = [  # (n, s, p, m)
    (3, 2, 1, 5), (13, 5, 1, 8), (24, 24, 4, 9), (24, 24, 4, 16), (24, 24, 4, 17), (65, 63, 2, 20),
    (32, 32, 8, 20), (91, 91, 1, 18), (64, 43, 3, 17), (91, 91, 3, 9), (120, 111, 5, 20)]


@pytest.fixture(scope="module")
def ctx():
    c = Context(0)
    yield c
    c.workspace_check()
    c.close()


def solve(ctx, method, pr, C, m, **kw):
    op = ctx.op_create_dense(to_dev(pr.A), to_dev(pr.B))
    X = to_dev(np.zeros_like(C))
    fn = ctx.tgmres_solve if method == "gmres" else ctx.tfom_solve
    res = fn(op, to_dev(C), X, restart=m, tol=1e-10, **kw)
    X = from_dev(X)
    op.close()
    return X, res


@pytest.mark.parametrize("method", ["gmres", "fom"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "n%d_s%d_p%d_m%d" % c)
def test_history_matches_mgs(ctx, method, case):
    n, s, p, m = case
    pr = inputs.dense_problem(n, s, p, seed=900 + n)
    C = kr.sylv_apply(pr.A, pr.B, pr.Xstar)
    X, res = solve(ctx, method, pr, C, m)
    ref = kr.restarted_solve(method, pr.A, pr.B, C, m=m, tol=1e-10)
    # both sweeps lose orthogonality like u kappa: estimates differ far less than the tolerance they are cut at
    assert res.status == 0 and len(res.history) == len(ref.history)
    np.testing.assert_allclose(res.history, ref.history, rtol=0, atol=1e-12 * ref.normC)
    assert tp.norm(C - kr.sylv_apply(pr.A, pr.B, X)) <= 1e-10 * tp.norm(C)


@pytest.mark.parametrize("case", [(24, 24, 4, 20), (32, 32, 8, 9), (91, 91, 1, 17), (120, 110, 4, 20)],
                         ids=lambda c: "n%d_s%d_p%d_m%d" % c)
def test_fp32_basis(ctx, case):
    """An FP32 basis: estimates of the first inner steps against FP64 ones (FP32 products of n + s terms and sums
    of FP32 vectors, a few hundred roundings of 6e-8 relative to the residual they start from)."""
    n, s, p, m = case
    pr = inputs.dense_problem(n, s, p, seed=950 + n)
    C = kr.sylv_apply(pr.A, pr.B, pr.Xstar)
    X, res = solve(ctx, "gmres", pr, C, m, precision="mixed_fp32")
    ref = kr.restarted_solve("gmres", pr.A, pr.B, C, m=m, tol=1e-10)
    first = min(len(ref.history), len(res.history), m, 8)
    np.testing.assert_allclose(res.history[:first], ref.history[:first], rtol=0, atol=2e-5 * ref.normC)
    assert res.status == 0 and tp.norm(C - kr.sylv_apply(pr.A, pr.B, X)) <= 1e-10 * tp.norm(C)


@pytest.mark.parametrize("method", ["gmres", "fom"])
@pytest.mark.parametrize("case", [(24, 24, 4, 20), (91, 91, 1, 17), (60, 64, 16, 12)],
                         ids=lambda c: "n%d_s%d_p%d_m%d" % c)
def test_launched_ahead_gives_the_same_bits(ctx, monkeypatch, method, case):
    """Steps launched ahead come up while their predecessors still run; step by step they do not."""
    n, s, p, m = case
    pr = inputs.dense_problem(n, s, p, seed=970 + n)
    C = kr.sylv_apply(pr.A, pr.B, pr.Xstar)
    runs = [solve(ctx, method, pr, C, m) for _ in range(5)]
    monkeypatch.setenv("TSTAR_NO_LAUNCH_AHEAD", "1")
    X, res = solve(ctx, method, pr, C, m)
    for Xa, ra in runs:
        assert np.array_equal(Xa, X) and np.array_equal(np.asarray(ra.history), np.asarray(res.history))
