"""Expired waits of the emulated FP64 product, without a fault: with TSTAR_TEST_STALL_TMA=1 its producer loads the
first k-block only.  That block's MMAs run, the MMA warp's wait for the next one expires, the kernel waits for the
MMAs it issued, frees its tensor memory and returns; the solve reports TS_ERR_TIMEOUT and the context goes on."""
import pytest

from oracle import krylov as kr, tproduct as tp
from paper_2405_09233_gb300 import inputs
from tests.gpu_helpers import to_dev, from_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("digits", [3, 6, 7])
def test_emulated_product(monkeypatch, digits):
    import torch
    from paper_2405_09233_gb300 import Context, TstarError
    ctx = Context(0)
    pr = inputs.dense_problem(96, 40, 4, seed=3)
    C = kr.sylv_apply(pr.A, pr.B, pr.Xstar)
    op = ctx.op_create_dense(to_dev(pr.A), to_dev(pr.B))
    Cd = to_dev(C)
    X = torch.zeros_like(Cd)
    solve = dict(engine="ozaki", ozaki_digits=digits, tol=1e-10 if digits > 3 else 1e-4)
    monkeypatch.setenv("TSTAR_TEST_STALL_TMA", "1")
    with pytest.raises(TstarError) as e:
        ctx.tgmres_solve(op, Cd, X, restart=1, **solve)
    assert e.value.status == -5, e.value          # TS_ERR_TIMEOUT
    monkeypatch.delenv("TSTAR_TEST_STALL_TMA")
    X.zero_()
    res = ctx.tgmres_solve(op, Cd, X, restart=20, **solve)
    assert res.status == 0, res
    assert tp.norm(C - kr.sylv_apply(pr.A, pr.B, from_dev(X))) <= 1.01 * solve["tol"] * tp.norm(C)
    op.close()
    ctx.workspace_check()
    ctx.close()
