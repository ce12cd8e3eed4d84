"""The tensor-core slice products with more tiles than SMs (persistent walk) against fewer: an operator whose first
block column alone fits one wave gives the same bits there, whatever walks the tiles."""
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


@pytest.mark.parametrize("precision", ["mixed_bf16", "mixed_tf32", "mixed_tf32x3"])
@pytest.mark.parametrize("n,s,p", [(1000, 700, 7), (640, 640, 16), (300, 1100, 4), (2000, 130, 6)])
def test_columns_do_not_depend_on_the_walk(ctx, n, s, p, precision):
    """With B = 0 every column of M(X) = A*X depends on its own column of X only, so applying A to the first 64
    columns (few tiles) and to all of them (more tiles than SMs) runs the same MMAs in the same order."""
    g = torch.Generator(device="cuda")
    g.manual_seed(n + s)
    A = torch.randn((p, n, n), dtype=torch.float64, device="cuda", generator=g)
    X = torch.randn((p, s, n), dtype=torch.float32, device="cuda", generator=g)
    zero = lambda k: torch.zeros((p, k, k), dtype=torch.float64, device="cuda")
    whole = ctx.sylv_apply_lowp(ctx.op_create_dense(A, zero(s)), X, precision)
    part = ctx.sylv_apply_lowp(ctx.op_create_dense(A, zero(64)), X[:, :64].contiguous(), precision)
    assert torch.equal(whole[:, :64], part)
    last = ctx.sylv_apply_lowp(ctx.op_create_dense(A, zero(30)), X[:, s - 30:].contiguous(), precision)
    assert torch.equal(whole[:, s - 30:], last)
