"""A batch whose digits of X exceed the emulated products' workspace (4 GiB): it goes through it in groups."""
import numpy as np
import pytest

from oracle import krylov as kr
from paper_2405_09233_gb300 import Context, inputs
from tests.gpu_helpers import from_dev, to_dev

pytestmark = pytest.mark.gpu


def test_workspace_does_not_grow_with_the_batch():
    import torch
    n = s = 8
    p, count, digits, restart = 16, 28000, 6, 4
    K = p // 2 + 1
    planes = count * 2 * digits * K * (3 * s * 64 + 2 * n * 64)   # rows padded to 64: 276 KB an instance, 7.7 GB
    # what else grows with the batch: the basis and three vectors, two spectra; and tables, with a factor of 1.5
    rest = 1.5 * count * (8 * n * s * p * (restart + 4) + 2 * 16 * n * s * K)
    assert planes > 4 * 2 ** 30 + 0.9 * rest
    ctx = Context(0)
    pr = inputs.dense_problem(n, s, p, seed=1)
    C = to_dev(kr.sylv_apply(pr.A, pr.B, pr.Xstar))
    A, B = to_dev(pr.A), to_dev(pr.B)
    ops = [ctx.op_create_dense(A, B) for _ in range(count)]
    Y = torch.empty_like(C)
    for op in ops:
        ctx.sylv_apply_ozaki(op, C, Y, digits=digits)   # the operators' own digits
    X = torch.zeros((count, p, s, n), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    status, infos, statuses = ctx.batched_solve(ops, [C] * count, list(X), restart=restart, tol=1e-10, engine="ozaki",
                                                ozaki_digits=digits)
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] <= 4 * 2 ** 30 + rest
    assert status == 0 and set(statuses) == {0}
    assert torch.equal(X, X[:1].expand_as(X))            # the same equation in every group
    assert np.abs(from_dev(X[0]) - pr.Xstar).max() <= 1e-8 * np.abs(pr.Xstar).max()
    for op in ops:
        op.close()
    ctx.workspace_check()
    ctx.close()
