"""Batches called on a stream of the caller's own (a non-blocking one): the same bits as on the default stream, on the
first call of a context, where every table is new."""
import numpy as np
import pytest
import torch

from oracle import krylov as kr
from paper_2405_09233_gb300 import Context, inputs
from tests.gpu_helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,engine", [("fp64", "dfma"), ("mixed_bf16", "ozaki"), ("mixed_fp32", "dfma")])
def test_side_stream(tmp_path, monkeypatch, precision, engine):
    monkeypatch.setenv("TSTAR_TUNE_CACHE", str(tmp_path / "tune"))   # the same launch shapes in both contexts
    shapes = [(70, 20, 4), (130, 66, 3), (33, 9, 8), (96, 96, 4)]
    prs = [inputs.dense_problem(*s, seed=sum(s)) for s in shapes]
    Cs = [to_dev(kr.sylv_apply(q.A, q.B, q.Xstar)) for q in prs]
    out = []
    for stream in (torch.cuda.default_stream(), torch.cuda.Stream()):
        ctx = Context(0)
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            ops = [ctx.op_create_dense(to_dev(q.A), to_dev(q.B)) for q in prs]
            Xs = [torch.zeros_like(C) for C in Cs]
            status, _, _ = ctx.batched_solve(ops, Cs, Xs, tol=1e-10, precision=precision, engine=engine)
            assert status == 0
            stream.synchronize()
        out.append([X.cpu().numpy() for X in Xs])
        for op in ops:
            op.close()
        ctx.workspace_check()
        ctx.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
