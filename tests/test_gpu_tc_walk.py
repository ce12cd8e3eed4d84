"""The persistent walk of the single operator's tensor-core products (more tiles than SMs, at most 256 stages a tile),
with the column tile fixed through the tuning cache so that the form is known: against the form with one CTA per tile
(bit for bit), against the oracle, and when a wait expires."""
import numpy as np
import pytest

from oracle import krylov as kr, tproduct as tp
from paper_2405_09233_gb300 import Context, TstarError, inputs
from tests.gpu_helpers import from_dev, to_dev
from tests.test_gpu_lowp import U
from tests.test_gpu_tune import _device_tag, _key

pytestmark = pytest.mark.gpu

# (n, s, p): column tiles that walk persistently
WALKS = {(1000, 700, 7): (64, 128), (640, 640, 16): (64, 128), (300, 1100, 4): (64,), (2000, 130, 6): (64,)}


def walks(shape, prec, bn):
    import torch
    n, s, p = shape
    elems, parts = (64, 1) if prec == "mixed_bf16" else (32, 3 if prec == "mixed_tf32x3" else 1)
    tiles = -(-n // 128) * -(-s // bn) * (p // 2 + 1)
    stages = parts * (-(-n // elems) + -(-s // elems))
    return bn <= 128 and stages <= 256 and tiles > torch.cuda.get_device_properties(0).multi_processor_count


def forced(tmp_path, monkeypatch, tag, shape, prec, bn):
    cache = tmp_path / f"forced_{bn}.txt"
    cache.write_text(f"{tag} {_key(shape, prec)} {bn}\n")
    monkeypatch.setenv("TSTAR_TUNE_CACHE", str(cache))
    return Context(0)


@pytest.mark.parametrize("prec", ["mixed_bf16", "mixed_tf32", "mixed_tf32x3"])
@pytest.mark.parametrize("shape", WALKS, ids=lambda s: "x".join(map(str, s)))
def test_products(tmp_path, monkeypatch, shape, prec):
    import torch
    n, s, p = shape
    tag = _device_tag(tmp_path, monkeypatch)
    pr = inputs.dense_problem(n, s, p, seed=n + s, scale=0.3)
    X32 = inputs.random_tensor(shape, seed=p).astype(np.float32)
    out = {}
    for bn in (64, 128, 256):
        assert walks(shape, prec, bn) == (bn in WALKS[shape])
        with forced(tmp_path, monkeypatch, tag, shape, prec, bn) as ctx:
            op = ctx.op_create_dense(to_dev(pr.A), to_dev(pr.B))
            out[bn] = from_dev(ctx.sylv_apply_lowp(op, torch.from_numpy(inputs.to_device_layout(X32)).cuda(), prec))
            assert ctx.tune_entries()[_key(shape, prec)] == bn
            op.close()
            ctx.workspace_check()
    for bn in WALKS[shape]:
        assert np.array_equal(out[bn].view(np.uint32), out[256].view(np.uint32)), bn
    # the bound of test_gpu_lowp
    ref = kr.sylv_apply(pr.A, pr.B, X32.astype(np.float64))
    Ab, Bb, Xb = (np.abs(T).sum(axis=2) for T in (pr.A, pr.B, X32.astype(np.float64)))
    bound = 4.0 * (2 * U[prec] + (n + s + p) * 2.0 ** -24) * (Ab @ Xb + Xb @ Bb)[:, :, None]
    assert np.all(np.abs(out[64].astype(np.float64) - ref) <= bound)


@pytest.mark.parametrize("prec", ["mixed_bf16", "mixed_tf32x3"])
def test_expired_wait(tmp_path, monkeypatch, prec):
    """As test_gpu_failure, on the persistent walk: the stalled product times out, the context goes on."""
    import torch
    shape = (300, 1100, 4)
    tag = _device_tag(tmp_path, monkeypatch)
    assert walks(shape, prec, 64)
    pr = inputs.dense_problem(*shape, seed=3)
    Cd = to_dev(kr.sylv_apply(pr.A, pr.B, pr.Xstar))
    with forced(tmp_path, monkeypatch, tag, shape, prec, 64) as ctx:
        op = ctx.op_create_dense(to_dev(pr.A), to_dev(pr.B))
        X = torch.zeros_like(Cd)
        monkeypatch.setenv("TSTAR_TEST_STALL_TMA", "1")
        with pytest.raises(TstarError) as e:
            ctx.tgmres_solve(op, Cd, X, restart=3, tol=1e-10, precision=prec, max_outer=1)
        assert e.value.status == -5, e.value          # TS_ERR_TIMEOUT
        monkeypatch.delenv("TSTAR_TEST_STALL_TMA")
        X.zero_()
        res = ctx.tgmres_solve(op, Cd, X, restart=20, tol=1e-10, precision=prec)
        assert res.status == 0, res
        assert tp.norm(from_dev(X) - pr.Xstar) <= 1e-8 * tp.norm(pr.Xstar)
        op.close()
        ctx.workspace_check()
