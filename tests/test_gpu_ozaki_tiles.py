"""The emulated-FP64 product at the edges of its tiles (128 rows; 64 columns, 128 in a real slice; 32-deep
k-blocks, two per unit with up to 4 digits) and of its fixed point (its caps bind for few unknowns), for every
digit count, held to the bound derived in test_gpu_ozaki."""
import numpy as np
import pytest

from oracle import krylov as kr, tproduct as tp
from paper_2405_09233_gb300 import Context, inputs
from tests.gpu_helpers import fp64_product_bound, from_dev, to_dev
from tests.test_gpu_ozaki import ozaki_bound

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (2, 1, 2), (8, 8, 3), (20, 12, 2), (31, 33, 2), (32, 32, 1), (40, 24, 3), (64, 64, 2), (65, 64, 4),
          (64, 65, 3), (65, 129, 2), (128, 127, 3), (129, 128, 2), (257, 97, 3), (96, 257, 1)]


@pytest.fixture(scope="module")
def ctx():
    c = Context(0)
    yield c
    c.workspace_check()
    c.close()


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_every_digit_count(ctx, shape):
    n, s, p = shape
    A, B = inputs.random_tensor((n, n, p), seed=n + 1), inputs.random_tensor((s, s, p), seed=s + 2)
    X = inputs.random_tensor((n, s, p), seed=p + 3)
    op = ctx.op_create_dense(to_dev(A), to_dev(B))
    ref = kr.sylv_apply(A, B, X)
    fp64 = (fp64_product_bound(np.abs(A), np.abs(X), tp.tprod, p + n)
            + fp64_product_bound(np.abs(X), np.abs(B), tp.tprod, p + s))
    for digits in (8, 7, 6, 5, 4, 3):      # prepared with 8, then through the leading ones
        Y = from_dev(ctx.sylv_apply_ozaki(op, to_dev(X), digits=digits))
        err = np.abs(Y - ref)
        assert np.all(err <= fp64 + ozaki_bound(A, B, X, digits)), (digits, err.max())
    op.close()


def test_extreme_entries(ctx):
    """Every digit at its largest magnitude: all entries just below a power of two, one sign per operand."""
    n, s, p = 130, 66, 1
    v = np.nextafter(1.0, 0.0)
    A, B, X = np.full((n, n, p), -v), np.full((s, s, p), v), np.full((n, s, p), v)
    op = ctx.op_create_dense(to_dev(A), to_dev(B))
    for digits in (8, 6, 5, 4, 3):
        Y = from_dev(ctx.sylv_apply_ozaki(op, to_dev(X), digits=digits))
        np.testing.assert_allclose(Y, -(n + s) * v * v, rtol=0, atol=float(ozaki_bound(A, B, X, digits)) + 1e-12)
    op.close()
