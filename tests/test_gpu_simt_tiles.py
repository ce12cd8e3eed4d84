"""CUDA-core slice products (FP64 and FP32) at sizes that the dispatch sends to its different tiles, ragged
in every direction, against numpy's FFT route in FP64."""
import numpy as np
import pytest

from paper_2405_09233_gb300 import Context, inputs
from tests.gpu_helpers import U64, from_dev, to_dev

pytestmark = pytest.mark.gpu

SHAPES = [(65, 1, 1), (65, 3, 2), (66, 66, 3), (97, 200, 9), (129, 64, 16), (256, 256, 8), (300, 33, 6), (500, 130, 12),
          (512, 128, 16), (700, 9, 5), (1000, 17, 2)]


@pytest.fixture(scope="module")
def ctx():
    c = Context(0)
    yield c
    c.workspace_check()
    c.close()


def product(A, X):
    """A*X of (n1, n2, p) tensors by the DFT along mode 3."""
    Ah, Xh = np.fft.rfft(A, axis=2), np.fft.rfft(X, axis=2)
    return np.fft.irfft(np.einsum("ilk,ljk->ijk", Ah, Xh, optimize=True), n=A.shape[2], axis=2)


def problem(n, s, p):
    A, B = inputs.random_tensor((n, n, p), seed=n), inputs.random_tensor((s, s, p), seed=s + 1)
    X = inputs.random_tensor((n, s, p), seed=p + 2)
    # Every entry sums p (n + s) products, formed by DFTs and per-slice sums; each operation rounds at most u
    # of a magnitude bounded by (|A| * |X| + |X| * |B|)(i, j, k), and a factor 8 covers the transforms and
    # the three-product complex form.
    size = product(np.abs(A), np.abs(X)) + product(np.abs(X), np.abs(B))
    return A, B, X, product(A, X) - product(X, B), 8.0 * (p + n + s) * size


@pytest.mark.parametrize("dims", SHAPES, ids=lambda d: "n%d_s%d_p%d" % d)
def test_fp64_product(ctx, dims):
    A, B, X, ref, size = problem(*dims)
    op = ctx.op_create_dense(to_dev(A), to_dev(B))
    Y = from_dev(ctx.sylv_apply(op, to_dev(X)))
    assert np.all(np.abs(Y - ref) <= U64 * size)


@pytest.mark.parametrize("dims", SHAPES, ids=lambda d: "n%d_s%d_p%d" % d)
def test_fp32_product(ctx, dims):
    A, B, X, ref, size = problem(*dims)
    op = ctx.op_create_dense(to_dev(A), to_dev(B))
    Y = from_dev(ctx.sylv_apply_lowp(op, to_dev(X).float(), "mixed_fp32"))
    assert np.all(np.abs(Y - ref) <= 2.0 ** -24 * size)
