"""The emulated-FP64 product against its own definition in exact integers: with p = 1 (the DFTs are the identity) and
a fixed point that holds every kept digit pair, Y is the kept pairs' sum, rounded once."""
import math

import numpy as np
import pytest

from paper_2405_09233_gb300 import Context, inputs
from tests.gpu_helpers import from_dev, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = Context(0)
    yield c
    c.workspace_check()
    c.close()


def exponent(*tensors):
    """max |entry| < 2^(E - 1)."""
    return math.frexp(max(np.abs(t).max() for t in tensors))[1] + 1


def digits_of(Z, E, S):
    """Balanced base-256 digits of round(Z 2^(8 S - E)), halves away from zero: S int64 matrices, most significant
    first, |d| <= 128."""
    q = np.array([[int(math.floor(abs(math.ldexp(v, 8 * S - E)) + 0.5)) * (1 if v >= 0 else -1) for v in row]
                  for row in Z], dtype=object)
    out = []
    for _ in range(S - 1):
        low = (q + 128) % 256 - 128
        out.append(low.astype(np.int64))
        q = (q - low) // 256
    out.append(q.astype(np.int64))
    return out[::-1]


@pytest.mark.parametrize("digits", [3, 4, 5, 6])
@pytest.mark.parametrize("shape", [(3, 2), (40, 24), (33, 90), (140, 70)], ids=lambda s: "n%d_s%d" % s)
def test_kept_pairs_are_summed_exactly(ctx, shape, digits):
    n, s = shape
    S = digits
    F = 63 - math.ceil(math.log2(2 * (n + s)))
    if 8 * (S + 1) > F:
        pytest.skip("the fixed point rounds the lowest pairs")
    A, B = (inputs.random_tensor((k, k, 1), seed=k) for k in (n, s))
    X = inputs.random_tensor((n, s, 1), seed=n + s)
    Eo, Ex = exponent(A, B), exponent(X)
    dA, dB, dX = (digits_of(Z[:, :, 0], E, S) for Z, E in ((A, Eo), (B, Eo), (X, Ex)))
    total = np.zeros((n, s), dtype=object)
    for u in range(1, S + 1):
        for v in range(1, S + 2 - u):   # digits u of the operator and v of X, u + v <= S + 1
            pair = dA[u - 1] @ dX[v - 1] - dX[v - 1] @ dB[u - 1]
            total += pair.astype(object) * 256 ** (S + 1 - u - v)
    want = np.array([[math.ldexp(float(t), Eo + Ex - 8 * (S + 1)) for t in row] for row in total])
    op = ctx.op_create_dense(to_dev(A), to_dev(B))
    got = from_dev(ctx.sylv_apply_ozaki(op, to_dev(X), digits=S))[:, :, 0]
    op.close()
    assert np.array_equal(got, want), np.abs(got - want).max()
