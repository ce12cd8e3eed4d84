"""Transforms of tube lengths that are no power of two: shared out over threads where tubes are few, one thread
per tube where they are many, and both planar layouts of the tensor-core operands in one pass."""
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


def _randn(seed, *shape):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(shape, dtype=torch.float64, device="cuda", generator=g)


def _product(A, X):
    return torch.fft.irfft(torch.matmul(torch.fft.rfft(X, dim=0), torch.fft.rfft(A, dim=0)), n=A.shape[0], dim=0)


@pytest.mark.parametrize("p", [1, 3, 5, 6, 7, 9, 12, 15, 17, 24, 31])
@pytest.mark.parametrize("n1,n2,m", [(3, 2, 1), (33, 70, 5), (300, 200, 100), (420, 80, 400)])
def test_tstar(ctx, n1, n2, m, p):
    A, X = _randn(p, p, n2, n1), _randn(p + 1, p, m, n2)
    ref = _product(A, X)
    # sums of n2 p products of standard normals, each entry sqrt(n2 p) large: 64 roundings of that size
    assert float((ctx.tstar(A, X) - ref).abs().max()) <= 64 * 2.0 ** -53 * max(float(ref.abs().max()), (n2 * p) ** 0.5)


@pytest.mark.parametrize("precision,bits", [("mixed_bf16", 9), ("mixed_tf32", 11), ("mixed_tf32x3", 21),
                                            ("mixed_fp32", 24)])
@pytest.mark.parametrize("n,s,p", [(24, 8, 3), (130, 33, 7), (65, 31, 12), (257, 129, 31), (700, 300, 6)])
def test_lowp_layouts(ctx, n, s, p, precision, bits):
    """Unit operators pass the transformed operand through, in the column-major layout (A = I, B = 0) and in the
    row-major one (A = 0, B = -I): what comes back is X with every coefficient rounded to `bits` bits, and
    p-term FP32 sums before and after."""
    X = _randn(3, p, s, n).float()
    zero = lambda k: torch.zeros(p, k, k, dtype=torch.float64, device="cuda")
    tol = 2.0 ** -bits + 2 * p * 2.0 ** -24
    for left in (True, False):
        A, B = zero(n), zero(s)
        if left:
            A[0].fill_diagonal_(1.0)
        else:
            B[0].fill_diagonal_(-1.0)
        Y = ctx.sylv_apply_lowp(ctx.op_create_dense(A, B), X, precision).double()
        assert float((Y - X.double()).norm()) <= tol * float(X.double().norm())
