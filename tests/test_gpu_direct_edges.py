"""t-Bartels-Stewart at the sizes where its kernels change form: the Schur factors in shared memory (T and Q
up to s = 84, T alone up to 119) or global memory, triangles of one block (32) or more, multipliers beyond
the staged 512, and entries whose squares leave the FP64 range."""
import numpy as np
import pytest

from oracle import krylov as kr
from paper_2405_09233_gb300 import Context, TstarError, binding, inputs
from .gpu_helpers import from_dev, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = Context(0)
    yield c
    c.workspace_check()
    c.close()


# The family's M has condition number about 10 (spectra of A and -B in [1, 7]), so a backward stable
# solver's relative error stays below ~ (n + s) u 10 times a modest constant: 1e-11 at these sizes.
RTOL = 1e-11


@pytest.mark.parametrize("dims", [(1, 1, 1), (1, 2, 3), (2, 1, 2), (3, 3, 1), (31, 2, 2), (32, 33, 1), (33, 32, 2),
                                  (65, 5, 4), (8, 84, 1), (8, 85, 1), (4, 119, 1), (4, 120, 1), (600, 1, 1)],
                         ids=lambda d: "n%d_s%d_p%d" % d)
def test_recovers_the_solution(ctx, dims):
    pr = inputs.dense_problem(*dims, seed=sum(dims))
    C = kr.sylv_apply(pr.A, pr.B, pr.Xstar)
    X = from_dev(ctx.t_bartels_stewart(to_dev(pr.A), to_dev(pr.B), to_dev(C)))
    np.testing.assert_allclose(X, pr.Xstar, rtol=0, atol=RTOL * np.abs(pr.Xstar).max())


@pytest.mark.parametrize("power", [-560, 520])
def test_powers_of_two_far_from_one(ctx, power):
    """Scaling A, B and C by one power of two leaves X as it is; the squares of such entries are 0 or Inf."""
    pr = inputs.dense_problem(40, 36, 3, seed=9)
    C = kr.sylv_apply(pr.A, pr.B, pr.Xstar)
    f = 2.0 ** power
    X = from_dev(ctx.t_bartels_stewart(to_dev(pr.A * f), to_dev(pr.B * f), to_dev(C * f)))
    np.testing.assert_allclose(X, pr.Xstar, rtol=0, atol=RTOL * np.abs(pr.Xstar).max())


def test_non_finite_b_is_reported(ctx):
    pr = inputs.dense_problem(6, 5, 2, seed=1)
    pr.B[2, 3, 0] = np.nan
    with pytest.raises(TstarError) as e:
        ctx.t_bartels_stewart(to_dev(pr.A), to_dev(pr.B), to_dev(pr.Xstar))
    assert e.value.status == binding.TS_SINGULAR
