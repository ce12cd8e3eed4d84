"""Statistics of a small operator's one-launch application: booked whole, as the header says."""
import math

import pytest

from paper_2405_09233_gb300 import Context, inputs
from tests.gpu_helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,s,p,one", [(24, 24, 4, True), (16, 16, 31, True), (96, 96, 1, True), (300, 200, 4, False)])
def test_small_application(n, s, p, one):
    K = p // 2 + 1
    real = 2 if p % 2 == 0 else 1
    product = n * s * (n + s) * (8 * (K - real) + 2 * real)
    with Context(0) as ctx:
        pr = inputs.dense_problem(n, s, p, seed=1)
        op = ctx.op_create_dense(to_dev(pr.A), to_dev(pr.B))
        X = to_dev(pr.Xstar)
        ctx.stats_enable(True)
        ctx.stats_reset()
        ctx.sylv_apply(op, X)
        st = ctx.stats_get()
        assert (st.gemm_launches, st.fft_launches) == ((1, 0) if one else (1, 2))
        assert st.launches == (1 if one else 3)
        dfts = 2 * n * s * 2.5 * p * math.log2(p) if one else 0.0
        assert st.gemm_flops == pytest.approx(product + dfts, rel=1e-12)
        op.close()
