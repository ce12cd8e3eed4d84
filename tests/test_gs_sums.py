"""Inner products of an FP32 Krylov basis hold at least what FP64 sums of the same FP32 groups hold."""
import subprocess

import numpy as np
import pytest

from oracle import krylov as kr
from paper_2405_09233_gb300 import Context, build, inputs
from tests.gpu_helpers import to_dev

SOURCE = r"""
#include <cstdio>
#include <cmath>
#include <random>
#include "gs_sweep.cuh"
// The largest ratio of a Triple sum's error to the FP64 bound n 2^-53 sum |x|, over chains and trees of n terms whose
// exponents spread over `spread` powers of two; the exact sums are 128-bit integers (multiples of 2^-80).
int main() {
  std::mt19937_64 r(7);
  double worst = 0.0;
  for (int n : {2, 3, 16, 100, 3000, 20000})
    for (int spread : {1, 12, 30, 50})
      for (int sign = 0; sign < 2; ++sign)
        for (int rep = 0; rep < 20; ++rep) {
          ts::Triple part[16];
          __int128 exact = 0;
          double mag = 0.0;
          for (int i = 0; i < n; ++i) {
            const float x = std::ldexp((float)((1 << 23) + (int)(r() & 0x7fffff)), -23 - (int)(r() % spread)) *
                            (sign && (r() & 1) ? -1.f : 1.f);
            ts::add_to(part[i % 16], x);
            exact += (__int128)std::ldexp((double)x, 80);
            mag += std::fabs((double)x);
          }
          for (int s = 8; s > 0; s /= 2)
            for (int i = 0; i < s; ++i) part[i] = ts::add_sums(part[i], part[i + s]);
          __int128 got = 0;   // the terms, their sums and rounding errors are multiples of 2^-72
          for (float p : {part[0].hi, part[0].mid, part[0].lo}) got += (__int128)std::ldexp((double)p, 80);
          const double err = std::fabs((double)(got - exact)) * std::ldexp(1.0, -80);
          const double rounded = std::fabs(ts::value_of(part[0]) - (double)exact * std::ldexp(1.0, -80));
          worst = std::fmax(worst, std::fmax(err, rounded) / (n * std::ldexp(1.0, -53) * mag));
        }
  std::printf("%.3e\n", worst);
  // a single product is added exactly
  ts::Triple t;
  const float a[1] = {1.f + std::ldexp(1.f, -23)}, b[1] = {1.f - std::ldexp(1.f, -24)};
  ts::add_products(t, a, b);
  std::printf("%d\n", ts::value_of(t) == (double)a[0] * (double)b[0]);
}
"""


def test_sums_against_exact_ones(tmp_path):
    """Host build of the kernels' own addition; the three parts must beat the a-priori bound of FP64 summation."""
    (tmp_path / "sums.cu").write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC,
                    str(tmp_path / "sums.cu"), "-o", str(tmp_path / "sums")], check=True, capture_output=True)
    out = subprocess.run([str(tmp_path / "sums")], check=True, capture_output=True, text=True).stdout.split()
    assert float(out[0]) <= 1.0 and out[1] == "1", out


def equal_products():
    """p = 1, A = 0, B = diag(c, 2c, ..): C of +-1 entries (V_1 = C / 64 exactly), M(V_1) = -b_j V_1, so every
    product <V_1, M(V_1)> adds is c or 2c times 2^-12: sums of two and of four are exact in FP32, FP32 chains of
    eight err by 1.5e-7.  The first estimate is ||C|| sd / sqrt(mean^2 + sd^2) of b's entries."""
    n, s, c = 512, 8, 13421860 * 2.0 ** -23
    b = np.where(np.arange(s) % 2 == 0, c, 2 * c)
    C = np.where(inputs.random_tensor((n, s, 1), seed=5) > 0, 1.0, -1.0)
    first = np.std(b) / np.hypot(np.mean(b), np.std(b))
    return np.zeros((n, n, 1)), np.diag(b)[:, :, None], C, first


# FP32 roundings left: the pairs or fours of squares under the norm (2^-24 each way, halved by the root, at most
# 3 of them) and the subtraction of the projection.
RTOL = 2.0 ** -24


@pytest.mark.gpu
def test_cluster_step():
    ctx = Context(0)
    A, B, C, first = equal_products()
    op = ctx.op_create_dense(to_dev(A), to_dev(B))
    X = to_dev(np.zeros_like(C))
    res = ctx.tgmres_solve(op, to_dev(C), X, restart=1, tol=1e-10, precision="mixed_fp32", max_outer=1)
    assert abs(res.history[0] / 64.0 / first - 1.0) <= RTOL, res.history[0] / 64.0 / first - 1.0
    op.close()
    ctx.close()


@pytest.mark.gpu
def test_batch():
    ctx = Context(0)
    A, B, C, first = equal_products()
    ops = [ctx.op_create_dense(to_dev(A), to_dev(B)) for _ in range(2)]
    Xs = [to_dev(np.zeros_like(C)) for _ in range(2)]
    res = ctx.batched_solve(ops, [to_dev(C)] * 2, Xs, restart=1, tol=1e-10, precision="mixed_fp32", max_outer=1)
    for info in res[1]:
        assert abs(info.relres_est / first - 1.0) <= RTOL, info.relres_est / first - 1.0
    for op in ops:
        op.close()
    ctx.close()
