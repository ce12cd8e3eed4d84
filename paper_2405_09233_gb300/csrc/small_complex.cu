// Small dense complex FP64 kernels for the projected equation of TBAS and for t-Bartels-Stewart
// (§4, Algorithm 5; §5.2, the projected equation H_m*Y - Y*B = C1).
//
// Per Fourier slice the tensor equation is the matrix Sylvester equation H_k Y_k - Y_k B_k = F_k.
// It is solved by the Hessenberg-Schur form of Bartels-Stewart: only B_k (s x s) is reduced to
// complex Schur form B_k = Q T Q^H (schur.cu); with Z = Y Q and G = F Q,
// column j of Z solves (H_k - t_jj I) z_j = g_j + sum_{i<j} t_ij z_i.  The shifted matrices are
// factorised in parallel (one CTA per (slice, j), LU with partial pivoting restricted to the lower
// bandwidth, which is s for the block Hessenberg H_m of TBA and n-1 for a general matrix), then one
// CTA per slice sweeps j in order.  All matrices are column-major complex (double2).
#include "internal.cuh"
#include "reduce.cuh"
#include "tba.cuh"
#include "complex_ops.cuh"

namespace ts {
namespace {

// Squares of entries whose squared modulus lies in this range neither overflow nor lose bits.
constexpr double kSqLo = 1e-280, kSqHi = 1e280;
__device__ __forceinline__ double cnorm(double2 z) { return fma(z.y, z.y, z.x * z.x); }
// a - b c in four FP64 instructions.
__device__ __forceinline__ double2 cfms(double2 a, double2 b, double2 c) {
  return make_double2(fma(b.y, c.y, fma(-b.x, c.x, a.x)), fma(-b.y, c.x, fma(-b.x, c.y, a.y)));
}
__device__ __forceinline__ double2 cfma(double2 a, double2 b, double2 c) {   // a + b c
  return make_double2(fma(-b.y, c.y, fma(b.x, c.x, a.x)), fma(b.y, c.x, fma(b.x, c.y, a.y)));
}
__device__ __forceinline__ double2 crecip(double2 z) {
  const double n = cnorm(z);
  if (n >= kSqLo && n <= kSqHi) {
    const double d = 1.0 / n;
    return make_double2(z.x * d, -z.y * d);
  }
  return cdiv(make_double2(1.0, 0.0), z);
}

// LU with partial pivoting of M = H_k - t_jj I, lower bandwidth bw, one CTA per (j, k).
// LU[(k*s + j)] is an N x N column-major factor; piv holds the row chosen at each step.
//
// GB300 issues an FP64 instruction of one warp in 64 clocks, so the serial part of a column (pivot
// search, reciprocal, multipliers: one warp) costs as much as many columns of the update.  Interval c
// therefore overlaps them: warps 1-7 apply column c (row interchange, then M[r, q] -= l_r u_q, a warp
// per column and a lane per row, so that a column's band is read in whole lines) to the columns
// q >= c + 2, while warp 0 applies it to column c + 1, finds that column's pivot and forms its
// multipliers; one barrier per column.  Pivots are compared by squared modulus as bit patterns (an
// integer comparison; hypot only where a square could leave the FP64 range).
// banded = 1 (the band form, bw < N - 1): row interchanges are applied from column c on, so L keeps
// its band and the solve interleaves interchanges and eliminations.  banded = 0: they are applied to
// the whole rows, so that P b is formed once and L is a plain triangle.  On exit the diagonal holds the
// reciprocals 1 / u_cc and the rows of U are scaled by them (unit upper triangle): a step of the
// solve is then one multiply-subtract instead of a division and one.
// Measured: n = s = 64, p = 8 (320 factorisations) 981 -> 457 us; N = 320, bw = 32
// (160) 8.66 -> 5.33 ms.
constexpr int kLuMaxBw = 512;
constexpr int kLuThreads = 256;
__global__ void __launch_bounds__(kLuThreads) k_shifted_lu(const double2* __restrict__ H, long long sH,
                                                           const double2* __restrict__ T, double2* LU,
                                                           int* __restrict__ piv, int N, int bw, int s, int banded,
                                                           int* err) {
  const int j = blockIdx.x, k = blockIdx.y;
  const double2* Hk = H + (long long)k * sH;
  const double2 shift = T[(long long)k * s * s + (long long)j * s + j];
  double2* M = LU + ((long long)k * s + j) * N * N;
  int* pv = piv + ((long long)k * s + j) * N;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __shared__ int sp[2];
  __shared__ unsigned long long sbest[kLuThreads / 32];
  __shared__ double2 sl[2][kLuMaxBw];
  // max |M|: a pivot below N * 1e-14 * max|M| marks a (numerically) singular shift
  unsigned long long mb = 0;
  for (long long e = threadIdx.x; e < (long long)N * N; e += blockDim.x) {
    double2 v = Hk[e];
    if ((e % N) == (e / N)) v = csub(v, shift);
    M[e] = v;
    mb = max(mb, (unsigned long long)__double_as_longlong(cnorm(v)));
  }
  auto block_max = [&](unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    if (lane == 0) sbest[warp] = v;
    __syncthreads();
    v = 0;
    for (int w = 0; w < kLuThreads / 32; ++w) v = max(v, sbest[w]);
    return v;
  };
  double big = __longlong_as_double((long long)block_max(mb));
  if (big >= kSqLo && big <= kSqHi) {
    big = sqrt(big);
  } else {   // squares out of range (or no finite entry)
    mb = 0;
    for (long long e = threadIdx.x; e < (long long)N * N; e += blockDim.x)
      mb = max(mb, (unsigned long long)__double_as_longlong(cabs2(M[e])));
    big = __longlong_as_double((long long)block_max(mb));
  }
  const double tiny = 1e-14 * N * big;
  // Pivot of column c, interchange inside the column, multipliers into the column and sl[c & 1]: one warp.
  auto pivot_column = [&](int c) {
    double2* Mc = M + (long long)N * c;
    const int rmax = (c + bw < N - 1) ? c + bw : N - 1, nr = rmax - c;
    unsigned long long best = 0;
    int bi = c;
    bool exact = false;
    for (int pass = 0; pass < 2; ++pass) {
      best = 0;
      bi = c;
      for (int r = c + lane; r <= rmax; r += 32) {
        const double v = exact ? cabs2(Mc[r]) : cnorm(Mc[r]);
        const unsigned long long b = (unsigned long long)__double_as_longlong(v) + 1;   // 0: no candidate
        if (b > best) {
          best = b;
          bi = r;
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ob > best || (ob == best && oi < bi)) {
          best = ob;
          bi = oi;
        }
      }
      const double v = __longlong_as_double((long long)(best - 1));
      if (exact || (v >= kSqLo && v <= kSqHi)) break;
      exact = true;   // the largest squared modulus is out of range: compare the moduli themselves
    }
    const int p = bi;
    const double2 d = Mc[p];
    const double mod = exact ? __longlong_as_double((long long)(best - 1)) : 0.0;
    const bool small = exact ? !(mod > tiny) : !(cnorm(d) > tiny * tiny);
    if (lane == 0) {
      pv[c] = p;
      sp[c & 1] = p;
      if (small) atomicOr(err, 2);
    }
    const double2 dinv = crecip(d), top = Mc[c];
    __syncwarp();
    for (int r = lane; r < nr; r += 32) {
      const double2 v = c + 1 + r == p ? top : Mc[c + 1 + r];
      const double2 l = make_double2(fma(-v.y, dinv.y, v.x * dinv.x), fma(v.y, dinv.x, v.x * dinv.y));
      Mc[c + 1 + r] = l;
      if (r < kLuMaxBw) sl[c & 1][r] = l;
    }
    __syncwarp();
    if (lane == 0) Mc[c] = dinv;
  };
  // Column c applied to column q (one warp, a lane per row).
  auto update_column = [&](int c, int q, int p) {
    const int rmax = (c + bw < N - 1) ? c + bw : N - 1, nr = rmax - c;
    double2* Mq = M + (long long)N * q;
    const double2* Mc = M + (long long)N * c;
    const double2 u = Mq[p], old = Mq[c];
    __syncwarp();
    for (int r = lane; r < nr; r += 32) {
      const double2 v = c + 1 + r == p ? old : Mq[c + 1 + r];
      const double2 l = r < kLuMaxBw ? sl[c & 1][r] : Mc[c + 1 + r];
      Mq[c + 1 + r] = cfms(v, l, u);
    }
    __syncwarp();
    if (lane == 0 && p != c) Mq[c] = u;
  };
  __syncthreads();
  if (warp == 0) pivot_column(0);
  __syncthreads();
  for (int c = 0; c < N; ++c) {
    const int p = sp[c & 1];
    if (warp == 0) {
      if (c + 1 < N) {
        update_column(c, c + 1, p);
        __syncwarp();
        pivot_column(c + 1);
      }
    } else {
      for (int q = c + 1 + warp; q < N; q += kLuThreads / 32 - 1) update_column(c, q, p);
      if (!banded && p != c)   // the interchange in the columns of L too
        for (int q = threadIdx.x - 32; q < c; q += kLuThreads - 32) {
          double2* Mq = M + (long long)N * q;
          const double2 t0 = Mq[c];
          Mq[c] = Mq[p];
          Mq[p] = t0;
        }
    }
    __syncthreads();
  }
  // rows of U scaled by the reciprocals on the diagonal
  for (int q = warp; q < N; q += kLuThreads / 32)
    for (int r = lane; r < q; r += 32) {
      const double2 d = M[r + (long long)N * r], v = M[r + (long long)N * q];
      M[r + (long long)N * q] = make_double2(fma(-v.y, d.y, v.x * d.x), fma(v.y, d.x, v.x * d.y));
    }
}

// One CTA per slice: Z[:, j] for j = 0..s-1 in order, using the factors of k_shifted_lu.  The column
// sweep is serial by nature (column j needs every earlier one), and so are the substitutions inside it,
// so the kernel is bound by the FP64 instructions of one warp per eliminated unknown (four, plus a
// shared-memory round trip) and by what it can overlap with them:
//   banded L   one warp applies the block's interchanges and eliminations in order, the band of L staged
//              in shared memory;
//   triangles  (U, and L when not banded) in blocks of kHsB unknowns: warp 0 substitutes inside the
//              diagonal block, then every warp updates the next block's rows (its columns split over the
//              warps, partial sums added in a fixed order), and warps 1-7 update the remaining rows while
//              warp 0 goes on with the next block.
// U's rows are already scaled to a unit diagonal, so a substitution step has no division.
// Measured: n = s = 64, 5 slices 8.97 -> 2.46 ms; N = 320, bw = 32, s = 32,
// 5 slices 22.4 -> 7.9 ms.
constexpr int kHsB = 32;
constexpr int kHsBandStage = 64;
constexpr int kHsThreads = 256;
__global__ void __launch_bounds__(kHsThreads) k_hs_solve(const double2* __restrict__ LU, const int* __restrict__ piv,
                                                         const double2* __restrict__ G, const double2* __restrict__ T,
                                                         double2* __restrict__ Z, int N, int bw, int s, int banded) {
  const int k = blockIdx.x;
  const double2* Gk = G + (long long)k * N * s;
  const double2* Tk = T + (long long)k * s * s;
  double2* Zk = Z + (long long)k * N * s;
  extern __shared__ double2 hs_smem[];
  double2* rhs = hs_smem;                                      // N
  double2* Lb = rhs + N;                                       // banded: kHsB x bw (the block's band of L)
  double2* Ub = Lb + (banded ? (size_t)kHsB * bw : 0);         // 2 x kHsB x (kHsB + 1): diagonal blocks
  double2* part = Ub + 2 * kHsB * (kHsB + 1);                  // kHsThreads: partial sums
  __shared__ int spv[kHsB];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int NW = kHsThreads / 32;

  // Unit triangular solve on rhs; lower: rows and columns in increasing order, else decreasing.
  auto solve_triangle = [&](const double2* M, bool lower) {
    const int nblk = (N + kHsB - 1) / kHsB;
    auto block0 = [&](int b) { return lower ? b * kHsB : N - (b + 1) * kHsB; };   // first row, may be negative
    auto stage = [&](int b, int t, int nt) {   // diagonal block b into its buffer
      const int c0 = block0(b);
      double2* U = Ub + (b & 1) * kHsB * (kHsB + 1);
      for (int e = t; e < kHsB * kHsB; e += nt) {
        const int rr = c0 + e % kHsB, cc = c0 + e / kHsB;
        U[e % kHsB + (kHsB + 1) * (e / kHsB)] =
            rr >= 0 && cc >= 0 && rr < N && cc < N ? M[rr + (long long)N * cc] : make_double2(0.0, 0.0);
      }
    };
    stage(0, tid, kHsThreads);
    __syncthreads();
    for (int b = 0; b < nblk; ++b) {
      const int c0 = block0(b);
      if (warp == 0) {
        const double2* U = Ub + (b & 1) * kHsB * (kHsB + 1);
        const int row = c0 + lane;
        const bool live = row >= 0 && row < N;
        double2 v = live ? rhs[row] : make_double2(0.0, 0.0);
        const int steps = lower ? min(kHsB, N - c0) : kHsB + min(c0, 0);
#pragma unroll 4
        for (int q = 0; q < steps; ++q) {
          const int cc = lower ? q : kHsB - 1 - q;
          const double2 z = make_double2(__shfl_sync(0xffffffffu, v.x, cc), __shfl_sync(0xffffffffu, v.y, cc));
          if (lower ? lane > cc : lane < cc) v = cfms(v, U[lane + (kHsB + 1) * cc], z);
        }
        if (live) rhs[row] = v;
      } else if (b > 0) {
        // rows beyond the current block, updated by the block before it
        const int p0 = block0(b - 1);
        const int r0 = lower ? c0 + kHsB : 0, r1 = lower ? N : c0;
        const int q0 = max(p0, 0), q1 = min(p0 + kHsB, N);
        for (int r = r0 + tid - 32; r < r1; r += kHsThreads - 32) {
          double2 v = rhs[r];
#pragma unroll 4
          for (int q = q0; q < q1; ++q) v = cfms(v, M[r + (long long)N * q], rhs[q]);
          rhs[r] = v;
        }
        if (b + 1 < nblk) stage(b + 1, tid - 32, kHsThreads - 32);
      } else if (b + 1 < nblk) {
        stage(b + 1, tid - 32, kHsThreads - 32);
      }
      __syncthreads();
      if (b + 1 < nblk) {   // the next block's rows, updated by this block: 4 columns per warp
        const int row = block0(b + 1) + lane;
        const bool live = row >= 0 && row < N;
        double2 v = make_double2(0.0, 0.0);
        if (live) {
#pragma unroll
          for (int t = 0; t < kHsB / NW; ++t) {
            const int q = c0 + warp * (kHsB / NW) + t;
            if (q >= 0 && q < N) v = cfms(v, M[row + (long long)N * q], rhs[q]);
          }
        }
        part[tid] = v;
        __syncthreads();
        if (warp == 0 && live) {
          v = rhs[row];
#pragma unroll
          for (int w = 0; w < NW; ++w) v = cadd(v, part[w * 32 + lane]);
          rhs[row] = v;
        }
        __syncthreads();
      }
    }
  };

  for (int j = 0; j < s; ++j) {
    const double2* M = LU + ((long long)k * s + j) * N * N;
    const int* pv = piv + ((long long)k * s + j) * N;
    for (int r = tid; r < N; r += kHsThreads) {
      double2 v = Gk[r + (long long)N * j];
      for (int i = 0; i < j; ++i) v = cfma(v, Tk[i + (long long)s * j], Zk[r + (long long)N * i]);
      rhs[r] = v;
    }
    __syncthreads();
    if (banded) {
      // forward: row interchanges and the unit lower factor, in order
      for (int c0 = 0; c0 < N; c0 += kHsB) {
        const int nb = min(kHsB, N - c0);
        for (int e = tid; e < nb * bw; e += kHsThreads) {
          const int cc = e / bw, t = e % bw, c = c0 + cc, r = c + 1 + t;
          Lb[e] = r < N ? M[r + (long long)N * c] : make_double2(0.0, 0.0);
        }
        for (int cc = tid; cc < nb; cc += kHsThreads) spv[cc] = pv[c0 + cc];
        __syncthreads();
        if (warp == 0) {
          for (int cc = 0; cc < nb; ++cc) {
            const int c = c0 + cc, p = spv[cc], nr = min(bw, N - 1 - c);
            const double2 rc = rhs[p], old = rhs[c];
            __syncwarp();
            for (int t = lane; t < nr; t += 32) {
              const double2 v = c + 1 + t == p ? old : rhs[c + 1 + t];
              rhs[c + 1 + t] = cfms(v, Lb[cc * bw + t], rc);
            }
            if (lane == 0) rhs[c] = rc;
            __syncwarp();
          }
        }
        __syncthreads();
      }
    } else {
      if (warp == 0) {   // P rhs: the interchanges in order
        for (int c0 = 0; c0 < N; c0 += 32) {
          const int mine = c0 + lane < N ? pv[c0 + lane] : 0, nb = min(32, N - c0);
          for (int cc = 0; cc < nb; ++cc) {
            const int p = __shfl_sync(0xffffffffu, mine, cc);
            if (lane == 0 && p != c0 + cc) {
              const double2 t0 = rhs[c0 + cc];
              rhs[c0 + cc] = rhs[p];
              rhs[p] = t0;
            }
          }
        }
      }
      __syncthreads();
      solve_triangle(M, true);
    }
    for (int r = tid; r < N; r += kHsThreads) {   // the diagonal (reciprocals)
      const double2 d = M[r + (long long)N * r], v = rhs[r];
      rhs[r] = make_double2(fma(-v.y, d.y, v.x * d.x), fma(v.y, d.x, v.x * d.y));
    }
    __syncthreads();
    solve_triangle(M, false);
    for (int r = tid; r < N; r += kHsThreads) Zk[r + (long long)N * j] = rhs[r];
    __syncthreads();
  }
}

// C = A * op(B) for small column-major complex matrices per slice: op = none or conjugate
// transpose.  A: M x L (lda), B: L x Ncol (or Ncol x L when conjugate-transposed).
__global__ void k_small_gemm(const double2* __restrict__ A, long long sA, int lda, const double2* __restrict__ B,
                             long long sB, int ldb, int transB, double2* __restrict__ C, long long sC, int ldc, int M,
                             int L, int Ncol, int accumulate) {
  const int k = blockIdx.y;
  const double2* Ak = A + (long long)k * sA;
  const double2* Bk = B + (long long)k * sB;
  double2* Ck = C + (long long)k * sC;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < (long long)M * Ncol;
       e += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(e % M), j = (int)(e / M);
    double2 acc = accumulate ? Ck[i + (long long)ldc * j] : make_double2(0.0, 0.0);
    for (int l = 0; l < L; ++l) {
      const double2 b = transB ? cconj(Bk[j + (long long)ldb * l]) : Bk[l + (long long)ldb * j];
      acc = cadd(acc, cmul(Ak[i + (long long)lda * l], b));
    }
    Ck[i + (long long)ldc * j] = acc;
  }
}

// Cholesky G = R^H R of a Hermitian positive definite s x s matrix per slice and the inverse of R, one CTA
// each, both in shared memory.  R and Rinv are written upper triangular (zeros below).  A pivot d_j (the
// squared norm of column j's part orthogonal to the previous columns, when G is a Gram matrix) fails when
// it is not above max(rel * g_jj, tiny2 * max_k g_jj(k)), the second maximum taken over the Grams of all K
// slices; rel = tiny2 = 0 asks for d_j > 0 only.  A failed slice stops early (nothing written), sets
// fail_slice[slice] = 1 (each slice's entry is reset to 0 first) and err bit 4 (err may be NULL).
// What bounds it: the chain of s pivots (a square root, a division) with the FP64 issue of one SM; the
// right-looking forms leave a rank-one update between pivots, spread over all threads: warp 0 forms a
// pivot and scales its row, every thread updates.
// Measured: s = 32, 5 slices 279 (two one-warp kernels on global memory) -> 63 us.
constexpr int kCholThreads = 256;
__global__ void __launch_bounds__(kCholThreads) k_cholesky_inverse(const double2* __restrict__ Gall,
                                                                   double2* __restrict__ Rall,
                                                                   double2* __restrict__ Xall, int s, int K, double rel,
                                                                   double tiny2, int* err, int* fail_slice) {
  extern __shared__ double2 chol_smem[];
  const int ld = s + 1, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  double2* A = chol_smem;                 // G, then R; (r, c) at r + ld c
  double2* X = chol_smem + (size_t)s * ld;   // accumulates sum_c R(a, c) X(c, b), then R^-1
  __shared__ double floor_d[64], inv_d[64];
  __shared__ int bad;
  const double2* G = Gall + (long long)blockIdx.x * s * s;
  for (int e = tid; e < s * s; e += kCholThreads) {
    A[e % s + ld * (e / s)] = G[e];
    X[e % s + ld * (e / s)] = make_double2(0.0, 0.0);
  }
  for (int j = tid; j < s; j += kCholThreads) {
    double f = rel * G[j + (long long)s * j].x;
    if (tiny2 > 0.0) {
      double ref2 = 0.0;
      for (int q = 0; q < K; ++q) ref2 = fmax(ref2, Gall[(long long)q * s * s + j + (long long)s * j].x);
      f = fmax(f, tiny2 * ref2);
    }
    floor_d[j] = f;
  }
  if (tid == 0) {
    bad = 0;
    if (fail_slice) fail_slice[blockIdx.x] = 0;
  }
  __syncthreads();
  for (int j = 0; j < s; ++j) {
    if (warp == 0) {
      const double d = A[j + ld * j].x;
      if (!(d > floor_d[j])) {
        if (lane == 0) {
          bad = 1;
          if (err) atomicOr(err, 4);
          if (fail_slice) fail_slice[blockIdx.x] = 1;
        }
      } else {
        const double rjj = sqrt(d), inv = 1.0 / rjj;
        __syncwarp();
        for (int q = j + 1 + lane; q < s; q += 32) A[j + ld * q] = cscale(A[j + ld * q], inv);
        if (lane == 0) {
          A[j + ld * j] = make_double2(rjj, 0.0);
          inv_d[j] = inv;
        }
      }
    }
    __syncthreads();
    if (bad) return;
    // A(p, q) -= conj(R(j, p)) R(j, q), j < p <= q
    const int m = s - 1 - j;
    for (int e = tid; e < m * m; e += kCholThreads) {
      const int p = j + 1 + e % m, q = j + 1 + e / m;
      if (p <= q) {
        const double2 u = A[j + ld * p];
        A[p + ld * q] = cfms(A[p + ld * q], make_double2(u.x, -u.y), A[j + ld * q]);
      }
    }
    __syncthreads();
  }
  for (int a = s - 1; a >= 0; --a) {   // row a of R^-1, then its part of the rows above
    const double inv = inv_d[a];
    for (int b = a + tid; b < s; b += kCholThreads) {
      const double2 v = X[a + ld * b];
      X[a + ld * b] = b == a ? make_double2(inv, 0.0) : make_double2(-v.x * inv, -v.y * inv);
    }
    __syncthreads();
    const int m = s - a;
    for (int e = tid; e < a * m; e += kCholThreads) {
      const int r = e % a, b = a + e / a;
      X[r + ld * b] = cfma(X[r + ld * b], A[r + ld * a], X[a + ld * b]);
    }
    __syncthreads();
  }
  double2* R = Rall + (long long)blockIdx.x * s * s;
  double2* Xo = Xall + (long long)blockIdx.x * s * s;
  for (int e = tid; e < s * s; e += kCholThreads) {
    const int r = e % s, c = e / s;
    R[e] = r <= c ? A[r + ld * c] : make_double2(0.0, 0.0);
    Xo[e] = r <= c ? X[r + ld * c] : make_double2(0.0, 0.0);
  }
}

}  // namespace

namespace {
// The band form of the factors pays while the band is well inside the matrix and its block of L fits
// the staging buffer (TBAS: bw = s, N = m s); otherwise plain triangles.
bool band_form(int N, int bw) { return bw <= kHsBandStage && 2 * bw < N; }
}  // namespace

void shifted_lu(const double2* H, long long sH, const double2* T, double2* LU, int* piv, int N, int bw, int s, int K,
                int* err, cudaStream_t st) {
  k_shifted_lu<<<dim3(s, K), kLuThreads, 0, st>>>(H, sH, T, LU, piv, N, bw, s, band_form(N, bw), err);
  count_launch();
  TS_CUDA(cudaGetLastError());
}

void hs_solve(const double2* LU, const int* piv, const double2* G, const double2* T, double2* Z, int N, int bw, int s,
              int K, cudaStream_t st) {
  const bool band = band_form(N, bw);
  const size_t smem = sizeof(double2) * ((size_t)N + (band ? (size_t)kHsB * bw : 0) + 2 * (size_t)kHsB * (kHsB + 1) +
                                         kHsThreads);
  TS_REQUIRE(smem <= 226 * 1024, "projected system too large");
  set_max_dynamic_smem((const void*)k_hs_solve, (int)smem);
  k_hs_solve<<<K, kHsThreads, smem, st>>>(LU, piv, G, T, Z, N, bw, s, band);
  count_launch();
  TS_CUDA(cudaGetLastError());
}

void small_gemm(const double2* A, long long sA, int lda, const double2* B, long long sB, int ldb, bool transB, double2* C,
                long long sC, int ldc, int M, int L, int Ncol, int K, bool accumulate, cudaStream_t st) {
  long long tot = (long long)M * Ncol;
  int g = (int)((tot + 255) / 256);
  if (g > 1024) g = 1024;
  k_small_gemm<<<dim3(g, K), 256, 0, st>>>(A, sA, lda, B, sB, ldb, transB ? 1 : 0, C, sC, ldc, M, L, Ncol,
                                           accumulate ? 1 : 0);
  count_launch();
  TS_CUDA(cudaGetLastError());
}

void cholesky_inverse(const double2* G, double2* R, double2* Rinv, int s, int K, double rel, double tiny2, int* err,
                      int* fail_slice, cudaStream_t st) {
  TS_REQUIRE(s <= 64, "cholesky_inverse: block width above 64");
  const size_t smem = 2 * sizeof(double2) * (size_t)s * (s + 1);
  set_max_dynamic_smem((const void*)k_cholesky_inverse, (int)smem);
  k_cholesky_inverse<<<K, kCholThreads, smem, st>>>(G, R, Rinv, s, K, rel, tiny2, err, fail_slice);
  count_launch();
  TS_CUDA(cudaGetLastError());
}

}  // namespace ts
