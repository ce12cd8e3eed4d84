// The small FP64 problems of tGMRES and tFOM, kept on the device so the Arnoldi loop never
// waits for the host between steps.
//
// tGMRES (§3.3): y = argmin || beta e1 - Htilde_k y ||_2.  The QR factorisation of Htilde_k that
// Proposition 3.4 refers to is built one column at a time with Givens rotations: column j of H
// receives the j earlier rotations, a new rotation zeroes h_{j+1,j}, and the rotated right-hand
// side g gives the residual norm |gamma_{j+1}| = |g_{j+1}| without forming y.
// tFOM (§3.2): H_k y = beta e1 by Gaussian elimination with partial pivoting (a Hessenberg
// matrix only needs a choice between rows c and c+1 at column c), also one column at a time: the
// eliminations of the columns before k - 1 do not depend on k, and the last column has none; the estimate
// is h_{k+1,k} |y_k| (Proposition 3.3), y_k = (right-hand side)_k / (last pivot).
#include <algorithm>
#include "internal.cuh"
#include "reduce.cuh"
#include "gs_sweep.cuh"

namespace ts {
namespace {

constexpr int kMaxM = 256;     // longest restart

// tFOM keeps its eliminated columns in R, the multipliers and row choices in cs and sn, its right-hand side in g.
struct Layout {
  int m;
  __host__ __device__ size_t H() const { return 0; }
  __host__ __device__ size_t R() const { return (size_t)(m + 1) * m; }
  __host__ __device__ size_t cs() const { return R() + (size_t)(m + 1) * m; }
  __host__ __device__ size_t sn() const { return cs() + m; }
  __host__ __device__ size_t g() const { return sn() + m; }
  __host__ __device__ size_t y() const { return g() + m + 1; }
  __host__ __device__ size_t est() const { return y() + m; }
  __host__ __device__ size_t beta() const { return est() + 8; }
  __host__ __device__ size_t gram() const { return beta() + 8; }   // row i: <V_i, V_l>, l in i's block before i
  __host__ __device__ size_t hist() const { return gram() + (size_t)(m + 1) * kGB; }
  __host__ __device__ size_t total() const { return hist() + m; }
};

constexpr double kBreakdownRel = 1e-14;

__global__ void k_ks_init(double* st, int m, const double* beta_in) {
  Layout L{m};
  const double beta = beta_in[0];
  for (int i = threadIdx.x; i < (m + 1) * m; i += blockDim.x) {
    st[L.H() + i] = 0.0;
    st[L.R() + i] = 0.0;
  }
  for (int i = threadIdx.x; i <= m; i += blockDim.x) st[L.g() + i] = (i == 0) ? beta : 0.0;
  for (int i = threadIdx.x; i < m; i += blockDim.x) st[L.y() + i] = 0.0;
  if (threadIdx.x == 0) {
    st[L.beta()] = beta;
    st[L.beta() + 1] = beta > 0.0 ? 1.0 / beta : 0.0;
    for (int q = 0; q < 8; ++q) st[L.est() + q] = 0.0;
  }
}

// est[0] = estimate, est[1] = 1/h_{j+1,j}, est[2] = h_{j+1,j}, est[3] = flags (1 breakdown,
// 2 singular, 4 non-finite), est[4] = steps taken in this cycle (j + 1); hist[j] = estimate of
// step j.  In a graph-captured cycle, `handle` is the conditional handle of step j + 1 (0 for the
// last step) and the update decides whether the cycle goes on: it sets that handle to 0 on breakdown,
// a bad step, an estimate <= stop[0] (the tolerance times ||C||) or <= stop[1] (the inner tolerance
// of mixed precision, or -1).  `gate` is closed under the same conditions (launched-ahead cycles).
struct StepEnd {
  cudaGraphConditionalHandle handle;
  const double* stop;
  int* gate;
};

// The column update of step j.  One thread runs it; what it reads is staged in shared memory by all threads
// first (ks_load), so that it does not wait on a chain of dependent global loads.
struct KsStage {
  double cs[kMaxM], sn[kMaxM];
  double g, diag, sub, beta, stop0, stop1;
};

__device__ __forceinline__ void ks_load(KsStage& S, const double* st, int m, int j, int method, const StepEnd& end,
                                        int t, int nt) {
  Layout L{m};
  const int ld = m + 1;
  for (int i = t; i < j; i += nt) {
    S.cs[i] = st[L.cs() + i];
    S.sn[i] = st[L.sn() + i];
  }
  if (t == nt - 1) S.beta = st[L.beta()];
  if (t == nt - 2 && end.stop) {
    S.stop0 = end.stop[0];
    S.stop1 = end.stop[1];
  }
  if (t == nt - 3) S.g = method != 0 && j > 0 ? st[L.g() + j - 1] : st[L.g() + j];
  if (t == nt - 4 && method != 0 && j > 0) {
    S.diag = st[L.R() + (j - 1) + (size_t)ld * (j - 1)];
    S.sub = st[L.H() + j + (size_t)ld * (j - 1)];
  }
}

// tFOM: the elimination of column j - 1, which step j's row makes possible.
__device__ __forceinline__ void ks_pivot(KsStage& S, double* st, int m, int j, int method) {
  if (method == 0 || j == 0) return;
  Layout L{m};
  const double t = S.diag, b = S.sub, rhs = S.g;
  const bool swap = fabs(b) > fabs(t);
  const double piv = swap ? b : t, f = piv != 0.0 ? (swap ? t : b) / piv : 0.0;
  S.cs[j - 1] = f;
  S.sn[j - 1] = swap ? 1.0 : 0.0;
  st[L.cs() + j - 1] = f;
  st[L.sn() + j - 1] = swap ? 1.0 : 0.0;
  st[L.R() + (j - 1) + (size_t)(m + 1) * (j - 1)] = piv;
  st[L.g() + j - 1] = swap ? 0.0 : rhs;
  S.g = swap ? rhs : 0.0 - f * rhs;
}

// The earlier rotations (tGMRES) or eliminations (tFOM) on entries c0 .. c1 - 1 of column j; t is the entry
// carried from row to row.
__device__ __forceinline__ void ks_rotate(const KsStage& S, double* st, int m, int j, int method, int c0, int c1,
                                          const double* h, double& t) {
  double* R = st + Layout{m}.R() + (size_t)(m + 1) * j;
  for (int i = c0; i < c1; ++i) {
    const double b = h[i - c0];
    if (i == 0) {
      t = b;
      continue;
    }
    const double c = S.cs[i - 1], s = S.sn[i - 1];
    if (method == 0) {
      R[i - 1] = c * t + s * b;
      t = c * b - s * t;
    } else {
      const double top = s != 0.0 ? b : t, bot = s != 0.0 ? t : b;
      R[i - 1] = top;
      t = bot - c * top;
    }
  }
}

// sqrt(x) and its reciprocal.  rsqrt and one correction where x is in the middle of the range: half the
// FP64 instructions of sqrt and a division.
__device__ __forceinline__ void root(double x, double& r, double& inv) {
  if (x > 1e-280 && x < 1e280) {
    inv = rsqrt(x);
    r = x * inv;
    r = fma(0.5 * inv, fma(-r, r, x), r);
  } else {
    r = sqrt(x);
    inv = r > 0.0 ? 1.0 / r : 0.0;
  }
}

__device__ __forceinline__ void ks_finish(const KsStage& S, double* st, int m, int j, int method, double t, double hn,
                                          double inv, const StepEnd& end) {
  Layout L{m};
  const int ld = m + 1;
  double* R = st + L.R() + (size_t)ld * j;
  st[L.H() + (j + 1) + (size_t)ld * j] = hn;
  double flags = (hn <= kBreakdownRel * S.beta) ? 1.0 : 0.0;
  double est;
  if (method == 0) {
    double r, ri, c = 1.0, s = 0.0;
    const double q = fma(t, t, hn * hn);
    if (q > 1e-280 && q < 1e280) {
      root(q, r, ri);
      c = t * ri;
      s = hn * ri;
    } else {
      r = hypot(t, hn);
      if (r > 0.0) {
        c = t / r;
        s = hn / r;
      }
    }
    st[L.cs() + j] = c;
    st[L.sn() + j] = s;
    R[j] = r;
    R[j + 1] = 0.0;
    const double gn = -s * S.g;
    st[L.g() + j] = c * S.g;
    st[L.g() + j + 1] = gn;
    est = fabs(gn);
  } else {
    R[j] = t;
    st[L.g() + j] = S.g;
    if (t == 0.0) {
      flags += 2.0;
      est = INFINITY;
    } else {
      est = hn * fabs(S.g / t);
    }
  }
  if (!isfinite(est) || !isfinite(hn)) flags += 4.0;
  st[L.est()] = est;
  st[L.est() + 1] = inv;
  st[L.est() + 2] = hn;
  st[L.est() + 3] = flags;
  st[L.est() + 4] = j + 1;
  st[L.hist() + j] = est;
  if (end.handle || end.gate) {
    const bool go = flags == 0.0 && !(est <= S.stop0) && !(est <= S.stop1);
    if (!go) {
      if (end.handle) cudaGraphSetConditional(end.handle, 0);
      if (end.gate) *end.gate = 0;
    }
  }
}

// Everything of inner step j after W = M(V_j), for vectors of at most kArnMaxN entries, in one launch of a
// thread-block cluster of CL <= kArnCL CTAs: the sweep, h_{j+1,j} = ||W||, the column update (by one thread
// of CTA 0, a warp that does nothing else, beside the sweep) and V_{j+1} = W / h_{j+1,j}.  CTA c owns a
// contiguous part of the vectors in shared memory, W for the whole step and the basis one block ahead
// (cp.async).  Warp q forms the inner products with the block's vector q, stores the sum into every CTA's
// shared memory, and after one cluster barrier each CTA adds all parts in the same fixed order, so every CTA
// holds the same coefficients, bit for bit.  All CTAs pass the same barriers (j is a kernel argument; the gate
// is read once, before the first barrier, and written by CTA 0 only after the last), the first barrier
// precedes every remote store and no remote store follows the last one.
//
// Bound by FP64 issue (64 clocks per warp instruction and sub-partition) and by the reduction's round trip.
// The 20 steps of a cycle, vector by vector -> by blocks: 2304 FP64 entries 517 -> 260 us, 8000 FP64 931 ->
// 448, 8000 FP32 861 -> 294 (with FP64 sums over eight products; Triples over two take 2% less).
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

constexpr int kArnCL = 8, kArnWarps = 8, kArnThreads = 32 * (kArnWarps + 1), kArnMaxN = kArnCL * 1024;

__device__ __forceinline__ void cluster_sync_all() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

template <typename T>
__device__ __forceinline__ void cp_async_one(T* dst, const T* src) {
  if constexpr (sizeof(T) == 8)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}

template <typename T>
__global__ void __launch_bounds__(kArnThreads, 1)
    k_arnoldi_cluster(const T* __restrict__ W, T* __restrict__ V, long long ldv, int N, int j, int m, double* st,
                      int method, StepEnd end) {
  step_kernel_begin();
  if (end.gate && *end.gate == 0) return;   // launched ahead of a cycle that has already ended (all CTAs alike)
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double slots[2][kArnCL * 2 * kGB];
  __shared__ double sh[kGB], sG[kGB * kGB], snorm[2];
  __shared__ KsStage S;
  uint32_t rank, ncta;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(ncta));
  const int t = threadIdx.x, lane = t & 31, wp = t >> 5;
  const int Nc = (N + (int)ncta - 1) / (int)ncta, e0 = (int)rank * Nc;
  const int cnt = max(0, min(Nc, N - e0));
  T* w = reinterpret_cast<T*>(smem_raw);
  T* stage = w + Nc;                        // two blocks of kGB parts
  Layout L{m};
  double *H = st + L.H() + (size_t)(m + 1) * j, *G = st + L.gram();
  const int nblk = j / kGB + 1;
  auto in_block = [&](int b) { return min(kGB, j + 1 - kGB * b); };
  auto fetch = [&](int b) {                 // block b's parts, by the sweep's warps
    if (wp < in_block(b) && wp < kArnWarps) {
      T* d = stage + (size_t)((b & 1) * kGB + wp) * Nc;
      const T* v = V + (long long)(kGB * b + wp) * ldv + e0;
      for (int q = lane; q < cnt; q += 32) cp_async_one(d + q, v + q);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  double gnext = 0.0;
  auto fetch_gram = [&](int b) {            // a row of V_j itself is not there yet (and not used)
    if (t < kGB * kGB && t / kGB < in_block(b) && kGB * b + t / kGB < j) gnext = G[(size_t)(kGB * b) * kGB + t];
  };
  for (int q = t; q < cnt; q += kArnThreads) cp_async_one(w + q, W + e0 + q);
  fetch(0);
  fetch_gram(0);
  if (rank == 0) ks_load(S, st, m, j, method, end, t, kArnThreads);
  cluster_sync_all();   // every CTA of the cluster runs before any remote store
  const bool ks = rank == 0 && t == 32 * kArnWarps;
  if (ks) ks_pivot(S, st, m, j, method);
  double carry = 0.0, nrm = 0.0;
  int buf = 0;
  auto store_all = [&](double x, int at, int c) {   // x into slot `at` of CTA c
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_addr(&slots[buf][at])), "r"(c));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(remote), "d"(x) : "memory");
  };
  for (int b = 0; b < nblk; ++b) {
    const int nb = in_block(b);
    const bool last = b + 1 == nblk;
    if (t < kGB * kGB) sG[t] = gnext;
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (!last) {
      fetch(b + 1);
      fetch_gram(b + 1);
    }
    const T* blk = stage + (size_t)(b & 1) * kGB * Nc;
    if (wp < nb && wp < kArnWarps) {
      const T *v = blk + (size_t)wp * Nc, *vj = blk + (size_t)(nb - 1) * Nc;
      const bool gram = last && wp < nb - 1;
      double x = 0.0, y = 0.0;
      if constexpr (sizeof(T) == 8) {
        for (int q = lane; q < cnt; q += 32) {
          x = fma(v[q], w[q], x);
          if (gram) y = fma(v[q], vj[q], y);
        }
      } else {
        Triple f, g;
        for (int q = lane; q < cnt; q += 64) {   // products summed in pairs, the pairs in Triples
          const bool two = q + 32 < cnt;
          const float v2[2] = {v[q], two ? v[q + 32] : 0.f}, w2[2] = {w[q], two ? w[q + 32] : 0.f};
          add_products(f, v2, w2);
          if (gram) {
            const float j2[2] = {vj[q], two ? vj[q + 32] : 0.f};
            add_products(g, v2, j2);
          }
        }
        x = value_of(f);
        if (gram) y = value_of(g);
      }
      // lanes 0-15 end with the sum of x, lanes 16-31 with that of y
      const double o = __shfl_xor_sync(0xffffffffu, lane < 16 ? y : x, 16);
      x = (lane < 16 ? x : y) + o;
#pragma unroll
      for (int d = 8; d > 0; d >>= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
      const int c = lane & 15;
      if (c < (int)ncta && (lane < 16 || gram)) store_all(x, (int)rank * 2 * kGB + (lane >> 4) * kGB + wp, c);
    }
    cluster_sync_all();
    if (wp == 0) {
      const int q = lane & 15;
      const bool used = q < kGB ? q < nb : (last && q - kGB < nb - 1);
      double x = 0.0;
      if (used)
        for (int c = lane >> 4; c < (int)ncta; c += 2) x += slots[buf][c * 2 * kGB + q];
      x += __shfl_xor_sync(0xffffffffu, x, 16);
      double row[kGB - 1];
#pragma unroll
      for (int l = 0; l < kGB - 1; ++l) {
        const double gj = __shfl_sync(0xffffffffu, x, kGB + l);
        row[l] = last && lane == nb - 1 ? gj : sG[(lane & 7) * kGB + l];
      }
      if (last && rank == 0 && lane >= kGB && lane < kGB + nb - 1) G[(size_t)j * kGB + lane - kGB] = x;
      x = gs_forward(x, row, nb, lane);
      if (lane < nb) {
        sh[lane] = x;
        if (rank == 0) H[kGB * b + lane] = x;
      }
    }
    __syncthreads();
    if (wp < kArnWarps) {
      T h[kGB];
#pragma unroll
      for (int q = 0; q < kGB; ++q) h[q] = q < nb ? (T)sh[q] : T(0);
      float f = 0.f;
      for (int e = t, u = 0; e < cnt; e += 32 * kArnWarps, ++u) {
        T x = w[e];
#pragma unroll
        for (int q = 0; q < kGB; ++q)
          if (q < nb) x = x - h[q] * blk[(size_t)q * Nc + e];
        w[e] = x;
        if (last) {
          if constexpr (sizeof(T) == 8) {
            nrm = fma(x, x, nrm);
          } else {
            f = fmaf(x, x, f);
            if ((u & 1) == 1) {
              nrm += (double)f;
              f = 0.f;
            }
          }
        }
      }
      if (sizeof(T) == 4 && last) nrm += (double)f;
    } else if (ks) {
      ks_rotate(S, st, m, j, method, kGB * b, kGB * b + nb, sh, carry);
    }
    buf ^= 1;
  }
  if (wp < kArnWarps) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) nrm += __shfl_xor_sync(0xffffffffu, nrm, d);
    if (lane < (int)ncta) store_all(nrm, (int)rank * 2 * kGB + wp, lane);
  }
  cluster_sync_all();
  if (wp == 0) {
    double x = 0.0;
    for (int q = lane; q < (int)ncta * kArnWarps; q += 32) x += slots[buf][(q / kArnWarps) * 2 * kGB + q % kArnWarps];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
    double hn, inv;
    root(x, hn, inv);
    if (lane == 0) {
      snorm[0] = hn;
      snorm[1] = inv;
    }
  }
  __syncthreads();
  if (wp < kArnWarps) {
    const T inv = (T)snorm[1];
    T* Vn = V + (long long)(j + 1) * ldv + e0;
    for (int e = t; e < cnt; e += 32 * kArnWarps) Vn[e] = w[e] * inv;
  } else if (ks) {
    ks_finish(S, st, m, j, method, carry, snorm[0], snorm[1], end);
  }
}

// Longer vectors: the same step as a chain of launches over the whole chip, one per block of the sweep and
// two more.  Pass b = -1 forms the first block's inner products; pass b subtracts block b and forms those of
// block b + 1, or ||W||^2 after the last.  A CTA writes its sums to P[sum][CTA]; the next launch adds them
// up in every CTA (in the same order, so all have the same coefficients).
// Bound by memory from about a million entries on (FP32: 16.8M entries, 20 steps move 37.6 GB in 6.6 ms), by
// round trips below.  The sweeps of a 20-step cycle, against a launch per basis vector (reading W, V_i and
// V_i+1, writing W) above 65536 entries and one cluster launch per step below: FP64, 61440 entries 1877 ->
// 542 us, 262144 1534 -> 745, 4.2M 8474 -> 5556; FP32, 1.05M 1944 -> 888, 16.8M 10303 -> 6427 (sums in two
// FP32 parts; in three, 3% more).  The line to
// the cluster form lies where both take the same time (FP64, 8000 entries in the cluster 457 us, 8200 here 451).
constexpr int kGsBlocks = 152;

template <typename T, int PK, int VB>
__global__ void __launch_bounds__(512, 1)
    k_gs_pass(T* __restrict__ W, const T* __restrict__ V, long long ldv, long long NP, int j, int b,
              const double* __restrict__ Pin, double* __restrict__ Pout, double* st, int m, const int* gate) {
  step_kernel_begin();
  if (gate && *gate == 0) return;
  const GsPass g(j, b);
  Layout L{m};
  T h[VB];
  gs_coefficients<T, VB>(g, Pin, kGsBlocks, 0, gridDim.x, st + L.gram(), st + L.H() + (size_t)(m + 1) * j,
                         blockIdx.x == 0, h);
  GsSums<T, VB> sums;
  gs_stream<T, PK, VB>(g, W, V, ldv, (long long)blockIdx.x * blockDim.x + threadIdx.x, NP,
                       (long long)gridDim.x * blockDim.x, h, sums);
  gs_store<T, VB>(g, sums, Pout, kGsBlocks, blockIdx.x);
}

// h_{j+1,j} from the last pass's sums, V_{j+1} = W / h_{j+1,j}, and the column update (the last CTA).
template <typename T, int PK>
__global__ void __launch_bounds__(512, 1)
    k_gs_finish(const T* __restrict__ W, T* __restrict__ Vn, long long NP, const double* __restrict__ Pin, int nparts,
                int j, int m, double* st, int method, StepEnd end) {
  step_kernel_begin();
  __shared__ double snorm[2];
  __shared__ double col[kMaxM];
  __shared__ KsStage S;
  const int t = threadIdx.x, lane = t & 31;
  const bool update = blockIdx.x == gridDim.x - 1;
  Layout L{m};
  // Only the CTA that may close the gate looks at it: after the end of a cycle the others form a V_{j+1} that
  // nothing reads.
  if (update && end.gate && *end.gate == 0) return;
  if (update) {
    ks_load(S, st, m, j, method, end, t, blockDim.x);
    for (int i = t; i <= j; i += blockDim.x) col[i] = st[L.H() + i + (size_t)(m + 1) * j];
    __syncthreads();
  }
  double carry = 0.0;
  if (update && t == 32) {
    ks_pivot(S, st, m, j, method);
    ks_rotate(S, st, m, j, method, 0, j + 1, col, carry);
  }
  if (t < 32) {
    double x = 0.0, hn, inv;
    for (int c = lane; c < nparts; c += 32) x += Pin[c];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
    root(x, hn, inv);
    if (lane == 0) {
      snorm[0] = hn;
      snorm[1] = inv;
    }
  }
  __syncthreads();
  if (update) {
    if (t == 32) ks_finish(S, st, m, j, method, carry, snorm[0], snorm[1], end);
    return;
  }
  const T inv = (T)snorm[1];
  const long long stride = (long long)(gridDim.x - 1) * blockDim.x;
  for (long long p = (long long)blockIdx.x * blockDim.x + t; p < NP; p += stride) {
    T w[PK];
    ld_pack<T, PK>(W, p, w);
#pragma unroll
    for (int c = 0; c < PK; ++c) w[c] = w[c] * inv;
    st_pack<T, PK>(Vn, p, w);
  }
}

// Back substitution R_k y = g_k (tGMRES: after the rotations; tFOM: after the eliminations).  Thread r keeps
// row r: each solved entry is broadcast and subtracted by all rows at once, and the diagonal's reciprocals are
// formed together beforehand (one thread, term by term with a division per row, took 16 us at k = 18).
// Up to kSolveStage columns come from shared memory.
constexpr int kSolveStage = 64;
__global__ void k_ks_solve(double* st, int m, int k) {
  __shared__ double sR[kSolveStage * kSolveStage], sy[kMaxM];
  Layout L{m};
  const int ld = m + 1, t = threadIdx.x;
  const double* R = st + L.R();
  const bool staged = k <= kSolveStage;
  if (staged)
    for (int e = t; e < k * k; e += blockDim.x) sR[e % k + kSolveStage * (e / k)] = R[e % k + ld * (e / k)];
  double v = t < k ? st[L.g() + t] : 0.0;
  const double d = t < k ? R[t + ld * t] : 1.0;
  // a quotient as a product with the reciprocal, unless the reciprocal is not a normal number
  const double inv = 1.0 / d;
  const bool ok = fabs(inv) > 1e-290 && fabs(inv) < 1e290;
  __syncthreads();
  for (int c = k - 1; c >= 0; --c) {
    const double r = t < c ? (staged ? sR[t + kSolveStage * c] : R[t + ld * c]) : 0.0;
    if (t == c) sy[c] = ok ? v * inv : v / d;
    __syncthreads();
    if (t < c) v -= r * sy[c];
  }
  if (t < k) st[L.y() + t] = sy[t];
}

}  // namespace

size_t krylov_state_bytes(int m) { return Layout{m}.total() * sizeof(double); }
double* ks_y(void* s, int m) { return static_cast<double*>(s) + Layout{m}.y(); }
double* ks_est(void* s, int m) { return static_cast<double*>(s) + Layout{m}.est(); }
double* ks_beta(void* s, int m) { return static_cast<double*>(s) + Layout{m}.beta(); }

void ks_init(void* state, int m, const double* beta_and_inv, cudaStream_t st) {
  k_ks_init<<<1, 256, 0, st>>>(static_cast<double*>(state), m, beta_and_inv);
  count_launch();
  TS_CUDA(cudaGetLastError());
}

double* ks_hist(void* s, int m) { return static_cast<double*>(s) + Layout{m}.hist(); }

template <typename T>
void launch_arnoldi_cluster(const T* W, T* V, long long ldv, int N, int j, int m, double* s, int method,
                            const StepEnd& end, cudaStream_t st) {
  // CTAs: one per 64 entries up to kArnCL
  const int cl = std::min(kArnCL, std::max(1, (N + 63) / 64));
  const int smem = (int)sizeof(T) * ((N + cl - 1) / cl) * (2 * kGB + 1);
  if (smem > 32 * 1024) set_max_dynamic_smem(reinterpret_cast<const void*>(&k_arnoldi_cluster<T>), smem);
  launch_step_kernel(k_arnoldi_cluster<T>, end.gate != nullptr, cl, kArnThreads, smem, cl, st, W, V, ldv, N, j, m, s,
                     method, end);
  count_launch();
}

template <typename T, int PK>
void launch_gs(T* W, T* V, long long ldv, long long NP, int j, int m, double* s, int method, double* P,
               const StepEnd& end, cudaStream_t st) {
  // one CTA per SM while there is work; few warps where it is little (their sums are FP64 work too)
  const long long per = (NP + kGsBlocks - 1) / kGsBlocks;
  const int nt = per >= 2048 ? 512 : (per >= 512 ? 256 : 128);
  const int nb = (int)std::min<long long>(kGsBlocks, (NP + nt - 1) / nt);
  double* Pb[2] = {P, P + (size_t)kGsSums * kGsBlocks};
  const int nblk = j / kGB + 1;
  for (int b = -1; b < nblk; ++b) {
    launch_step_kernel(j < 4 ? k_gs_pass<T, PK, 4> : k_gs_pass<T, PK, 8>, end.gate != nullptr, nb, nt, 0, 0, st, W, V,
                       ldv, NP, j, b, Pb[(b + 2) & 1], Pb[(b + 1) & 1], s, m, end.gate);
    count_launch();
  }
  launch_step_kernel(k_gs_finish<T, PK>, end.gate != nullptr, nb + 1, nt, 0, 0, st, W, V + (long long)(j + 1) * ldv, NP,
                     Pb[nblk & 1], nb, j, m, s, method, end);
  count_launch();
}

// Every kernel a step of any j may launch is loaded: a capture cannot load one on its first launch.
template <typename T>
void arnoldi_load() {
  cudaFuncAttributes fa;
  constexpr int PK = 16 / sizeof(T);
  const void* fns[] = {(const void*)k_arnoldi_cluster<T>,  (const void*)k_gs_pass<T, PK, 4>,
                       (const void*)k_gs_pass<T, PK, 8>,   (const void*)k_gs_pass<T, 1, 4>,
                       (const void*)k_gs_pass<T, 1, 8>,    (const void*)k_gs_finish<T, PK>,
                       (const void*)k_gs_finish<T, 1>};
  for (const void* f : fns) TS_CUDA(cudaFuncGetAttributes(&fa, f));
}
template void arnoldi_load<double>();
template void arnoldi_load<float>();

size_t arnoldi_scratch_bytes() { return sizeof(double) * 2 * kGsSums * kGsBlocks; }

template <typename T>
void arnoldi_step(T* W, T* V, long long ldv, long long N, int j, int m, void* state, int method, double* scratch,
                  cudaStream_t st, cudaGraphConditionalHandle handle, const double* stop, int* gate) {
  TS_REQUIRE(N >= 1 && j >= 0 && j < m && m <= kMaxM, "arnoldi_step: bad size");
  double* s = static_cast<double*>(state);
  const StepEnd end{handle, stop, gate};
  constexpr int PK = 16 / sizeof(T);
  const auto aligned = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  if (N <= kArnMaxN)
    launch_arnoldi_cluster<T>(W, V, ldv, (int)N, j, m, s, method, end, st);
  else if (N % PK == 0 && ldv % PK == 0 && aligned(W) && aligned(V))
    launch_gs<T, PK>(W, V, ldv, N / PK, j, m, s, method, scratch, end, st);
  else
    launch_gs<T, 1>(W, V, ldv, N, j, m, s, method, scratch, end, st);
  TS_CUDA(cudaGetLastError());
}
template void arnoldi_step<double>(double*, double*, long long, long long, int, int, void*, int, double*, cudaStream_t,
                                   cudaGraphConditionalHandle, const double*, int*);
template void arnoldi_step<float>(float*, float*, long long, long long, int, int, void*, int, double*, cudaStream_t,
                                  cudaGraphConditionalHandle, const double*, int*);

void ks_solve(void* state, int m, int k, cudaStream_t st) {
  TS_REQUIRE(k <= kMaxM, "ks_solve: bad size");
  if (k <= 0) return;
  k_ks_solve<<<1, (k + 31) / 32 * 32, 0, st>>>(static_cast<double*>(state), m, k);
  count_launch();
  TS_CUDA(cudaGetLastError());
}

}  // namespace ts
