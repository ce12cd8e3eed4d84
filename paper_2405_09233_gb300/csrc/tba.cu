// Tubal Block Arnoldi (Algorithm 7) and TBAS(m) (Algorithm 8), and t-Bartels-Stewart
// (Algorithm 5), on one GB300 in FP64.
//
// Everything runs in the Fourier domain (Eq. (5)): the T-product decouples into K = p/2 + 1
// independent complex slices, the T-transpose becomes the conjugate transpose of each slice, and
// a tube becomes one complex number per slice.  So, slice by slice:
//   * Tubal-QR (Algorithm 6) of a full-rank n x s block is the thin QR with a positive real
//     diagonal -- unique, whatever algorithm computes it.  It is computed by CholeskyQR2 (Gram
//     matrix, small Cholesky, triangular multiply, twice), which keeps the work in GEMM-shaped
//     passes; slices of a (nearly) rank-deficient block run Algorithm 6's Gram-Schmidt with the
//     Normalize tie-break instead.
//   * The block MGS step H_ij = V_i^H W, W -= V_i H_ij is a tall-skinny Gram and an update.
//   * The projected equation H_m Y - Y B = C1 (Eq. (46)) is solved per slice by Hessenberg-Schur
//     (small_complex.cu) and X += V_m Y.
// Block vectors are stored slice by slice as row-major n x s complex matrices, so that a warp
// reading one row of V reads s contiguous entries: the sparse A_k V product (one warp per row,
// union CSR pattern of all frontal slices, complex values per slice), the Gram and the updates are
// all coalesced.  Norms use Parseval: ||X||^2 = (1/p) sum_k w_k ||X_k||^2, w = 1 for k = 0 and
// k = p/2, 2 otherwise.
#include <algorithm>
#include <cmath>
#include <vector>
#include <type_traits>
#include "internal.cuh"
#include "apply.cuh"
#include "reduce.cuh"
#include "tba.cuh"

namespace ts {
void ensure_f32_operator(ts_op* op, cudaStream_t st);  // lowprec.cu
namespace {

__device__ __forceinline__ double2 cfma(double2 a, double2 b, double2 c) {  // a*b + c
  return make_double2(fma(a.x, b.x, fma(-a.y, b.y, c.x)), fma(a.x, b.y, fma(a.y, b.x, c.y)));
}
__device__ __forceinline__ float2 cfma(float2 a, float2 b, float2 c) {  // a*b + c, FP32
  return make_float2(fmaf(a.x, b.x, fmaf(-a.y, b.y, c.x)), fmaf(a.x, b.y, fmaf(a.y, b.x, c.y)));
}
template <typename C2> struct RealOf;
template <> struct RealOf<double2> { using T = double; };
template <> struct RealOf<float2> { using T = float; };
__device__ __forceinline__ double2 to_c2(double2 v, double2*) { return v; }
__device__ __forceinline__ float2 to_c2(double2 v, float2*) { return make_float2((float)v.x, (float)v.y); }
__device__ __forceinline__ double2 widen(float2 v) { return make_double2(v.x, v.y); }
__device__ __forceinline__ double2 widen(double2 v) { return v; }
__device__ __forceinline__ double slice_weight(int k, int p) {
  return (k == 0 || (p % 2 == 0 && k == p / 2)) ? 1.0 : 2.0;
}

__device__ __forceinline__ double neg(double v) {   // without an FP64 instruction
  return __longlong_as_double(__double_as_longlong(v) ^ (long long)0x8000000000000000ull);
}
__device__ __forceinline__ float neg(float v) { return -v; }

constexpr int kMaxS = 64;           // block width supported by the row kernels

// C2: double2 (FP64), or float2 for the FP32 inner cycle of mixed-precision TBAS (MODE 0 only).
template <typename C2>
struct RowsArgsT {
  const int* rowptr;      // sparse pattern (nullptr: dense A_k column-major in Ad)
  const int* col;
  const C2* vals;         // K x nnz
  const C2* Ad;           // K x n x n column-major (dense operator)
  long long nnz;
  const C2* V;            // K x n x s row-major
  const double2* Brow;    // K x s x s row-major (B_k)
  const double2* C;       // K x n x s row-major (residual mode)
  C2* Out;                // K x n x s row-major
  double* partials;       // residual mode: one per block
  int n, s, K, p;
};
using RowsArgs = RowsArgsT<double2>;

// MODE 0: Out = A_k V_k.  MODE 1: Out = A_k V_k - V_k B_k.  MODE 2: Out = C_k - (A_k V_k - V_k B_k)
// and partials of the Parseval-weighted squared norm.
// Lane layout: LT = 1 (s <= 32): the warp's lanes form groups of sp = s rounded up to a power of two,
// one group per row and one lane per column, so a warp works on 32 / sp rows at once (an idle
// FP64 lane costs as much as a busy one); LT = 2 (32 < s <= 64): one row per warp, two columns per
// lane.
template <int MODE, int LT, typename C2>
__global__ void __launch_bounds__(256) k_sylv_rows(RowsArgsT<C2> a) {
  static_assert(MODE == 0 || sizeof(C2) == 16, "the operator with B_k and the residual run in FP64");
  const int k = blockIdx.y;
  const bool real = k == 0 || (a.p % 2 == 0 && k == a.p / 2);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int sp = 32;
  if (LT == 1)
    while (sp / 2 >= a.s && sp > 1) sp /= 2;
  const int rpw = 32 / sp;                       // rows per warp
  const int sub = lane / sp, jl = lane % sp;
  const long long ns = (long long)a.n * a.s;
  const C2* Vk = a.V + k * ns;
  double local = 0.0;
  const int rows_step = gridDim.x * 8 * rpw;
  for (int ibase = (blockIdx.x * 8 + warp) * rpw; ibase < a.n; ibase += rows_step) {
    const int i = ibase + sub;
    const bool live = i < a.n;
    C2 acc[LT];
#pragma unroll
    for (int t = 0; t < LT; ++t) acc[t] = C2{0, 0};
    if (live) {
      if (real) {   // A_k, V_k and B_k real: one multiply-add of four
        const int q0 = a.rowptr ? a.rowptr[i] : 0, q1 = a.rowptr ? a.rowptr[i + 1] : a.n;
        const C2* vk = a.rowptr ? a.vals + (long long)k * a.nnz : a.Ad + (long long)k * a.n * a.n + i;
        for (int q = q0; q < q1; ++q) {
          const auto av = a.rowptr ? vk[q].x : vk[(long long)q * a.n].x;
          const C2* vr = Vk + (long long)(a.rowptr ? a.col[q] : q) * a.s;
#pragma unroll
          for (int t = 0; t < LT; ++t) {
            const int j = jl + 32 * t;
            if (j < a.s) acc[t].x = fma(av, vr[j].x, acc[t].x);
          }
        }
        if constexpr (MODE >= 1) {
          const double2* Bk = a.Brow + (long long)k * a.s * a.s;
          const double2* xr = Vk + (long long)i * a.s;
          for (int l = 0; l < a.s; ++l) {
            const double nx = neg(xr[l].x);
#pragma unroll
            for (int t = 0; t < LT; ++t) {
              const int j = jl + 32 * t;
              if (j < a.s) acc[t].x = fma(nx, Bk[(long long)l * a.s + j].x, acc[t].x);
            }
          }
        }
      } else if (a.rowptr) {
        const C2* vk = a.vals + (long long)k * a.nnz;
        for (int q = a.rowptr[i]; q < a.rowptr[i + 1]; ++q) {
          const C2 av = vk[q];
          const C2* vr = Vk + (long long)a.col[q] * a.s;
#pragma unroll
          for (int t = 0; t < LT; ++t) {
            const int j = jl + 32 * t;
            if (j < a.s) acc[t] = cfma(av, vr[j], acc[t]);
          }
        }
      } else {
        const C2* Ak = a.Ad + (long long)k * a.n * a.n;
        for (int l = 0; l < a.n; ++l) {
          const C2 av = Ak[(long long)l * a.n + i];
          const C2* vr = Vk + (long long)l * a.s;
#pragma unroll
          for (int t = 0; t < LT; ++t) {
            const int j = jl + 32 * t;
            if (j < a.s) acc[t] = cfma(av, vr[j], acc[t]);
          }
        }
      }
      if constexpr (MODE >= 1) {
        const double2* Bk = a.Brow + (long long)k * a.s * a.s;
        const double2* xr = Vk + (long long)i * a.s;
        for (int l = 0; !real && l < a.s; ++l) {
          const double2 xv = xr[l];
          const double2 nx = make_double2(-xv.x, -xv.y);
#pragma unroll
          for (int t = 0; t < LT; ++t) {
            const int j = jl + 32 * t;
            if (j < a.s) acc[t] = cfma(nx, Bk[(long long)l * a.s + j], acc[t]);
          }
        }
      }
#pragma unroll
      for (int t = 0; t < LT; ++t) {
        const int j = jl + 32 * t;
        if (j < a.s) {
          C2 v = acc[t];
          const long long o = k * ns + (long long)i * a.s + j;
          if constexpr (MODE == 2) {
            const double2 c = a.C[o];
            v = make_double2(c.x - v.x, real ? 0.0 : c.y - v.y);
            local = fma(v.x, v.x, local);
            if (!real) local = fma(v.y, v.y, local);
          }
          a.Out[o] = v;
        }
      }
    }
  }
  if (MODE == 2) {
    const double tot = block_sum(local) * slice_weight(k, a.p) / a.p;
    if (threadIdx.x == 0) a.partials[blockIdx.y * gridDim.x + blockIdx.x] = tot;
  }
}

// A launch's blocks dealt to the K slices: the real ones (k = 0 and, for even p, k = p/2), whose products
// are real, get a third of the blocks of a complex one.  Complex slices come first.
struct SliceParts {
  int K, nyq;
  int kc;        // complex slices k = 1 .. kc
  int nc, nr;    // blocks of a complex / real slice
  __host__ __device__ int blocks() const { return kc * nc + (K - kc) * nr; }
  __device__ __forceinline__ void of(int b, int& k, int& part, int& parts) const {
    if (b < kc * nc) {
      k = 1 + b / nc;
      part = b % nc;
      parts = nc;
    } else {
      b -= kc * nc;
      k = b / nr == 0 ? 0 : nyq;
      part = b % nr;
      parts = nr;
    }
  }
  // first block of slice k
  __device__ __forceinline__ int first(int k) const {
    return k == 0 ? kc * nc : (k == nyq ? kc * nc + nr : (k - 1) * nc);
  }
  __device__ __forceinline__ bool real(int k) const { return k == 0 || k == nyq; }
  __device__ __forceinline__ int parts(int k) const { return real(k) ? nr : nc; }
};
// About `blocks` blocks in all, none with fewer than `min_rows` of the n rows.
SliceParts slice_parts(int K, int nyq, int n, int blocks, int min_rows) {
  SliceParts q{K, nyq, K - 1 - (nyq >= 0 ? 1 : 0), 1, 1};
  const int units = 3 * q.kc + (K - q.kc), most = std::max(1, n / min_rows);
  q.nc = std::max(1, std::min(most, (int)(3.0 * blocks / units)));
  q.nr = std::max(1, std::min(most, (int)((double)blocks / units)));
  return q;
}

// Blocks of an FP32 Gram: a block's rows are added up in FP32 (then in FP64 over the blocks), so a slice has at least
// 2 x 152 / K of them, or one per 64 rows, the real slices too; with a third of a complex slice's blocks their
// chains were 4.6 times as long (n = 16384, p = 8: 1261 rows instead of 274).
SliceParts gram_parts_f32(int K, int nyq, int n, int sms) {
  SliceParts q = slice_parts(K, nyq, n, sms, 32);
  const int least = std::max(1, std::min(2 * sms / K, (n + 63) / 64));
  q.nc = std::max(q.nc, least);
  q.nr = std::max(q.nr, least);
  return q;
}

// Partial Gram matrices G_k = V_k^H W_k over row chunks: partials[block * s*s + a + s*b].
// Gauss's three-multiplication form: with u = conj(v), u w = (T1 - T3) + i (T1 + T2) where
// T1 = sum w_re (u_re + u_im), T2 = sum u_re (w_im - w_re), T3 = sum u_im (w_re + w_im); the sums
// of the factors are formed once per entry while staging, so a complex multiply-add costs three
// FMAs, and one in a real slice.  Each thread owns a 4 x 4 block of G; with HERM (V = W) only the blocks on
// and above the diagonal are formed.  The threads left over form further groups that split the staged
// rows and are summed in a fixed order at the end.
// What bounds it: the FP64 pipe (16 clocks of the SM per warp instruction), so one CTA of eight warps per
// SM saturates it as long as it never waits: the next rows are in registers while the staged ones are
// multiplied, staging is double buffered (one barrier per batch), columns are padded to a multiple of
// 4 only, and blocks are dealt to the slices by their cost.
// Measured (n = 16384, s = 32, p = 8): 546 -> 357 us, with V = W 214 us; s = 4: 205 -> 34 us.
// C2 = float2: FP32 inputs and accumulation over a block's rows (the inner cycle of mixed-precision TBAS; see
// gram_parts_f32); the partial Grams are written in FP64 either way.
constexpr int kGramMaxElems = 4;     // staged elements per thread and operand
struct GramShape {
  int sg, tiles, groups, rb;         // 4-wide column groups, 4 x 4 blocks, row groups, staged rows
  size_t smem;
};
template <typename R>
GramShape gram_shape(int s, bool herm) {
  GramShape g;
  g.sg = (s + 3) / 4;
  g.tiles = herm ? g.sg * (g.sg + 1) / 2 : g.sg * g.sg;
  g.groups = 256 / g.tiles;
  g.rb = (16 + g.groups - 1) / g.groups * g.groups;
  const size_t stage = 2 * 6 * (size_t)g.rb * 4 * g.sg;
  const size_t sum = (size_t)(g.groups - (g.groups + 1) / 2) * g.tiles * 32;
  g.smem = std::max(stage, sum) * sizeof(R);
  TS_REQUIRE(g.rb * 4 * g.sg <= 256 * kGramMaxElems, "gram: block width above kMaxS");
  return g;
}
template <typename C2, bool HERM>
__global__ void __launch_bounds__(256) k_gram(const C2* __restrict__ V, const C2* __restrict__ W, int n, int s,
                                              SliceParts sp, GramShape sh, double2* __restrict__ partials) {
  using R = typename RealOf<C2>::T;
  extern __shared__ unsigned char gram_smem[];
  R* stage = reinterpret_cast<R*>(gram_smem);
  int k, chunk, chunks;
  sp.of(blockIdx.x, k, chunk, chunks);
  const bool real = sp.real(k);
  const int tid = threadIdx.x, cols = 4 * sh.sg, plane = sh.rb * cols;
  const long long ns = (long long)n * s;
  const C2* Vk = V + k * ns;
  const C2* Wk = W + k * ns;
  const int t = tid % sh.tiles, grp = tid / sh.tiles;
  const bool live = grp < sh.groups;
  int ta = t % sh.sg, tb = t / sh.sg;
  if (HERM) {   // t = tb (tb + 1) / 2 + ta, ta <= tb
    tb = 0;
    while ((tb + 1) * (tb + 2) / 2 <= t) ++tb;
    ta = t - tb * (tb + 1) / 2;
  }
  const int a0 = ta * 4, b0 = tb * 4;
  const int rows = (n + chunks - 1) / chunks, r_begin = chunk * rows, r_end = min(n, r_begin + rows);
  C2 v[kGramMaxElems], w[kGramMaxElems];
  auto load = [&](int r0) {
#pragma unroll
    for (int q = 0; q < kGramMaxElems; ++q) {
      const int e = tid + 256 * q, rr = e / cols, cc = e % cols, r = r0 + rr;
      v[q] = w[q] = C2{0, 0};
      if (rr < sh.rb && r < r_end && cc < s) {
        v[q] = Vk[(long long)r * s + cc];
        if (!HERM) w[q] = Wk[(long long)r * s + cc];
      }
    }
  };
  R T1[4][4], T2[4][4], T3[4][4];
#pragma unroll
  for (int x = 0; x < 4; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y) T1[x][y] = T2[x][y] = T3[x][y] = R(0);
  load(r_begin);
  int buf = 0;
  for (int r0 = r_begin; r0 < r_end; r0 += sh.rb, buf ^= 1) {
    // planes: u_re, u_im, u_re + u_im of V; w_re, w_im - w_re, w_re + w_im of W
    R* st = stage + buf * 6 * plane;
#pragma unroll
    for (int q = 0; q < kGramMaxElems; ++q) {
      const int e = tid + 256 * q;
      if (e < plane) {
        const C2 x = v[q], y = HERM ? v[q] : w[q];
        st[e] = x.x;
        st[3 * plane + e] = y.x;
        if (!real) {
          st[plane + e] = neg(x.y);
          st[2 * plane + e] = x.x - x.y;
          st[4 * plane + e] = y.y - y.x;
          st[5 * plane + e] = y.x + y.y;
        }
      }
    }
    __syncthreads();   // also: every thread is done with the other buffer, which the next batch overwrites
    load(r0 + sh.rb);
    if (live) {
      auto vec = [&](const R* p, R (&o)[4]) {
#pragma unroll
        for (int x = 0; x < 4; ++x) o[x] = p[x];
      };
      if (real) {
        for (int rr = grp; rr < sh.rb; rr += sh.groups) {
          R p1[4], q1[4];
          vec(st + rr * cols + a0, p1);
          vec(st + 3 * plane + rr * cols + b0, q1);
#pragma unroll
          for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int y = 0; y < 4; ++y) T1[x][y] = fma(q1[y], p1[x], T1[x][y]);
        }
      } else {
        for (int rr = grp; rr < sh.rb; rr += sh.groups) {
          const R* row = st + rr * cols;
          R p[4], q[4];
          vec(row + 2 * plane + a0, p);
          vec(row + 3 * plane + b0, q);
#pragma unroll
          for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int y = 0; y < 4; ++y) T1[x][y] = fma(q[y], p[x], T1[x][y]);
          vec(row + a0, p);
          vec(row + 4 * plane + b0, q);
#pragma unroll
          for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int y = 0; y < 4; ++y) T2[x][y] = fma(p[x], q[y], T2[x][y]);
          vec(row + plane + a0, p);
          vec(row + 5 * plane + b0, q);
#pragma unroll
          for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int y = 0; y < 4; ++y) T3[x][y] = fma(p[x], q[y], T3[x][y]);
        }
      }
    }
  }
  // combined in R (T1 becomes Re, T2 Im), then the groups are halved until one is left
  if (!real) {
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        const R re = T1[x][y] - T3[x][y];
        T2[x][y] = T1[x][y] + T2[x][y];
        T1[x][y] = re;
      }
  }
  for (int cnt = sh.groups; cnt > 1;) {
    const int half = (cnt + 1) / 2;
    __syncthreads();
    if (live && grp >= half && grp < cnt) {
      R* o = stage + ((grp - half) * sh.tiles + t) * 32;
#pragma unroll
      for (int e = 0; e < 16; ++e) {
        o[(2 * e + t) & 31] = T1[e / 4][e % 4];   // rotated by the block index: the stores spread over the banks
        o[(2 * e + 1 + t) & 31] = T2[e / 4][e % 4];
      }
    }
    __syncthreads();
    if (live && grp < cnt - half) {
      const R* o = stage + (grp * sh.tiles + t) * 32;
#pragma unroll
      for (int e = 0; e < 16; ++e) {
        T1[e / 4][e % 4] += o[(2 * e + t) & 31];
        if (!real) T2[e / 4][e % 4] += o[(2 * e + 1 + t) & 31];
      }
    }
    cnt = half;
  }
  if (live && grp == 0) {
    double2* Pk = partials + (long long)blockIdx.x * s * s;
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        const int i = a0 + x, j = b0 + y;
        if (i < s && j < s) {
          const double re = (double)T1[x][y], im = real ? 0.0 : (double)T2[x][y];
          if (!HERM) {
            Pk[i + s * j] = make_double2(re, im);
          } else if (i <= j) {
            Pk[i + s * j] = make_double2(re, i == j ? 0.0 : im);
            if (i != j) Pk[j + s * i] = make_double2(re, neg(im));
          }
        }
      }
  }
}

// out_k (column-major, leading dimension ldo) = sum over a slice's blocks of the partial Grams, in a fixed
// order: four threads per entry, each every fourth block, then their sums.
__global__ void __launch_bounds__(256) k_gram_reduce(const double2* __restrict__ partials, SliceParts sp, int s,
                                                     double2* __restrict__ out, long long sOut, int ldo) {
  __shared__ double2 red[4][64];
  const int k = blockIdx.y, ss = s * s, sub = threadIdx.x / 64, e = blockIdx.x * 64 + threadIdx.x % 64;
  const int chunks = sp.parts(k);
  const double2* Pk = partials + (long long)sp.first(k) * ss;
  double2 acc = make_double2(0.0, 0.0);
  if (e < ss) {
#pragma unroll 4
    for (int c = sub; c < chunks; c += 4) {
      const double2 v = Pk[(long long)c * ss + e];
      acc.x += v.x;
      acc.y += v.y;
    }
  }
  red[sub][threadIdx.x % 64] = acc;
  __syncthreads();
  if (sub == 0 && e < ss) {
#pragma unroll
    for (int q = 1; q < 4; ++q) {
      const double2 v = red[q][threadIdx.x];
      acc.x += v.x;
      acc.y += v.y;
    }
    out[(long long)k * sOut + (e % s) + (long long)ldo * (e / s)] = acc;
  }
}

// Out_k = (accumulate ? Out_k : 0) + alpha * In_k M_k (in place allowed), M_k an s x s column-major
// block with leading dimension ldm.  NC consecutive columns of one row per thread, all
// threads of a row in one warp; Gauss's form with the planes M_re, M_im - M_re, M_re + M_im of M_k in
// shared memory: Re = T1 - T3, Im = T1 + T2 with T1 = sum (a_re + a_im) m_re, T2 = sum a_re (m_im - m_re),
// T3 = sum a_im (m_re + m_im), three FMAs per complex multiply-add; a real slice (the imaginary parts of
// In and M count as zero) takes one.
// What bounds it: the FP64 pipe; blocks are dealt to the slices by cost and rows to the warps of a slice
// round robin over its blocks, so that the last round is spread over the SMs, and NC matches s (eight
// columns computed for s = 4 were half padding).
// Measured (n = 16384, s = 32, p = 8): 532 -> 359 us; s = 4: 27.6 -> 12.2 us.
// Cin = float2 (the FP32 basis of mixed-precision TBAS): products in FP32; Cout may be double2 (the
// FP64 solution update X += V Y) or float2.
constexpr int kRowCols = 8;
template <int NC, typename Cin, typename Cout>
__global__ void __launch_bounds__(256) k_rows_mm(const Cin* In, Cout* Out, const double2* __restrict__ M,
                                                 long long sM, int ldm, int n, int s, SliceParts sp, double alpha,
                                                 int accumulate) {
  using R = typename RealOf<Cin>::T;
  int k, part, parts;
  sp.of(blockIdx.x, k, part, parts);
  const bool real = sp.real(k);
  extern __shared__ unsigned char smm_raw[];   // three s x s planes, l-major: plane[l * s + j]
  R* mr = reinterpret_cast<R*>(smm_raw);
  R* md = mr + s * s;
  R* mq = mr + 2 * s * s;
  const double2* Mk = M + (long long)k * sM;
  for (int e = threadIdx.x; e < s * s; e += blockDim.x) {
    const int l = e % s, j = e / s;
    const double2 v = Mk[l + (long long)ldm * j];
    mr[l * s + j] = (R)v.x;
    if (!real) {
      md[l * s + j] = (R)(v.y - v.x);
      mq[l * s + j] = (R)(v.x + v.y);
    }
  }
  __syncthreads();
  // Threads per row: a power of two (1, 2, 4, 8), so a row never straddles two warps.
  int tpr = 1;
  while (tpr * kRowCols < s) tpr *= 2;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, rpw = 32 / tpr;
  const int rloc = lane / tpr, c0 = lane % tpr * NC, c1 = min(c0 + NC, s);
  const long long ns = (long long)n * s;
  int col[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) col[c] = max(0, min(c0 + c, s - 1));
  const int step = parts * (int)(blockDim.x / 32) * rpw;
  for (int rbase = (warp * parts + part) * rpw; rbase < n; rbase += step) {
    const int i = rbase + rloc;
    const bool live = i < n;
    R T1[NC], T2[NC], T3[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) T1[c] = T2[c] = T3[c] = R(0);
    const long long ro = k * ns + (long long)i * s;
    if (live) {
      if (real) {
#pragma unroll 4
        for (int l = 0; l < s; ++l) {
          const R ar = In[ro + l].x;
#pragma unroll
          for (int c = 0; c < NC; ++c) T1[c] = fma(ar, mr[l * s + col[c]], T1[c]);
        }
      } else {
#pragma unroll 4
        for (int l = 0; l < s; ++l) {
          const Cin a = In[ro + l];
          const R sa = a.x + a.y;
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            T1[c] = fma(sa, mr[l * s + col[c]], T1[c]);
            T2[c] = fma(a.x, md[l * s + col[c]], T2[c]);
            T3[c] = fma(a.y, mq[l * s + col[c]], T3[c]);
          }
        }
      }
    }
    __syncwarp();   // every thread of the row has read In before any writes Out (in place)
    if (live) {
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const int j = c0 + c;
        if (j < c1) {
          // FP32 products are scaled in FP32 and converted at most once, since GB300's FP64 and
          // conversion rate would otherwise make this epilogue cost more than the s-term loop
          const R al = (R)alpha;
          R vr = al * (T1[c] - T3[c]), vi = real ? R(0) : al * (T1[c] + T2[c]);
          if constexpr (sizeof(Cout) == sizeof(Cin)) {
            if (accumulate) {
              const Cout o = Out[ro + j];
              vr += o.x;
              if (!real) vi += o.y;
            }
            Out[ro + j] = Cout{vr, vi};
          } else {
            double2 v = make_double2((double)vr, (double)vi);
            if (accumulate) {
              const double2 o = widen(Out[ro + j]);
              v.x += o.x;
              if (!real) v.y += o.y;
            }
            Out[ro + j] = to_c2(v, (Cout*)nullptr);
          }
        }
      }
    }
  }
}

// Algorithm 6 with Normalization1 on the Fourier slices whose first Cholesky pivot showed a (nearly)
// rank-deficient block (fail[k] = 1; other slices return at once): modified Gram-Schmidt over the s
// columns of W_k (row-major n x s, in place -> Q_k), r_ij = q_i^H w_j, w_j -= q_i r_ij, then
// a = ||w_j||.  Column j counts as zero in this slice when a <= tiny * ref_j, ref_j the largest norm of
// column j over all K slices before orthogonalisation (the square root of max_k G_k(j, j), G the Gram
// of the original block); then r_jj = 0 and q_j is the first unit vector e_i whose component
// orthogonal to q_0..q_{j-1} has squared norm >= 1/(2n), orthogonalised twice (classical
// Gram-Schmidt) and normalised.  Writes R_k (upper triangular, column-major) to R and the identity to
// Rinv, so the CholeskyQR2 steps that follow leave the slice as it is.  One CTA per slice; rows are
// strided over the threads (each thread only reads back the rows it wrote, so the block reductions
// are the only synchronisation needed).  A fallback for rare blocks: columns are read with stride s.
template <typename C2>
__global__ void __launch_bounds__(256) k_tubal_mgs(C2* __restrict__ W, const double2* __restrict__ G,
                                                   const int* __restrict__ fail, double2* __restrict__ R,
                                                   double2* __restrict__ Rinv, int n, int s, int K, double tiny) {
  const int k = blockIdx.x;
  if (!fail[k]) return;
  __shared__ double2 coef[kMaxS];
  const long long ns = (long long)n * s;
  C2* Wk = W + k * ns;
  double2* Rk = R + (long long)k * s * s;
  double2* Ik = Rinv + (long long)k * s * s;
  for (int e = threadIdx.x; e < s * s; e += blockDim.x) {
    Rk[e] = make_double2(0.0, 0.0);
    Ik[e] = make_double2(e % s == e / s ? 1.0 : 0.0, 0.0);
  }
  __syncthreads();
  auto ld = [&](int r, int c) { return widen(Wk[(long long)r * s + c]); };
  auto st = [&](int r, int c, double2 v) { Wk[(long long)r * s + c] = to_c2(v, (C2*)nullptr); };
  for (int j = 0; j < s; ++j) {
    double ref2 = 0.0;
    for (int q = 0; q < K; ++q) ref2 = fmax(ref2, G[(long long)q * s * s + j + (long long)s * j].x);
    for (int i = 0; i < j; ++i) {                       // r_ij = q_i^H w_j; w_j -= q_i r_ij
      double re = 0.0, im = 0.0;
      for (int r = threadIdx.x; r < n; r += blockDim.x) {
        const double2 q = ld(r, i), w = ld(r, j);
        re += q.x * w.x + q.y * w.y;
        im += q.x * w.y - q.y * w.x;
      }
      re = block_sum(re);
      im = block_sum(im);
      for (int r = threadIdx.x; r < n; r += blockDim.x) {
        const double2 q = ld(r, i), w = ld(r, j);
        st(r, j, make_double2(w.x - (q.x * re - q.y * im), w.y - (q.x * im + q.y * re)));
      }
      if (threadIdx.x == 0) Rk[i + (long long)s * j] = make_double2(re, im);
    }
    double a2 = 0.0;
    for (int r = threadIdx.x; r < n; r += blockDim.x) {
      const double2 w = ld(r, j);
      a2 += w.x * w.x + w.y * w.y;
    }
    const double a = sqrt(block_sum(a2));
    if (a > tiny * sqrt(ref2)) {                        // Normalize: q_j = w_j / a, r_jj = a
      const double inv = 1.0 / a;
      for (int r = threadIdx.x; r < n; r += blockDim.x) {
        const double2 w = ld(r, j);
        st(r, j, make_double2(w.x * inv, w.y * inv));
      }
      if (threadIdx.x == 0) Rk[j + (long long)s * j] = make_double2(a, 0.0);
      continue;
    }
    // rank-deficient slice of column j: r_jj = 0 (already), q_j = a unit vector orthogonal to q_<j
    for (int e = 0; e < n; ++e) {
      for (int r = threadIdx.x; r < n; r += blockDim.x) st(r, j, make_double2(r == e ? 1.0 : 0.0, 0.0));
      for (int pass = 0; pass < 2; ++pass) {
        for (int i = 0; i < j; ++i) {                   // c_i = q_i^H z for every i first (classical)
          double re = 0.0, im = 0.0;
          for (int r = threadIdx.x; r < n; r += blockDim.x) {
            const double2 q = ld(r, i), z = ld(r, j);
            re += q.x * z.x + q.y * z.y;
            im += q.x * z.y - q.y * z.x;
          }
          re = block_sum(re);
          im = block_sum(im);
          if (threadIdx.x == 0) coef[i] = make_double2(re, im);
        }
        __syncthreads();
        for (int r = threadIdx.x; r < n; r += blockDim.x) {
          double2 z = ld(r, j);
          for (int i = 0; i < j; ++i) {
            const double2 q = ld(r, i), c = coef[i];
            z.x -= q.x * c.x - q.y * c.y;
            z.y -= q.x * c.y + q.y * c.x;
          }
          st(r, j, z);
        }
        __syncthreads();                                // coef is rewritten by the next pass
      }
      double z2 = 0.0;
      for (int r = threadIdx.x; r < n; r += blockDim.x) {
        const double2 z = ld(r, j);
        z2 += z.x * z.x + z.y * z.y;
      }
      z2 = block_sum(z2);
      if (z2 >= 0.5 / n) {
        const double inv = 1.0 / sqrt(z2);
        for (int r = threadIdx.x; r < n; r += blockDim.x) {
          const double2 z = ld(r, j);
          st(r, j, make_double2(z.x * inv, z.y * inv));
        }
        break;
      }
    }
  }
}

// Column-major spectral [k][j][i] <-> row-major [k][i][j], 32 x 32 tiles.
__global__ void k_spec_transpose(const double2* __restrict__ in, double2* __restrict__ out, int rows, int cols) {
  // in: K x (cols x rows) with rows fastest; out: K x (rows x cols) with cols fastest
  __shared__ double2 tile[32][33];
  const int k = blockIdx.z;
  const long long off = (long long)k * rows * cols;
  const int r0 = blockIdx.x * 32, c0 = blockIdx.y * 32;
  for (int q = threadIdx.y; q < 32; q += blockDim.y) {
    const int r = r0 + threadIdx.x, c = c0 + q;
    if (r < rows && c < cols) tile[q][threadIdx.x] = in[off + (long long)c * rows + r];
  }
  __syncthreads();
  for (int q = threadIdx.y; q < 32; q += blockDim.y) {
    const int r = r0 + q, c = c0 + threadIdx.x;
    if (r < rows && c < cols) out[off + (long long)r * cols + c] = tile[threadIdx.x][q];
  }
}

// sum_k w_k/p * (squared Frobenius norm of the s x s block k of E) -> out[0]; traces of G -> out.
__global__ void k_weighted_fro(const double2* __restrict__ E, int s, int K, int p, double* out) {
  double local = 0.0;
  for (int e = threadIdx.x; e < K * s * s; e += blockDim.x) {
    const int k = e / (s * s);
    const double2 v = E[e];
    local += (v.x * v.x + v.y * v.y) * slice_weight(k, p) / p;
  }
  const double tot = block_sum(local);
  if (threadIdx.x == 0) out[0] = tot;
}

__global__ void k_weighted_trace(const double2* __restrict__ G, int s, int K, int p, double* out) {
  double local = 0.0;
  for (int e = threadIdx.x; e < K * s; e += blockDim.x) {
    const int k = e / s, d = e % s;
    local += G[(long long)k * s * s + d + (long long)s * d].x * slice_weight(k, p) / p;
  }
  const double tot = block_sum(local);
  if (threadIdx.x == 0) out[0] = tot;
}

__global__ void k_fill_c1(const double2* __restrict__ H0, double2* __restrict__ C1, int s, int N, int K) {
  // C1_k = [H0_k; 0] (N x s column-major)
  const long long tot = (long long)K * N * s;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < tot; e += (long long)gridDim.x * blockDim.x) {
    const int k = (int)(e / ((long long)N * s));
    const long long r = e % ((long long)N * s);
    const int i = (int)(r % N), j = (int)(r / N);
    C1[e] = i < s ? H0[(long long)k * s * s + i + (long long)s * j] : make_double2(0.0, 0.0);
  }
}

// B_k (column-major) -> row-major copy.
__global__ void k_row_major_small(const double2* __restrict__ B, double2* __restrict__ Br, int s, int K) {
  const long long tot = (long long)K * s * s;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < tot; e += (long long)gridDim.x * blockDim.x) {
    const int k = (int)(e / ((long long)s * s));
    const long long r = e % ((long long)s * s);
    const int row = (int)(r / s), colj = (int)(r % s);
    Br[e] = B[(long long)k * s * s + row + (long long)s * colj];
  }
}

int grid1d(long long work) {
  long long g = (work + 255) / 256;
  if (g > 152 * 8) g = 152 * 8;
  return (int)(g < 1 ? 1 : g);
}

struct TbaWork {
  int n, s, p, K, m;
  long long blk;            // K * n * s
  double2* V;               // (m + 1) blocks
  double2* X;               // spectral X, row-major
  double2* C;               // spectral C, row-major
  double2* R;               // spectral residual
  double2* tmp;             // column-major spectral scratch
  double2* Hm;              // K x (ms x ms) column-major
  double2* H0;              // K x s x s
  double2* Hlast;           // K x s x s
  double2* G;               // K x s x s (Gram / Cholesky scratch)
  double2* R1;              // K x s x s
  double2* Rinv;            // K x s x s
  double2* R2;              // K x s x s
  double2* gram_part;       // partial Grams
  SliceParts gram_parts, gram_parts32, row_parts;   // blocks of the Gram (FP64, FP32) and row products
  double2* LU;              // K x s x N x N
  int* piv;                 // K x s x N
  double2* Gp;              // K x N x s
  double2* Z;               // K x N x s
  double2* Y;               // K x N x s
  double2* E;               // K x s x s
  double* P;                // kRedBlocks partials
  double* sc;               // scalars
  int* err;                 // error bits
  int* fail;                // K flags: slices whose Tubal-QR took the Gram-Schmidt fallback
  KernelTimer* tm;          // per-kernel timing (kind 4: tubal Gram and block products)
};

}  // namespace

void SparseOp::release() {
  op_free(rowptr);
  op_free(col);
  op_free(vals);
  op_free(vals32);
  rowptr = col = nullptr;
  vals = nullptr;
  vals32 = nullptr;
}

void ensure_b_schur(ts_ctx* ctx, ts_op* op, cudaStream_t st) {
  if (op->schurT) return;
  const int s = op->s, K = op->K;
  op_alloc(op->schurT, sizeof(double2) * (size_t)K * s * s);
  op_alloc(op->schurQ, sizeof(double2) * (size_t)K * s * s);
  TS_CUDA(cudaMemcpyAsync(op->schurT, op->Bh, sizeof(double2) * (size_t)K * s * s, cudaMemcpyDeviceToDevice, st));
  int* err = static_cast<int*>(ctx->ws.get("schur_err", sizeof(int)));
  TS_CUDA(cudaMemsetAsync(err, 0, sizeof(int), st));
  schur_small(op->schurT, op->schurQ, s, K, err, st);
  int e = 0;
  TS_CUDA(cudaMemcpyAsync(&e, err, sizeof(int), cudaMemcpyDeviceToHost, st));
  TS_CUDA(cudaStreamSynchronize(st));
  if (e) {
    op_free(op->schurT);
    op_free(op->schurQ);
    op->schurT = op->schurQ = nullptr;
    throw Error{TS_SINGULAR, "complex Schur iteration of B_k did not converge"};
  }
}

namespace {

// W = A_k V_k in FP32 (the inner cycle of mixed-precision TBAS); FP32 copies of the operator's
// values are made on first use.
void rows_call_f32(ts_op* op, const float2* V, float2* Out, int n, int s, int K, int p, cudaStream_t st) {
  RowsArgsT<float2> a{};
  if (op->sp) {
    SparseOp& sp = *op->sp;
    if (!sp.vals32) {
      op_alloc(sp.vals32, sizeof(float2) * (size_t)K * sp.nnz);
      convert<double, float>(reinterpret_cast<const double*>(sp.vals), reinterpret_cast<float*>(sp.vals32),
                             2ll * K * sp.nnz, st);
    }
    a.rowptr = sp.rowptr;
    a.col = sp.col;
    a.vals = sp.vals32;
    a.nnz = sp.nnz;
  } else {
    ensure_f32_operator(op, st);
    a.Ad = op->Ah32;
  }
  a.V = V;
  a.Out = Out;
  a.n = n;
  a.s = s;
  a.K = K;
  a.p = p;
  const bool wide = s > 32;
  int sp = 32;
  while (!wide && sp / 2 >= s && sp > 1) sp /= 2;
  const int rows_per_block = 8 * (32 / sp);
  const int gx = std::max(1, std::min((n + rows_per_block - 1) / rows_per_block, 2 * 152 * 4 / K));
  if (wide) k_sylv_rows<0, 2><<<dim3(gx, K), 256, 0, st>>>(a);
  else k_sylv_rows<0, 1><<<dim3(gx, K), 256, 0, st>>>(a);
  count_launch();
  TS_CUDA(cudaGetLastError());
}

void rows_call(int mode, const ts_op* op, const double2* V, const double2* C, double2* Out, double* partials, int n,
               int s, int K, int p, cudaStream_t st) {
  RowsArgs a{};
  if (op->sp) {
    a.rowptr = op->sp->rowptr;
    a.col = op->sp->col;
    a.vals = op->sp->vals;
    a.nnz = op->sp->nnz;
  } else {
    a.Ad = op->Ah;
  }
  a.V = V;
  a.Brow = op->Bh_row;
  a.C = C;
  a.Out = Out;
  a.partials = partials;
  a.n = n;
  a.s = s;
  a.K = K;
  a.p = p;
  const bool wide = s > 32;
  int sp = 32;
  while (!wide && sp / 2 >= s && sp > 1) sp /= 2;
  const int rows_per_block = 8 * (32 / sp);
#define TS_SYLV_ROWS(M, GX)                                                           \
  do {                                                                                \
    if (wide) k_sylv_rows<M, 2><<<dim3((GX), K), 256, 0, st>>>(a);                    \
    else k_sylv_rows<M, 1><<<dim3((GX), K), 256, 0, st>>>(a);                         \
  } while (0)
  if (mode == 2) {
    const int gx = kRedBlocks / K;
    TS_CUDA(cudaMemsetAsync(partials, 0, sizeof(double) * kRedBlocks, st));
    TS_SYLV_ROWS(2, gx);
  } else {
    const int gx = std::max(1, std::min((n + rows_per_block - 1) / rows_per_block, 2 * 152 * 4 / K));
    if (mode == 0) TS_SYLV_ROWS(0, gx);
    else TS_SYLV_ROWS(1, gx);
  }
#undef TS_SYLV_ROWS
  count_launch();
  TS_CUDA(cudaGetLastError());
}

template <typename Cin, typename Cout>
void rows_mm(const TbaWork& w, const Cin* In, Cout* Out, const double2* M, long long sM, int ldm, double alpha,
             bool accumulate, cudaStream_t st) {
  using R = typename RealOf<Cin>::T;
  const int s = w.s;
  TS_REQUIRE(s <= kMaxS, "rows_mm: block width above kMaxS");
  int tpr = 1;
  while (tpr * kRowCols < s) tpr *= 2;
  const size_t smem = sizeof(R) * 3 * (size_t)s * s;
  auto run = [&](auto nc) {
    constexpr int NC = decltype(nc)::value;
    set_max_dynamic_smem((const void*)k_rows_mm<NC, Cin, Cout>, (int)(sizeof(R) * 3 * kMaxS * kMaxS));
    k_rows_mm<NC, Cin, Cout><<<w.row_parts.blocks(), 256, smem, st>>>(In, Out, M, sM, ldm, w.n, s, w.row_parts, alpha,
                                                                      accumulate ? 1 : 0);
  };
  switch ((s + tpr - 1) / tpr) {   // columns per thread
    case 1: run(std::integral_constant<int, 1>{}); break;
    case 2: run(std::integral_constant<int, 2>{}); break;
    case 3: run(std::integral_constant<int, 3>{}); break;
    case 4: run(std::integral_constant<int, 4>{}); break;
    case 5: run(std::integral_constant<int, 5>{}); break;
    case 6: run(std::integral_constant<int, 6>{}); break;
    case 7: run(std::integral_constant<int, 7>{}); break;
    default: run(std::integral_constant<int, 8>{}); break;
  }
  count_launch();
  TS_CUDA(cudaGetLastError());
}

// Algorithmic FLOPs of one (n x s)^H (n x s) or (n x s)(s x s) complex product over K slices.
double block_flops(const TbaWork& w) { return 8.0 * w.n * w.s * w.s * w.K; }

template <typename C2>
void gram(const TbaWork& w, const C2* V, const C2* W, double2* out, long long sOut, int ldo, cudaStream_t st) {
  w.tm->begin(st, 4, block_flops(w));
  const SliceParts& parts = sizeof(C2) == 16 ? w.gram_parts : w.gram_parts32;
  auto run = [&](auto herm) {
    constexpr bool HERM = decltype(herm)::value;
    const GramShape g = gram_shape<typename RealOf<C2>::T>(w.s, HERM);
    set_max_dynamic_smem((const void*)k_gram<C2, HERM>, (int)g.smem);
    k_gram<C2, HERM><<<parts.blocks(), 256, g.smem, st>>>(V, W, w.n, w.s, parts, g, w.gram_part);
  };
  if (V == W) run(std::true_type{});
  else run(std::false_type{});
  count_launch();
  TS_CUDA(cudaGetLastError());
  k_gram_reduce<<<dim3((w.s * w.s + 63) / 64, w.K), 256, 0, st>>>(w.gram_part, parts, w.s, out, sOut, ldo);
  count_launch();
  TS_CUDA(cudaGetLastError());
  w.tm->end(st);
}

template <typename Cin, typename Cout>
void rows_mm_timed(const TbaWork& w, const Cin* In, Cout* Out, const double2* M, long long sM, int ldm,
                   double alpha, bool accumulate, cudaStream_t st) {
  w.tm->begin(st, 4, block_flops(w));
  rows_mm(w, In, Out, M, sM, ldm, alpha, accumulate, st);
  w.tm->end(st);
}

// Tubal-QR of the block W (in place -> Q); R written to Rout (column-major, ldr).  Per Fourier slice
// the QR with a positive real diagonal is unique for a full-rank block, and CholeskyQR2 computes it
// in GEMM-shaped passes: G = W^H W, G = R1^H R1, W <- W R1^-1, again with R2, R = R2 R1.  A slice
// whose first Cholesky pivot says that a column is (nearly) dependent on the previous ones -- its
// orthogonal part below 1e-6 of its norm in FP64 (1e-3 in FP32), or its norm below the rank-deficiency
// scale of Normalization1 -- takes Algorithm 6 itself instead (k_tubal_mgs: Gram-Schmidt with the
// Normalize tie-break), whose Q the second CholeskyQR pass then only re-orthogonalises to rounding.
// Returns false when the second Cholesky fails (not expected after either first pass).  have_gram: w.G
// already holds W^H W.
template <typename C2>
bool tubal_qr(const TbaWork& w, C2* W, double2* Rout, long long sR, int ldr, bool have_gram, cudaStream_t st) {
  const int s = w.s, K = w.K;
  const long long ss = (long long)s * s;
  constexpr bool f64 = sizeof(C2) == 16;
  const double tiny = f64 ? 1e-12 : 1e-4;      // Normalization1: a slice is zero below tiny * ref_j
  const double rel = f64 ? 1e-12 : 1e-6;       // CholeskyQR is trusted for orthogonal parts above sqrt(rel)
  TS_CUDA(cudaMemsetAsync(w.err, 0, sizeof(int), st));
  if (!have_gram) gram(w, W, W, w.G, ss, s, st);
  cholesky_inverse(w.G, w.R1, w.Rinv, s, K, rel, tiny * tiny, nullptr, w.fail, st);
  k_tubal_mgs<C2><<<K, 256, 0, st>>>(W, w.G, w.fail, w.R1, w.Rinv, w.n, s, K, tiny);
  count_launch();
  TS_CUDA(cudaGetLastError());
  rows_mm_timed(w, W, W, w.Rinv, ss, s, 1.0, false, st);
  gram(w, W, W, w.G, ss, s, st);
  cholesky_inverse(w.G, w.R2, w.Rinv, s, K, 0.0, 0.0, w.err, nullptr, st);
  rows_mm_timed(w, W, W, w.Rinv, ss, s, 1.0, false, st);
  small_gemm(w.R2, ss, s, w.R1, ss, s, false, Rout, sR, ldr, s, s, s, K, false, st);   // R = R2 R1
  int e = 0;
  TS_CUDA(cudaMemcpyAsync(&e, w.err, sizeof(int), cudaMemcpyDeviceToHost, st));
  TS_CUDA(cudaStreamSynchronize(st));
  return e == 0;
}

double read_scalar(const double* d, ts_ctx* ctx, cudaStream_t st) {
  TS_CUDA(cudaMemcpyAsync(ctx->host_scalars + 32, d, sizeof(double), cudaMemcpyDeviceToHost, st));
  TS_CUDA(cudaStreamSynchronize(st));
  return ctx->host_scalars[32];
}

double weighted_trace(const TbaWork& w, const double2* G, ts_ctx* ctx, cudaStream_t st) {
  k_weighted_trace<<<1, 256, 0, st>>>(G, w.s, w.K, w.p, w.sc);
  count_launch();
  TS_CUDA(cudaGetLastError());
  return read_scalar(w.sc, ctx, st);
}

// R = C - M(X) in the spectral row-major layout; returns ||R||_F (real space).
double residual(ts_ctx* ctx, const ts_op* op, const TbaWork& w, cudaStream_t st) {
  rows_call(2, op, w.X, w.C, w.R, w.P, w.n, w.s, w.K, w.p, st);
  finalize_norm(w.P, w.sc, st);
  return read_scalar(w.sc, ctx, st);
}

void to_rows(const double* real, double2* spec_rows, double2* tmp, int n, int s, int p, cudaStream_t st) {
  const int K = num_slices(p);
  rfft_tube<double, double2>(real, tmp, (long long)n * s, p, st);
  k_spec_transpose<<<dim3((n + 31) / 32, (s + 31) / 32, K), dim3(32, 8), 0, st>>>(tmp, spec_rows, n, s);
  count_launch();
  TS_CUDA(cudaGetLastError());
}

void from_rows(const double2* spec_rows, double* real, double2* tmp, int n, int s, int p, cudaStream_t st) {
  const int K = num_slices(p);
  // row-major (n x s) is column-major (s x n): transpose with rows = s, cols = n
  k_spec_transpose<<<dim3((s + 31) / 32, (n + 31) / 32, K), dim3(32, 8), 0, st>>>(spec_rows, tmp, s, n);
  count_launch();
  TS_CUDA(cudaGetLastError());
  irfft_tube<double, double2>(tmp, real, (long long)n * s, p, IRFFT_STORE, nullptr, nullptr, st);
}

void ensure_brow(ts_op* op, cudaStream_t st) {
  if (op->Bh_row) return;
  const size_t b = sizeof(double2) * (size_t)op->K * op->s * op->s;
  op_alloc(op->Bh_row, b);
  k_row_major_small<<<grid1d((long long)op->K * op->s * op->s), 256, 0, st>>>(op->Bh, op->Bh_row, op->s, op->K);
  count_launch();
  TS_CUDA(cudaGetLastError());
}

TbaWork tba_work(ts_ctx* ctx, const ts_op* op, int m) {
  TbaWork w{};
  w.n = op->n; w.s = op->s; w.p = op->p; w.K = op->K; w.m = m;
  const int n = w.n, s = w.s, K = w.K, N = m * s;
  w.blk = (long long)K * n * s;
  const size_t blk = sizeof(double2) * (size_t)w.blk, ss = sizeof(double2) * (size_t)K * s * s;
  auto get = [&](const char* name, size_t bytes) { return ctx->ws.get(name, bytes); };
  w.V = (double2*)get("tba_V", blk * (m + 1));
  w.X = (double2*)get("tba_X", blk);
  w.C = (double2*)get("tba_C", blk);
  w.R = (double2*)get("tba_R", blk);
  w.tmp = (double2*)get("tba_tmp", blk);
  w.Hm = (double2*)get("tba_Hm", sizeof(double2) * (size_t)K * N * N);
  w.H0 = (double2*)get("tba_H0", ss);
  w.Hlast = (double2*)get("tba_Hlast", ss);
  w.G = (double2*)get("tba_G", ss);
  w.R1 = (double2*)get("tba_R1", ss);
  w.R2 = (double2*)get("tba_R2", ss);
  w.Rinv = (double2*)get("tba_Rinv", ss);
  const int nyq = nyquist_index(w.p);
  w.gram_parts = slice_parts(K, nyq, n, ctx->num_sms, 32);
  w.gram_parts32 = gram_parts_f32(K, nyq, n, ctx->num_sms);
  w.row_parts = slice_parts(K, nyq, n, 2 * ctx->num_sms, 32);
  w.gram_part = (double2*)get("tba_gram_part", sizeof(double2) * s * s *
                                                   (size_t)std::max(w.gram_parts.blocks(), w.gram_parts32.blocks()));
  w.LU = (double2*)get("tba_LU", sizeof(double2) * (size_t)K * s * N * N);
  w.piv = (int*)get("tba_piv", sizeof(int) * (size_t)K * s * N);
  w.Gp = (double2*)get("tba_Gp", sizeof(double2) * (size_t)K * N * s);
  w.Z = (double2*)get("tba_Z", sizeof(double2) * (size_t)K * N * s);
  w.Y = (double2*)get("tba_Y", sizeof(double2) * (size_t)K * N * s);
  w.E = (double2*)get("tba_E", ss);
  w.P = (double*)get("tba_P", sizeof(double) * kRedBlocks);
  w.sc = (double*)get("tba_sc", sizeof(double) * 16);
  w.err = (int*)get("tba_err", sizeof(int) * 4);
  w.fail = (int*)get("tba_fail", sizeof(int) * (size_t)K);
  w.tm = &ctx->timer;
  return w;
}

ts_status tbas_solve(ts_ctx* ctx, ts_op* op, const double* C, double* X, const ts_solve_opts& o, ts_solve_info& info,
                     cudaStream_t st) {
  const int n = op->n, s = op->s, p = op->p, K = op->K, m = o.restart;
  TS_REQUIRE(s <= kMaxS, "ts_tba_solve: block width s must be <= 64");
  TS_REQUIRE((long long)m * s <= 12000, "ts_tba_solve: m*s too large for the projected solve");
  ensure_brow(op, st);
  ensure_b_schur(ctx, op, st);
  TbaWork w = tba_work(ctx, op, m);
  const long long ss = (long long)s * s;
  int hist_len = 0, true_len = 0;
  auto push_hist = [&](double v) {
    if (o.history && hist_len < o.history_cap) o.history[hist_len] = v;
    ++hist_len;
  };
  auto push_true = [&](double v) {
    if (o.true_history && true_len < o.true_history_cap) o.true_history[true_len] = v;
    ++true_len;
  };
  to_rows(C, w.C, w.tmp, n, s, p, st);
  to_rows(X, w.X, w.tmp, n, s, p, st);
  // ||C||^2 = (1/p) sum_k w_k trace(C_k^H C_k)  (Parseval)
  gram(w, w.C, w.C, w.G, ss, s, st);
  const double normC = std::sqrt(std::max(0.0, weighted_trace(w, w.G, ctx, st)));
  double res = residual(ctx, op, w, st);
  info.normC = normC;
  info.applies_fp64 = 1;
  push_true(res);
  double last_est = res;
  auto finish = [&](ts_status stt) {
    from_rows(w.X, X, w.tmp, n, s, p, st);
    TS_CUDA(cudaStreamSynchronize(st));
    info.history_len = hist_len;
    info.true_history_len = true_len;
    if (o.precision == TS_MIXED_FP32) info.outer = info.cycles;
    info.relres_true = normC > 0 ? res / normC : res;
    info.relres_est = normC > 0 ? last_est / normC : last_est;
    return stt;
  };
  if (!std::isfinite(res) || !std::isfinite(normC)) return finish(TS_ERR_NONFINITE);
  if (normC == 0.0 || res <= o.tol * normC) return finish(TS_OK);
  const long long blk = w.blk;
  // Mixed precision (TS_MIXED_FP32): the block Krylov basis, the SpMM and the block products of each
  // cycle run in FP32; the Gram results, H_m, the projected solve, X and the true residual of every
  // restart stay FP64, so the restarts are steps of iterative refinement.
  const bool low = o.precision == TS_MIXED_FP32;
  float2* V32 = low ? (float2*)ctx->ws.get("tba_V32", sizeof(float2) * (size_t)blk * (m + 1)) : nullptr;
  const double breakdown_rel = low ? 1e-6 : 1e-13;
  // Work of one A V_j product over all K slices: the kernel forms 8 FLOPs per stored complex value
  // and block column (dense A: n^2 values per slice); algorithmically it reads the values, the
  // pattern and V once and writes W once.
  const double a_vals = op->sp ? (double)op->sp->nnz : (double)n * n;
  const double spmm_flops = 8.0 * a_vals * s * K;
  auto spmm_bytes = [&](size_t c2) {
    return (double)K * a_vals * c2 + (op->sp ? 4.0 * (a_vals + n + 1) : 0.0) + 2.0 * (double)K * n * s * c2;
  };
  for (int cycle = 0; cycle < o.max_restarts; ++cycle) {
    const int N = m * s;
    int mm = m;
    // One Tubal Block Arnoldi cycle on the basis V (double2 or float2): V_1 = Tubal-QR(R0), W = A V_j,
    // block MGS, Tubal-QR of W.  Returns false on a failed Tubal-QR.
    auto arnoldi = [&](auto* V) -> bool {
      using C2 = std::remove_pointer_t<decltype(V)>;
      if constexpr (sizeof(C2) == 16) {
        TS_CUDA(cudaMemcpyAsync(V, w.R, sizeof(double2) * blk, cudaMemcpyDeviceToDevice, st));
      } else {
        convert<double, float>(reinterpret_cast<const double*>(w.R), reinterpret_cast<float*>(V), 2 * blk, st);
      }
      if (!tubal_qr(w, V, w.H0, ss, s, false, st)) return false;
      TS_CUDA(cudaMemsetAsync(w.Hm, 0, sizeof(double2) * (size_t)K * N * N, st));
      for (int j = 0; j < m; ++j) {
        C2* Vj = V + (long long)j * blk;
        C2* Wb = V + (long long)(j + 1) * blk;
        w.tm->begin(st, 5, spmm_flops, spmm_bytes(sizeof(C2)));
        if constexpr (sizeof(C2) == 16) {
          rows_call(0, op, Vj, nullptr, Wb, nullptr, n, s, K, p, st);          // W = A * V_j (A, not M)
          ++info.applies_fp64;
        } else {
          rows_call_f32(op, Vj, Wb, n, s, K, p, st);
          ++info.applies_low;
        }
        w.tm->end(st);
        for (int i = 0; i <= j; ++i) {                                          // block MGS
          C2* Vi = V + (long long)i * blk;
          double2* Hij = w.Hm + (long long)i * s + (long long)N * j * s;       // block (i, j) of H_m
          gram(w, Vi, Wb, Hij, (long long)N * N, N, st);
          rows_mm_timed(w, Vi, Wb, Hij, (long long)N * N, N, -1.0, true, st);
        }
        gram(w, Wb, Wb, w.G, ss, s, st);
        const double wn = std::sqrt(std::max(0.0, weighted_trace(w, w.G, ctx, st)));
        ++info.iters;
        if (wn <= breakdown_rel * res) {                                        // block breakdown
          mm = j + 1;
          TS_CUDA(cudaMemsetAsync(w.Hlast, 0, sizeof(double2) * (size_t)K * ss, st));
          break;
        }
        double2* Hnext = (j + 1 < m) ? w.Hm + (long long)(j + 1) * s + (long long)N * j * s : w.Hlast;
        const long long sH = (j + 1 < m) ? (long long)N * N : ss;
        const int ldh = (j + 1 < m) ? N : s;
        if (!tubal_qr(w, Wb, Hnext, sH, ldh, true, st)) return false;   // w.G is still W^H W
      }
      return true;
    };
    if (!(low ? arnoldi(V32) : arnoldi(w.V))) return finish(TS_BREAKDOWN);
    const int Nm = mm * s;
    // Projected equation per slice: H_m Y - Y B = C1 = [H0; 0] by Hessenberg-Schur.
    // When the block space broke down early the leading Nm x Nm part of H_m is used.
    double2* Hproj = w.Hm;
    long long sHp = (long long)N * N;
    if (Nm != N) {
      double2* Hc = (double2*)ctx->ws.get("tba_Hcompact", sizeof(double2) * (size_t)K * Nm * Nm);
      for (int k = 0; k < K; ++k)
        TS_CUDA(cudaMemcpy2DAsync(Hc + (long long)k * Nm * Nm, sizeof(double2) * Nm, w.Hm + (long long)k * N * N,
                                  sizeof(double2) * N, sizeof(double2) * Nm, Nm, cudaMemcpyDeviceToDevice, st));
      Hproj = Hc;
      sHp = (long long)Nm * Nm;
    }
    k_fill_c1<<<grid1d((long long)K * Nm * s), 256, 0, st>>>(w.H0, w.Z, s, Nm, K);     // Z <- C1
    count_launch();
    TS_CUDA(cudaGetLastError());
    small_gemm(w.Z, (long long)Nm * s, Nm, op->schurQ, ss, s, false, w.Gp, (long long)Nm * s, Nm, Nm, s, s, K, false,
               st);                                                                     // G = C1 Q
    TS_CUDA(cudaMemsetAsync(w.err, 0, sizeof(int), st));
    shifted_lu(Hproj, sHp, op->schurT, w.LU, w.piv, Nm, std::min(s, Nm - 1), s, K, w.err, st);
    hs_solve(w.LU, w.piv, w.Gp, op->schurT, w.Z, Nm, std::min(s, Nm - 1), s, K, st);
    small_gemm(w.Z, (long long)Nm * s, Nm, op->schurQ, ss, s, true, w.Y, (long long)Nm * s, Nm, Nm, s, s, K, false,
               st);                                                                     // Y = Z Q^H
    // Proposition 5.2 estimate ||H_{m+1,m} E_m Y||
    small_gemm(w.Hlast, ss, s, w.Y + (long long)(mm - 1) * s, (long long)Nm * s, Nm, false, w.E, ss, s, s, s, s, K,
               false, st);
    k_weighted_fro<<<1, 256, 0, st>>>(w.E, s, K, p, w.sc + 4);
    count_launch();
    TS_CUDA(cudaGetLastError());
    // X += V_m Y
    for (int j = 0; j < mm; ++j) {
      if (low)
        rows_mm(w, V32 + (long long)j * blk, w.X, w.Y + (long long)j * s, (long long)Nm * s, Nm, 1.0, true, st);
      else
        rows_mm(w, w.V + (long long)j * blk, w.X, w.Y + (long long)j * s, (long long)Nm * s, Nm, 1.0, true, st);
    }
    int e = 0;
    TS_CUDA(cudaMemcpyAsync(&e, w.err, sizeof(int), cudaMemcpyDeviceToHost, st));
    const double est = std::sqrt(std::max(0.0, read_scalar(w.sc + 4, ctx, st)));
    if (e & 2) return finish(TS_SINGULAR);
    last_est = est;
    push_hist(est);
    ++info.cycles;
    res = residual(ctx, op, w, st);
    ++info.applies_fp64;
    push_true(res);
    if (!std::isfinite(res)) return finish(TS_ERR_NONFINITE);
    if (res <= o.tol * normC) return finish(TS_OK);
  }
  return finish(TS_NOT_CONVERGED);
}

}  // namespace

ts_status tba_entry(ts_ctx* ctx, const ts_op* cop, const double* C, double* X, const ts_solve_opts* opts,
                    ts_solve_info* info_out, ts_stream stream) {
  ts_op* op = const_cast<ts_op*>(cop);
  TS_REQUIRE(op && C && X && opts, "ts_tba_solve: null pointer");
  const ts_solve_opts& o = *opts;
  TS_REQUIRE(o.restart >= 1 && o.restart <= 256, "ts_tba_solve: restart must be in 1..256");
  TS_REQUIRE(o.max_restarts >= 1, "ts_tba_solve: max_restarts must be >= 1");
  TS_REQUIRE(o.tol > 0.0 && std::isfinite(o.tol), "ts_tba_solve: tol must be positive");
  if (o.precision != TS_FP64 && o.precision != TS_MIXED_FP32)
    throw Error{TS_ERR_UNSUPPORTED, "TBAS runs in FP64 or TS_MIXED_FP32 only"};
  if (o.fp64_engine != TS_ENGINE_DFMA) throw Error{TS_ERR_UNSUPPORTED, "TBAS runs on the FP64 DFMA engine only"};
  TS_CUDA(cudaSetDevice(ctx->device));
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  ts_solve_info info{};
  TS_CUDA(cudaEventRecord(ctx->ev0, st));
  const size_t N = (size_t)op->n * op->s * op->p;
  StagedIn c(ctx, "solve_inC", C, N, st);
  StagedOut x(ctx, "solve_ioX", X, N, true, st);
  ts_status s = tbas_solve(ctx, op, c.dev, x.dev, o, info, st);
  x.finish();
  TS_CUDA(cudaEventRecord(ctx->ev1, st));
  TS_CUDA(cudaEventSynchronize(ctx->ev1));
  float ms = 0.f;
  TS_CUDA(cudaEventElapsedTime(&ms, ctx->ev0, ctx->ev1));
  info.ms_total = ms;
  if (info_out) *info_out = info;
  return s;
}

// Dense operator apply for a sparse op (ts_sylv_apply / residuals): X real -> Y = M(X) real.
void apply_sparse_f64(ts_ctx* ctx, const ts_op* cop, const double* X, double* Y, cudaStream_t st) {
  ts_op* op = const_cast<ts_op*>(cop);
  ensure_brow(op, st);
  const int n = op->n, s = op->s, p = op->p, K = op->K;
  TS_REQUIRE(s <= kMaxS, "sparse operator: s must be <= 64");
  const size_t blk = sizeof(double2) * (size_t)K * n * s;
  double2* a = (double2*)ctx->ws.get("sp_a", blk);
  double2* b = (double2*)ctx->ws.get("sp_b", blk);
  double2* t = (double2*)ctx->ws.get("sp_t", blk);
  to_rows(X, a, t, n, s, p, st);
  rows_call(1, op, a, nullptr, b, nullptr, n, s, K, p, st);
  from_rows(b, Y, t, n, s, p, st);
}

// t-Bartels-Stewart (Algorithm 5) for small dense A (n x n x p), B (s x s x p): A*X - X*B = C.
void t_bartels_stewart_dev(ts_ctx* ctx, const double* A, int n, const double* B, int s, int p, const double* C,
                           double* X, cudaStream_t st) {
  const int K = num_slices(p);
  TS_REQUIRE((long long)K * s * n * n <= (1ll << 28), "ts_t_bartels_stewart: K*s*n^2 too large (small solver)");
  TS_REQUIRE(n <= 12000, "ts_t_bartels_stewart: n too large");
  double2* Ah = (double2*)ctx->ws.get("bs_Ah", sizeof(double2) * (size_t)K * n * n);
  double2* T = (double2*)ctx->ws.get("bs_T", sizeof(double2) * (size_t)K * s * s);
  double2* Q = (double2*)ctx->ws.get("bs_Q", sizeof(double2) * (size_t)K * s * s);
  double2* Ch = (double2*)ctx->ws.get("bs_Ch", sizeof(double2) * (size_t)K * n * s);
  double2* Gp = (double2*)ctx->ws.get("bs_G", sizeof(double2) * (size_t)K * n * s);
  double2* Z = (double2*)ctx->ws.get("bs_Z", sizeof(double2) * (size_t)K * n * s);
  double2* LU = (double2*)ctx->ws.get("bs_LU", sizeof(double2) * (size_t)K * s * n * n);
  int* piv = (int*)ctx->ws.get("bs_piv", sizeof(int) * (size_t)K * s * n);
  int* err = (int*)ctx->ws.get("bs_err", sizeof(int));
  rfft_tube<double, double2>(A, Ah, (long long)n * n, p, st);
  rfft_tube<double, double2>(B, T, (long long)s * s, p, st);
  rfft_tube<double, double2>(C, Ch, (long long)n * s, p, st);
  TS_CUDA(cudaMemsetAsync(err, 0, sizeof(int), st));
  schur_small(T, Q, s, K, err, st);                                                // B_k = Q T Q^H
  const long long ss = (long long)s * s;
  small_gemm(Ch, (long long)n * s, n, Q, ss, s, false, Gp, (long long)n * s, n, n, s, s, K, false, st);   // G = C Q
  shifted_lu(Ah, (long long)n * n, T, LU, piv, n, n - 1, s, K, err, st);           // A_k - t_jj I
  hs_solve(LU, piv, Gp, T, Z, n, n - 1, s, K, st);
  small_gemm(Z, (long long)n * s, n, Q, ss, s, true, Ch, (long long)n * s, n, n, s, s, K, false, st);     // X = Z Q^H
  irfft_tube<double, double2>(Ch, X, (long long)n * s, p, IRFFT_STORE, nullptr, nullptr, st);
  int e = 0;
  TS_CUDA(cudaMemcpyAsync(&e, err, sizeof(int), cudaMemcpyDeviceToHost, st));
  TS_CUDA(cudaStreamSynchronize(st));
  if (e & 1) throw Error{TS_SINGULAR, "complex Schur iteration of B_k did not converge"};
  if (e & 2) throw Error{TS_SINGULAR, "A_k - lambda I singular for an eigenvalue lambda of B_k (Theorem 2.1)"};
}

// Sparse operator from p CSR slices (host arrays): union pattern on the host, values' Fourier
// slices on the device.
void op_prepare_csr(ts_op* op, const int* rowptr, const int* col, const double* val, cudaStream_t st) {
  const int n = op->n, p = op->p, K = op->K;
  std::vector<int> urow(n + 1, 0);
  std::vector<int> ucol;
  std::vector<std::vector<int>> rows(n);
  for (int t = 0; t < p; ++t) {
    const int* rp = rowptr + (size_t)t * (n + 1);
    for (int i = 0; i < n; ++i) {
      TS_REQUIRE(rp[i] <= rp[i + 1], "ts_op_create_csr: row pointers must be non-decreasing");
      for (int q = rp[i]; q < rp[i + 1]; ++q) {
        TS_REQUIRE(col[q] >= 0 && col[q] < n, "ts_op_create_csr: column index out of range");
        rows[i].push_back(col[q]);
      }
    }
  }
  for (int i = 0; i < n; ++i) {
    std::sort(rows[i].begin(), rows[i].end());
    rows[i].erase(std::unique(rows[i].begin(), rows[i].end()), rows[i].end());
    urow[i + 1] = urow[i] + (int)rows[i].size();
    ucol.insert(ucol.end(), rows[i].begin(), rows[i].end());
  }
  const int nnz = urow[n];
  std::vector<double> uval((size_t)p * std::max(nnz, 1), 0.0);
  for (int t = 0; t < p; ++t) {
    const int* rp = rowptr + (size_t)t * (n + 1);
    for (int i = 0; i < n; ++i)
      for (int q = rp[i]; q < rp[i + 1]; ++q) {
        const int* b = ucol.data() + urow[i];
        const int* e = ucol.data() + urow[i + 1];
        const int pos = (int)(std::lower_bound(b, e, col[q]) - ucol.data());
        uval[(size_t)t * nnz + pos] += val[q];
      }
  }
  op->sp = new SparseOp();
  op->sp->nnz = nnz;
  op_alloc(op->sp->rowptr, sizeof(int) * (n + 1));
  op_alloc(op->sp->col, sizeof(int) * std::max(nnz, 1));
  op_alloc(op->sp->vals, sizeof(double2) * (size_t)K * std::max(nnz, 1));
  double* dval = (double*)op->ctx->ws.get("csr_stage_vals", sizeof(double) * (size_t)p * std::max(nnz, 1));
  TS_CUDA(cudaMemcpyAsync(op->sp->rowptr, urow.data(), sizeof(int) * (n + 1), cudaMemcpyHostToDevice, st));
  if (nnz > 0) {
    TS_CUDA(cudaMemcpyAsync(op->sp->col, ucol.data(), sizeof(int) * nnz, cudaMemcpyHostToDevice, st));
    TS_CUDA(cudaMemcpyAsync(dval, uval.data(), sizeof(double) * (size_t)p * nnz, cudaMemcpyHostToDevice, st));
    rfft_tube<double, double2>(dval, op->sp->vals, nnz, p, st);
  }
  TS_CUDA(cudaStreamSynchronize(st));
}

}  // namespace ts
