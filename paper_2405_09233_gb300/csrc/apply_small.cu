// The whole FP64 operator Y = M(X) (or Y = C - M(X)) of a small dense equation in one launch: DFT along
// mode 3, slice products A_k X_k - X_k B_k and inverse DFT.
//
// As three launches (rfft_tube, zgemm_slices_f64, irfft_tube) such an application is 3.1 + 4.9 + 3.4 us of
// kernels that mostly wait for a load round trip each, plus the gaps between them.  Here one CTA of four
// warps (one per SM sub-partition, the FP64 issue units) owns 4 x TN outputs of every slice:
//   1. the A_k rows and B_k columns it multiplies go to shared memory (cp.async) while its threads load and
//      transform the tubes of the X columns and X rows it needs (one tube per thread; a tube is transformed
//      again by every CTA that needs it, which is cheaper than a second launch while tiles are few);
//   2. the 4 TN outputs of a slice times 32 / TN slots over the concatenated reduction (n of A_k X_k, then s
//      of X_k B_k) fill the 128 threads; the slots' partial sums are added by a shuffle tree and over the
//      warps in order;
//   3. the inverse DFT runs as one direct sum per (output, t), all threads busy (a register FFT of the few
//      tubes would be one warp's serial chain).
// The rule that chooses it (apply_small_tile) compares the FP64 instructions of both forms.  Us per call, three
// launches -> one: 24 x 24 x 4 17.5 -> 11.8 (bound by the caller's launch rate), 32 x 32 x 8 21.7 -> 14.3,
// 48 x 48 x 4 19.6 -> 11.8, 96 x 96 x 1 38.8 -> 14.4, 16 x 16 x 31 143 -> 60.
#include <algorithm>
#include <cmath>
#include "internal.cuh"
#include "apply.cuh"
#include "reduce.cuh"
#include "fft_reg.cuh"

namespace ts {
namespace {

constexpr int kSmThreads = 128, kSmTM = 4, kSmMaxP = 32;

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

struct SmallApply {
  const double* X;
  double* Y;
  const double2 *Ah, *Bh;
  const double* C;        // non-null: Y = C - M(X), squares of Y summed per CTA into partials
  double* partials;
  const int* gate;
  int n, s, p, K, nyq, mtiles;
};

// Shared memory, in double2: the twiddles (c, s), then the panels.
struct SmallLayout {
  int tw, Xc, Xr, A, B, part, Yk, total;
  __host__ __device__ SmallLayout(int n, int s, int p, int K, int TN) {
    tw = 0;
    Xc = tw + p;
    Xr = Xc + K * n * TN;
    A = Xr + K * s * kSmTM;
    B = A + K * n * kSmTM;
    part = B + K * s * TN;
    Yk = part + K * 4 * kSmTM * TN;
    total = Yk + K * kSmTM * TN;
  }
};

// P: the tube length when POW2, else a bound on it (direct DFT of a.p <= P samples in registers).
template <int P, bool POW2, int TN>
__global__ void __launch_bounds__(kSmThreads) k_apply_small(SmallApply a) {
  step_kernel_begin();
  if (a.gate && *a.gate == 0) return;   // a cycle that already ended (launched ahead)
  extern __shared__ double2 sm[];
  const int n = a.n, s = a.s, K = a.K, p = POW2 ? P : a.p;
  const SmallLayout L(n, s, p, K, TN);
  double* tc = reinterpret_cast<double*>(sm + L.tw);
  double* tsn = tc + p;
  double2 *Xc = sm + L.Xc, *Xr = sm + L.Xr, *At = sm + L.A, *Bt = sm + L.B, *part = sm + L.part, *Yk = sm + L.Yk;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int i0 = (int)(blockIdx.x % a.mtiles) * kSmTM, j0 = (int)(blockIdx.x / a.mtiles) * TN;
  const long long T = (long long)n * s;

  for (int q = t; q < K * n * kSmTM; q += kSmThreads) {      // At[k][l][i] = A_k[i0 + i, l]
    const int i = q % kSmTM, kl = q / kSmTM;
    if (i0 + i < n) cp_async16(At + q, a.Ah + (long long)kl * n + i0 + i);
    else At[q] = make_double2(0.0, 0.0);
  }
  for (int q = t; q < K * s * TN; q += kSmThreads) {         // Bt[k][l][j] = B_k[l, j0 + j]
    const int l = q % s, j = (q / s) % TN, k = q / (s * TN);
    double2* d = Bt + (k * s + l) * TN + j;
    if (j0 + j < s) cp_async16(d, a.Bh + ((long long)k * s + j0 + j) * s + l);
    else *d = make_double2(0.0, 0.0);
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  if constexpr (!POW2) {
    fill_roots(tc, tsn, p, t, kSmThreads);
    __syncthreads();
  }

  // Tubes: the TN columns of X (Xc[k][l][j]), then its 4 rows (Xr[k][l][i]).
  const int ncol = TN * n;
  for (int q = t; q < ncol + kSmTM * s; q += kSmThreads) {
    int row, col, step;
    double2* dst;
    if (q < ncol) {
      row = q % n;
      col = j0 + q / n;
      dst = Xc + row * TN + q / n;
      step = n * TN;
    } else {
      const int r = q - ncol;
      row = i0 + r % kSmTM;
      col = r / kSmTM;
      dst = Xr + r;
      step = s * kSmTM;
    }
    const bool in = row < n && col < s;
    const double* src = a.X + (long long)col * n + row;
    if constexpr (POW2) {
      rfft_reg<double, P>([&](int u) { return in ? src[u * T] : 0.0; },
                          [&](int k, double re, double im) { dst[k * step] = make_double2(re, im); });
    } else {
      rfft_direct<double, P>([&](int u) { return in ? src[u * T] : 0.0; },
                             [&](int k, double re, double im) { dst[k * step] = make_double2(re, im); }, p, 0, 1,
                             [&](int r) { return tc[r]; }, [&](int r) { return tsn[r]; });
    }
  }
  if constexpr (POW2) {   // for the inverse
    for (int r = t; r < p; r += kSmThreads) {
      tc[r] = cos32(r * (32 / P));
      tsn[r] = sin32(r * (32 / P));
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();

  constexpr int OUT = kSmTM * TN, SLOTS = kSmThreads / OUT;
  const int o = t % OUT, i = o % kSmTM, j = o / kSmTM, slot = t / OUT;
  for (int k = 0; k < K; ++k) {
    const double2 *Ak = At + k * n * kSmTM + i, *Xk = Xc + k * n * TN + j;
    const double2 *Rk = Xr + k * s * kSmTM + i, *Bk = Bt + k * s * TN + j;
    double r0 = 0.0, r1 = 0.0, m0 = 0.0, m1 = 0.0;
    if (k == 0 || k == a.nyq) {
      for (int l = slot; l < n; l += SLOTS) r0 = fma(Ak[l * kSmTM].x, Xk[l * TN].x, r0);
      for (int l = slot; l < s; l += SLOTS) r1 = fma(-Rk[l * kSmTM].x, Bk[l * TN].x, r1);
    } else {
      for (int l = slot; l < n; l += SLOTS) {
        const double2 u = Ak[l * kSmTM], v = Xk[l * TN];
        r0 = fma(u.x, v.x, r0);
        r1 = fma(-u.y, v.y, r1);
        m0 = fma(u.x, v.y, m0);
        m1 = fma(u.y, v.x, m1);
      }
      for (int l = slot; l < s; l += SLOTS) {
        const double2 u = Rk[l * kSmTM], v = Bk[l * TN];
        r0 = fma(-u.x, v.x, r0);
        r1 = fma(u.y, v.y, r1);
        m0 = fma(-u.x, v.y, m0);
        m1 = fma(-u.y, v.x, m1);
      }
      m0 += m1;
#pragma unroll
      for (int d = 16; d >= OUT; d >>= 1) m0 += __shfl_down_sync(0xffffffffu, m0, d);
    }
    r0 += r1;
#pragma unroll
    for (int d = 16; d >= OUT; d >>= 1) r0 += __shfl_down_sync(0xffffffffu, r0, d);
    if (lane < OUT) part[(k * 4 + warp) * OUT + lane] = make_double2(r0, m0);
  }
  __syncthreads();
  for (int q = t; q < K * OUT; q += kSmThreads) {
    const double2* pk = part + (q / OUT) * 4 * OUT + q % OUT;
    const double2 b0 = pk[0], b1 = pk[OUT], b2 = pk[2 * OUT], b3 = pk[3 * OUT];
    // twice every slice that stands for a conjugate pair
    const int k = q / OUT;
    const double w = (k == 0 || k == a.nyq) ? 1.0 : 2.0;
    Yk[q] = make_double2(w * ((b0.x + b1.x) + (b2.x + b3.x)), w * ((b0.y + b1.y) + (b2.y + b3.y)));
  }
  __syncthreads();
  const double invp = 1.0 / p;
  double local = 0.0;
  for (int q = t; q < OUT * p; q += kSmThreads) {
    const int oo = q % OUT, u = q / OUT, row = i0 + oo % kSmTM, col = j0 + oo / kSmTM;
    if (row >= n || col >= s) continue;
    double y = 0.0, z = 0.0;
    int r = 0;
    for (int k = 0; k < K; ++k) {
      const double2 c = Yk[k * OUT + oo];
      y = fma(c.x, tc[r], y);
      if (k != 0 && k != a.nyq) z = fma(-c.y, tsn[r], z);
      r += u;
      if (r >= p) r -= p;
    }
    const long long e = u * T + (long long)col * n + row;
    double v = (y + z) * invp;
    if (a.C) {
      v = a.C[e] - v;
      local = fma(v, v, local);
    }
    a.Y[e] = v;
  }
  if (a.C) {
    const double tot = block_sum(local);
    if (t == 0) a.partials[blockIdx.x] = tot;
    if (blockIdx.x == 0)
      for (int b = gridDim.x + t; b < kRedBlocks; b += kSmThreads) a.partials[b] = 0.0;
  }
}

// FP64 instructions of the transform of one tube (a register FFT of a power of two, else direct sums).
double tube_ops(int p) {
  if (p <= 1) return 1.0;
  if ((p & (p - 1)) == 0) return p == 2 ? 2.0 : 2.5 * p * std::max(1.0, std::log2(p / 2.0)) - 1.0 * p;
  return 2.0 * ((p - 1) / 2) * (p / 2 + 1) + p;
}

// Clocks of the busiest SM: its four sub-partitions issue an FP64 instruction of a warp in 64 clocks each.
double small_cost(int n, int s, int p, int TN) {
  const int K = num_slices(p), nr = nyquist_index(p) > 0 ? 2 : 1;
  const long long tiles = (long long)((n + kSmTM - 1) / kSmTM) * ((s + TN - 1) / TN);
  const int tubes = TN * n + kSmTM * s, OUT = kSmTM * TN;
  const double per = 64.0 * ((tubes + kSmThreads - 1) / kSmThreads) * tube_ops(p) +
                     0.5 * OUT * (n + s) * (4.0 * (K - nr) + nr) + 1.0 * OUT * K * p + 3.0 * kSmThreads * K;
  return (double)((tiles + 151) / 152) * per;
}
// The three launches: the transforms run blocks of 256 tubes, the products fill the chip.
double split_cost(int n, int s, int p) {
  const int K = num_slices(p), nr = nyquist_index(p) > 0 ? 2 : 1;
  const double T = (double)n * s;
  const long long blocks = ((long long)n * s + 255) / 256;
  return 2.0 * ((blocks + 151) / 152) * (T > 128 ? 2 : 1) * 64.0 * tube_ops(p) +
         1.15 * T * (n + s) * (4.0 * (K - nr) + nr) / (2.0 * 152.0);
}
// Clocks of the two launches saved, with their round trips.  Both forms at sizes near the line (us per call,
// three launches / one): 300 x 20 x 3 67.8 / 58.7 and 40 x 100 x 6 47.2 / 37.0 differ by 20000 and 23500 in
// the costs above, 64 x 64 x 16 63.2 / 86.4 by 40000, 100 x 50 x 7 51.4 / 84.2 by 55000.
constexpr double kSplitLaunches = 26000.0;

template <int P, bool POW2>
void launch(const SmallApply& a, int tn, cudaStream_t st) {
  const int smem = (int)sizeof(double2) * SmallLayout(a.n, a.s, a.p, a.K, tn).total;
  const unsigned tiles = (unsigned)a.mtiles * ((a.s + tn - 1) / tn);
  auto go = [&](auto kernel) {
    if (smem > 48 * 1024) set_max_dynamic_smem(reinterpret_cast<const void*>(kernel), smem);
    launch_step_kernel(kernel, a.gate != nullptr, tiles, kSmThreads, smem, 0, st, a);
  };
  if (tn == 2) go(k_apply_small<P, POW2, 2>);
  else go(k_apply_small<P, POW2, 4>);
}

}  // namespace

int apply_small_tile(int n, int s, int p) {
  if (p > kSmMaxP) return 0;
  int best = 0;
  double cost = split_cost(n, s, p) + kSplitLaunches;
  for (int tn : {4, 2}) {
    const long long tiles = (long long)((n + kSmTM - 1) / kSmTM) * ((s + tn - 1) / tn);
    if (tiles > kRedBlocks || n + s > 2048) continue;
    if (sizeof(double2) * SmallLayout(n, s, p, num_slices(p), tn).total > 200 * 1024) continue;
    const double c = small_cost(n, s, p, tn);
    if (c < cost) {
      cost = c;
      best = tn;
    }
  }
  return best;
}

void apply_small_f64(const ts_op* op, int tn, const double* X, double* Y, const double* C, double* partials,
                     cudaStream_t st, const int* gate) {
  SmallApply a{};
  a.X = X; a.Y = Y; a.Ah = op->Ah; a.Bh = op->Bh; a.C = C; a.partials = partials; a.gate = gate;
  a.n = op->n; a.s = op->s; a.p = op->p; a.K = op->K; a.nyq = nyquist_index(op->p);
  a.mtiles = (op->n + kSmTM - 1) / kSmTM;
  switch (op->p) {
    case 2: launch<2, true>(a, tn, st); break;
    case 4: launch<4, true>(a, tn, st); break;
    case 8: launch<8, true>(a, tn, st); break;
    case 16: launch<16, true>(a, tn, st); break;
    case 32: launch<32, true>(a, tn, st); break;
    default:
      if (op->p <= 4) launch<4, false>(a, tn, st);
      else if (op->p <= 8) launch<8, false>(a, tn, st);
      else if (op->p <= 16) launch<16, false>(a, tn, st);
      else launch<32, false>(a, tn, st);
  }
  count_launch();
  TS_CUDA(cudaGetLastError());
}

}  // namespace ts
