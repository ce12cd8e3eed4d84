// Output tiles of the fused per-slice complex product (see gemm_simt.cu), shared by the grid-mapped
// kernels and the work-list kernel of the batched solver: Y_k(i0.., j0..) = A1_k B1_k + sgn2 A2_k B2_k for
// one tile; slices k == 0 and k == nyq are real.  sgn2 is +1 or -1 (any value when L2 == 0).
#pragma once
#include "internal.cuh"

namespace ts {

template <typename Real> struct CplxOf;
template <> struct CplxOf<double> { using T = double2; };
template <> struct CplxOf<float> { using T = float2; };

// FP64 tiles: BM x BN outputs for NT threads, TM rows of one column per thread (BM = NT / BN * TM,
// lanes along rows so that outputs are written in runs).
// What bounds it: the FP64 pipe, which takes 16 clocks of the SM for one warp's FMA.  Against that,
// shared memory needs no operand reuse at all (six 8-byte reads per three FMAs even with one output
// per thread) and neither does L2, so the tile's shape is free to follow the problem: narrow tiles
// pad a ragged s less, small ones spread evenly over the SMs, and what a small tile costs is the
// factor sums ar + ai, br + bi (one FP64 addition per staged entry, (BM + BN) / (3 BM BN) of the
// products).  The next block of operands is loaded into registers during the products and three or
// more CTAs share an SM, so the pipe does not wait for memory.  Every tile adds an entry's products in
// the same order: the choice never changes a result.
// Measured (products of M): n = 500, s = 130, p = 12 2058 -> 1376 us; n = s = 1024, p = 16 84.1 -> 81.9 ms
// (0.96 of the pipe); 300 x 200 x 100, p = 7 T-product 234 -> 141 us, all against one 64 x 64 (or 32 x 32)
// tile per CTA and per SM.
template <int NT, int BN, int TM>
struct F64Tile {
  static constexpr int TY = NT / BN, BM = TY * TM, BK = BM > 64 ? 8 : 16;
};

__device__ __forceinline__ double flip(double v, bool neg) {   // -v without an FP64 instruction
  return __longlong_as_double(__double_as_longlong(v) ^ (neg ? (long long)0x8000000000000000ull : 0ll));
}

template <int NT, int BN, int TM>
__device__ __forceinline__ void gemm_tile_f64(const ZGemmArgs& a, int k, int i0, int j0) {
  using Cfg = F64Tile<NT, BN, TM>;
  constexpr int BM = Cfg::BM, BK = Cfg::BK, TY = Cfg::TY;
  constexpr int LA = BM * BK / NT, LB = (BN * BK + NT - 1) / NT;
  static_assert(BM * BK % NT == 0, "tile shape");
  __shared__ double sA[3][BK][BM];
  __shared__ double sB[3][BK][BN + 1];
  if (a.gate && *a.gate == 0) return;
  const bool real = (k == 0) || (k == a.nyq);
  const int tid = threadIdx.x, row = tid % TY, col = tid / TY;
  double acc[3][TM];
#pragma unroll
  for (int z = 0; z < 3; ++z)
#pragma unroll
    for (int q = 0; q < TM; ++q) acc[z][q] = 0.0;
  double2 ra[LA], rb[LB];
  const int n1 = (a.L1 + BK - 1) / BK, n2 = (a.L2 + BK - 1) / BK;   // blocks of each product
  auto load = [&](int b) {
    const bool first = b < n1;
    const int L = first ? a.L1 : a.L2, l0 = (first ? b : b - n1) * BK;
    const int lda = first ? a.lda1 : a.lda2, ldb = first ? a.ldb1 : a.ldb2;
    const double2* A = first ? a.A1 + a.sA1 * k : a.A2 + a.sA2 * k;
    const double2* B = first ? a.B1 + a.sB1 * k : a.B2 + a.sB2 * k;
#pragma unroll
    for (int q = 0; q < LA; ++q) {   // column-major source: consecutive threads walk the rows
      const int e = tid + NT * q, r = e % BM, c = e / BM;
      ra[q] = make_double2(0.0, 0.0);
      if (i0 + r < a.M && l0 + c < L) ra[q] = A[(long long)(l0 + c) * lda + i0 + r];
    }
#pragma unroll
    for (int q = 0; q < LB; ++q) {   // consecutive threads walk down a column
      const int e = tid + NT * q, c = e % BK, jj = e / BK;
      rb[q] = make_double2(0.0, 0.0);
      if (jj < BN && j0 + jj < a.N && l0 + c < L) rb[q] = B[(long long)(j0 + jj) * ldb + l0 + c];
    }
  };
  load(0);
  for (int b = 0; b < n1 + n2; ++b) {
    const bool neg = b >= n1 && a.sgn2 < 0.0;
    __syncthreads();   // the products of the block before are done with the buffers
#pragma unroll
    for (int q = 0; q < LA; ++q) {
      const int e = tid + NT * q, r = e % BM, c = e / BM;
      sA[0][c][r] = ra[q].x;
      if (!real) {
        sA[1][c][r] = ra[q].y;
        sA[2][c][r] = ra[q].x + ra[q].y;
      }
    }
#pragma unroll
    for (int q = 0; q < LB; ++q) {
      const int e = tid + NT * q, c = e % BK, jj = e / BK;
      if (jj < BN) {
        const double x = flip(rb[q].x, neg), y = flip(rb[q].y, neg);
        sB[0][c][jj] = x;
        if (!real) {
          sB[1][c][jj] = y;
          sB[2][c][jj] = x + y;
        }
      }
    }
    __syncthreads();
    if (b + 1 < n1 + n2) load(b + 1);
    if (real) {
#pragma unroll 4
      for (int c = 0; c < BK; ++c) {
        const double bv = sB[0][c][col];
#pragma unroll
        for (int q = 0; q < TM; ++q) acc[0][q] = fma(sA[0][c][row + TY * q], bv, acc[0][q]);
      }
    } else {
#pragma unroll 4
      for (int c = 0; c < BK; ++c) {
#pragma unroll
        for (int z = 0; z < 3; ++z) {
          const double bv = sB[z][c][col];
#pragma unroll
          for (int q = 0; q < TM; ++q) acc[z][q] = fma(sA[z][c][row + TY * q], bv, acc[z][q]);
        }
      }
    }
  }
  const int j = j0 + col;
  if (j >= a.N) return;
  double2* Y = a.Y + a.sY * k + (long long)j * a.ldy;
#pragma unroll
  for (int q = 0; q < TM; ++q) {
    const int i = i0 + row + TY * q;
    if (i < a.M)
      Y[i] = real ? make_double2(acc[0][q], 0.0)
                  : make_double2(acc[0][q] - acc[1][q], acc[2][q] - acc[0][q] - acc[1][q]);
  }
}

// FP32 tiles: BM x BN outputs, an 8 x 4 block of outputs per thread.  G groups of threads split each block
// of the reduction (G > 1 for small tiles, which have few such blocks); their sums are added in order at
// the end.
// What bounds it: FP32 issue and shared-memory reads alike.  A warp reads 128 bytes of shared memory per
// clock whether or not lanes share an address, so an 8 x 4 complex block (24 values per 96 FMAs) just
// balances the two, and a 4 x 4 one is bound by the reads.  The factor sums are therefore formed in
// registers (a third staged plane cost more reads than it saved additions), the products are packed
// FMAs on pairs of rows, operands are loaded one block ahead into registers and stored to the other of
// two shared-memory buffers (one barrier per block), rows of B padded by four words so that its
// transposed stores spread over the banks.
// Measured: n = 512, s = 128, p = 16 165 -> 65 us; (4 x 4 blocks, three staged planes and two barriers per
// block before); n = s = 1024, p = 16 2.18 ms, 0.56 of the FP32 rate.
template <int BM, int BN, int G>
struct F32Tile {
  static constexpr int BK = 16, PB = BN + 4, T = BM * BN / 32, NT = T * G;
  static constexpr int kBuf = 2 * BK * (BM + PB);                      // floats of one buffer
  static constexpr int kSum = G > 1 ? (G - 1) * T * 96 : 0;            // floats of the groups' sums
  static constexpr int kSmem = (2 * kBuf > kSum ? 2 * kBuf : kSum) * (int)sizeof(float);
  static_assert(kSmem <= 48 * 1024, "dynamic shared memory without opt-in");
};

using f32x2 = unsigned long long;   // two packed FP32 values
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32x2 dup2(float v) {
  f32x2 d;
  asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(v));
  return d;
}
__device__ __forceinline__ void split2(f32x2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}

template <int BM, int BN, int G>
__device__ __forceinline__ void gemm_tile_f32(const CGemmArgs& a, int k, int i0, int j0) {
  using Cfg = F32Tile<BM, BN, G>;
  constexpr int TM = 8, TN = 4, BK = Cfg::BK, NT = Cfg::NT, PB = Cfg::PB, TY = BM / TM, T = Cfg::T;
  constexpr int LA = BM * BK / NT, LB = BN * BK / NT;
  static_assert(T % 32 == 0 && BK % G == 0 && BM * BK % NT == 0 && BN * BK % NT == 0, "tile shape");
  extern __shared__ __align__(16) float f32_smem[];
  if (a.gate && *a.gate == 0) return;
  const bool real = (k == 0) || (k == a.nyq);
  const int tid = threadIdx.x, grp = tid / T, ty = tid % T % TY, tx = tid % T / TY;
  f32x2 acc[3][TM / 2][TN];   // rows in pairs
#pragma unroll
  for (int z = 0; z < 3; ++z)
#pragma unroll
    for (int q = 0; q < TM / 2; ++q)
#pragma unroll
      for (int r = 0; r < TN; ++r) acc[z][q][r] = 0ull;
  float2 ra[LA], rb[LB];
  const int n1 = (a.L1 + BK - 1) / BK, n2 = (a.L2 + BK - 1) / BK;
  auto load = [&](int b) {
    const bool first = b < n1;
    const int L = first ? a.L1 : a.L2, l0 = (first ? b : b - n1) * BK;
    const int lda = first ? a.lda1 : a.lda2, ldb = first ? a.ldb1 : a.ldb2;
    const float2* A = first ? a.A1 + a.sA1 * k : a.A2 + a.sA2 * k;
    const float2* B = first ? a.B1 + a.sB1 * k : a.B2 + a.sB2 * k;
#pragma unroll
    for (int q = 0; q < LA; ++q) {
      const int e = tid + NT * q, r = e % BM, c = e / BM;
      ra[q] = make_float2(0.f, 0.f);
      if (i0 + r < a.M && l0 + c < L) ra[q] = A[(long long)(l0 + c) * lda + i0 + r];
    }
#pragma unroll
    for (int q = 0; q < LB; ++q) {
      const int e = tid + NT * q, c = e % BK, jj = e / BK;
      rb[q] = make_float2(0.f, 0.f);
      if (j0 + jj < a.N && l0 + c < L) rb[q] = B[(long long)(j0 + jj) * ldb + l0 + c];
    }
  };
  const float sgn2 = (float)a.sgn2;
  auto store = [&](int b) {   // block b's registers into buffer b & 1
    float* sA = f32_smem + (b & 1) * Cfg::kBuf;
    float* sB = sA + 2 * BK * BM;
    const float sgn = b >= n1 ? sgn2 : 1.f;
#pragma unroll
    for (int q = 0; q < LA; ++q) {
      const int e = tid + NT * q;
      sA[e] = ra[q].x;
      if (!real) sA[BK * BM + e] = ra[q].y;
    }
#pragma unroll
    for (int q = 0; q < LB; ++q) {
      const int e = tid + NT * q, o = e % BK * PB + e / BK;
      sB[o] = rb[q].x * sgn;
      if (!real) sB[BK * PB + o] = rb[q].y * sgn;
    }
  };
  load(0);
  store(0);
  __syncthreads();
  for (int b = 0; b < n1 + n2; ++b) {
    if (b + 1 < n1 + n2) load(b + 1);
    const float* sA = f32_smem + (b & 1) * Cfg::kBuf + ty * 4;
    const float* sB = f32_smem + (b & 1) * Cfg::kBuf + 2 * BK * BM + tx * TN;
    auto rows = [&](const float* p, f32x2 (&v)[TM / 2]) {   // rows 4 ty + (4 TY) h ..
#pragma unroll
      for (int h = 0; h < TM / 4; ++h) {
        const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(p + h * 4 * TY);
        v[2 * h] = q.x;
        v[2 * h + 1] = q.y;
      }
    };
    auto cols = [&](const float* p, f32x2 (&v)[TN]) {
      const float4 q = *reinterpret_cast<const float4*>(p);
      v[0] = dup2(q.x);
      v[1] = dup2(q.y);
      v[2] = dup2(q.z);
      v[3] = dup2(q.w);
    };
    auto products = [&](int z, const f32x2 (&x)[TM / 2], const f32x2 (&y)[TN]) {
#pragma unroll
      for (int q = 0; q < TM / 2; ++q)
#pragma unroll
        for (int r = 0; r < TN; ++r) acc[z][q][r] = fma2(x[q], y[r], acc[z][q][r]);
    };
    if (real) {
#pragma unroll 4
      for (int c = grp * (BK / G); c < (grp + 1) * (BK / G); ++c) {
        f32x2 ar[TM / 2], br[TN];
        rows(sA + c * BM, ar);
        cols(sB + c * PB, br);
        products(0, ar, br);
      }
    } else {
#pragma unroll 4
      for (int c = grp * (BK / G); c < (grp + 1) * (BK / G); ++c) {
        f32x2 ar[TM / 2], ai[TM / 2], br[TN], bi[TN];
        rows(sA + c * BM, ar);
        cols(sB + c * PB, br);
        rows(sA + (BK + c) * BM, ai);
        cols(sB + (BK + c) * PB, bi);
        products(0, ar, br);
        products(1, ai, bi);
#pragma unroll
        for (int q = 0; q < TM / 2; ++q) ar[q] = add2(ar[q], ai[q]);
#pragma unroll
        for (int r = 0; r < TN; ++r) br[r] = add2(br[r], bi[r]);
        products(2, ar, br);
      }
    }
    if (b + 1 < n1 + n2) store(b + 1);   // the other buffer: last read before the previous barrier
    __syncthreads();
  }
  if constexpr (G > 1) {   // the other groups' sums, in order
    f32x2* sum = reinterpret_cast<f32x2*>(f32_smem);
    constexpr int E = 3 * (TM / 2) * TN;
    if (grp > 0)
#pragma unroll
      for (int e = 0; e < E; ++e) sum[((grp - 1) * E + e) * T + tid % T] = (&acc[0][0][0])[e];
    __syncthreads();
    if (grp > 0) return;
#pragma unroll
    for (int g = 0; g < G - 1; ++g)
#pragma unroll
      for (int e = 0; e < E; ++e) (&acc[0][0][0])[e] = add2((&acc[0][0][0])[e], sum[(g * E + e) * T + tid]);
  }
  float2* Y = a.Y + a.sY * k;
#pragma unroll
  for (int r = 0; r < TN; ++r) {
    const int j = j0 + tx * TN + r;
    if (j >= a.N) continue;
#pragma unroll
    for (int q = 0; q < TM / 2; ++q) {
      float t1[2], t2[2], t3[2];
      split2(acc[0][q][r], t1[0], t1[1]);
      split2(acc[1][q][r], t2[0], t2[1]);
      split2(acc[2][q][r], t3[0], t3[1]);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int i = i0 + ty * 4 + (q / 2) * 4 * TY + q % 2 * 2 + u;
        if (i < a.M)
          Y[(long long)j * a.ldy + i] =
              real ? make_float2(t1[u], 0.f) : make_float2(t1[u] - t2[u], t3[u] - t1[u] - t2[u]);
      }
    }
  }
}

// Products whose reduction lengths L1, L2 are at most kTinyL (the latency-bound small problems):
// one 8 x 4 output tile per CTA of four warps.  Each phase's operand panels (8 rows of A1 or A2,
// 4 columns of B1 or B2, over the whole reduction) go to shared memory in one round trip; then warp
// w forms the 32 outputs' partial sums over its quarter of the concatenated reduction (phase 1's l,
// then phase 2's) and warp 0 adds the four partials in order.  GB300's FP64 pipe issues one warp's
// DFMA in 64 clocks per SM sub-partition, so a single warp per tile (one sub-partition of four) ran
// ~9 us at n = s = 24, and a 16 x 16 tile of 256 threads spent most of ~19 us on padded work.
constexpr int kTinyL = 64, kTinyBM = 8, kTinyBN = 4, kTinyThreads = 128;

// One 8 x 4 tile (output rows i0.., columns j0..) of slice k; blockDim.x == kTinyThreads.
template <typename Real>
__device__ __forceinline__ void gemm_tiny_tile(const GemmArgs<typename CplxOf<Real>::T>& a, int k, int i0, int j0) {
  using Cplx = typename CplxOf<Real>::T;
  __shared__ Real sA[2][3][kTinyL][kTinyBM];
  __shared__ Real sB[2][3][kTinyL][kTinyBN];
  __shared__ Real sP[kTinyThreads / 32][3][32];
  if (a.gate && *a.gate == 0) return;
  const bool real = (k == 0) || (k == a.nyq);
  const int t = threadIdx.x;
  constexpr int QA = kTinyBM * kTinyL / kTinyThreads, QB = kTinyBN * kTinyL / kTinyThreads;
  for (int phase = 0; phase < 2; ++phase) {
    const int L = phase == 0 ? a.L1 : a.L2;
    const Cplx* A = phase == 0 ? a.A1 + a.sA1 * k : a.A2 + a.sA2 * k;
    const Cplx* B = phase == 0 ? a.B1 + a.sB1 * k : a.B2 + a.sB2 * k;
    const int lda = phase == 0 ? a.lda1 : a.lda2;
    const int ldb = phase == 0 ? a.ldb1 : a.ldb2;
    const Real sgn = phase == 0 ? Real(1) : Real(a.sgn2);
    // Every load of the phase's panels goes to registers first (fixed trip counts, predicated), so
    // all are in flight at once; a loop that stored each value to shared memory before the next load
    // ran one round trip per element.
    Cplx va[QA], vb[QB];
#pragma unroll
    for (int q = 0; q < QA; ++q) {   // A panel: rows i0.., column-major source
      const int e = t + kTinyThreads * q, r = e % kTinyBM, c = e / kTinyBM;
      va[q].x = Real(0);
      va[q].y = Real(0);
      if (e < kTinyBM * L && i0 + r < a.M) va[q] = A[(long long)c * lda + i0 + r];
    }
#pragma unroll
    for (int q = 0; q < QB; ++q) {   // B panel: columns j0.., contiguous down a column
      const int e = t + kTinyThreads * q;
      const int c = L > 0 ? e % L : 0, jj = L > 0 ? e / L : 0;
      vb[q].x = Real(0);
      vb[q].y = Real(0);
      if (e < kTinyBN * L && j0 + jj < a.N) vb[q] = B[(long long)(j0 + jj) * ldb + c];
    }
#pragma unroll
    for (int q = 0; q < QA; ++q) {
      const int e = t + kTinyThreads * q, r = e % kTinyBM, c = e / kTinyBM;
      if (e < kTinyBM * L) {
        Cplx v = va[q];
        if (real) v.y = Real(0);
        sA[phase][0][c][r] = v.x;
        sA[phase][1][c][r] = v.y;
        sA[phase][2][c][r] = v.x + v.y;
      }
    }
#pragma unroll
    for (int q = 0; q < QB; ++q) {
      const int e = t + kTinyThreads * q;
      if (e < kTinyBN * L) {
        const int c = e % L, jj = e / L;
        Cplx v = vb[q];
        if (real) v.y = Real(0);
        v.x *= sgn;
        v.y *= sgn;
        sB[phase][0][c][jj] = v.x;
        sB[phase][1][c][jj] = v.y;
        sB[phase][2][c][jj] = v.x + v.y;
      }
    }
  }
  __syncthreads();
  const int lane = t % 32, w = t / 32, r = lane % kTinyBM, jj = lane / kTinyBM;
  constexpr int NW = kTinyThreads / 32;
  const int Lt = a.L1 + a.L2, q0 = (Lt * w) / NW, q1 = (Lt * (w + 1)) / NW;
  Real acc[3] = {Real(0), Real(0), Real(0)};
  for (int q = q0; q < q1; ++q) {
    const int phase = q < a.L1 ? 0 : 1, c = q < a.L1 ? q : q - a.L1;
    if (real) {
      acc[0] = fma(sA[phase][0][c][r], sB[phase][0][c][jj], acc[0]);
    } else {
#pragma unroll
      for (int z = 0; z < 3; ++z) acc[z] = fma(sA[phase][z][c][r], sB[phase][z][c][jj], acc[z]);
    }
  }
#pragma unroll
  for (int z = 0; z < 3; ++z) sP[w][z][lane] = acc[z];
  __syncthreads();
  if (w != 0) return;
#pragma unroll
  for (int z = 0; z < 3; ++z) {
    Real v = sP[0][z][lane];
#pragma unroll
    for (int u = 1; u < NW; ++u) v += sP[u][z][lane];
    acc[z] = v;
  }
  const int i = i0 + r, j = j0 + jj;
  if (i < a.M && j < a.N) {
    Cplx v;
    if (real) {
      v.x = acc[0];
      v.y = Real(0);
    } else {
      v.x = acc[0] - acc[1];
      v.y = acc[2] - acc[0] - acc[1];
    }
    a.Y[a.sY * k + (long long)j * a.ldy + i] = v;
  }
}

}  // namespace ts
