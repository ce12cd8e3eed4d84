// The Gram-Schmidt sweep of an Arnoldi step by blocks of basis vectors: the pieces its kernels share.
//
// The sweep takes kGB basis vectors at a time.  Modified Gram-Schmidt's coefficients against
// V_b .. V_b+7 solve (I + L) h = d, d_i = <V_i, W> and L the strictly lower part of the block's Gram matrix
// <V_i, V_l>: h_i = <V_i, W - sum_{l<i} h_l V_l> written out.  So one reduction gives eight coefficients where
// a sweep vector by vector waits for eight, each behind the other; the Gram row of V_j (at most 7 more inner
// products) is formed once, in step j, whose last block it completes.  The result is modified Gram-Schmidt's
// up to rounding: the estimates of every step agree with FP64 MGS's to 1e-12 ||C|| in the tests, and the basis
// loses orthogonality alike (||V^T V - I|| after 40 steps at n = 400, condition 1e4, the two sweeps written out in
// numpy: FP64 1.9e-13 vector by vector, 2.5e-13 by blocks; FP32 5.9e-5 and 6.6e-5).
#pragma once
#include <cuda_runtime.h>
#include <type_traits>
#include "pack.cuh"
#include "reduce.cuh"

namespace ts {

constexpr int kGB = 8;              // basis vectors per block of the sweep
constexpr int kGsSums = 2 * kGB;    // sums of a pass: <V_q, W>, then <V_q, V_j> in step j's last block

// One warp: lane r < nb holds d_r on entry and h_r on return; row is the lane's Gram row (l < its own r).
__device__ __forceinline__ double gs_forward(double d, const double (&row)[kGB - 1], int nb, int lane) {
#pragma unroll
  for (int l = 0; l < kGB - 1; ++l) {
    const double hl = __shfl_sync(0xffffffffu, d, l);
    if (l + 1 < nb && lane > l && lane < nb) d = fma(-row[l], hl, d);
  }
  return d;
}

// A sum kept as FP64, or as an unevaluated sum of three FP32 numbers.  Every addition's rounding error is added
// to the next smaller part (Knuth's two-sum); what the smallest part rounds away is 2^-72 of the running sum per
// addition, so n additions err by less than FP64's n 2^-53 up to n = 2^19, without an FP64 instruction.
struct Triple {
  float hi = 0.f, mid = 0.f, lo = 0.f;
};
__host__ __device__ __forceinline__ float two_sum(float a, float b, float& err) {
  const float sum = a + b, g = sum - a;
  err = (a - (sum - g)) + (b - g);
  return sum;
}
__host__ __device__ __forceinline__ double add_sums(double a, double b) { return a + b; }
__host__ __device__ __forceinline__ Triple add_sums(Triple a, Triple b) {
  Triple s;
  float e1, e2, e3;
  s.hi = two_sum(a.hi, b.hi, e1);
  s.mid = two_sum(a.mid, b.mid, e2);
  s.mid = two_sum(s.mid, e1, e3);
  s.lo = (a.lo + b.lo) + (e2 + e3);
  return s;
}
__host__ __device__ __forceinline__ void add_to(Triple& s, float x) {
  float e1, e2;
  s.hi = two_sum(s.hi, x, e1);
  s.mid = two_sum(s.mid, e1, e2);
  s.lo += e2;
}
__device__ __forceinline__ double shfl_sum(double a, int mask) { return __shfl_xor_sync(0xffffffffu, a, mask); }
__device__ __forceinline__ Triple shfl_sum(Triple a, int mask) {
  Triple s;
  s.hi = __shfl_xor_sync(0xffffffffu, a.hi, mask);
  s.mid = __shfl_xor_sync(0xffffffffu, a.mid, mask);
  s.lo = __shfl_xor_sync(0xffffffffu, a.lo, mask);
  return s;
}
__host__ __device__ __forceinline__ double value_of(double a) { return a; }
__host__ __device__ __forceinline__ double value_of(Triple a) {
  return (double)a.hi + ((double)a.mid + (double)a.lo);
}

// s += <x, y>: term by term in FP64; of FP32 vectors a pack's products are summed in FP32 (pack.cuh), a single
// product is added exactly.
template <int PK>
__host__ __device__ __forceinline__ void add_products(double& s, const double (&x)[PK], const double (&y)[PK]) {
#pragma unroll
  for (int c = 0; c < PK; ++c) s = fma(x[c], y[c], s);
}
template <int PK>
__host__ __device__ __forceinline__ void add_products(Triple& s, const float (&x)[PK], const float (&y)[PK]) {
  float f = x[0] * y[0];
  if constexpr (PK == 1) {
    const float e = fmaf(x[0], y[0], -f);
    add_to(s, f);
    float e2;
    s.mid = two_sum(s.mid, e, e2);
    s.lo += e2;
  } else {
#pragma unroll
    for (int c = 1; c < PK; ++c) f = fmaf(x[c], y[c], f);
    add_to(s, f);
  }
}

// v[0..NV-1] summed over the warp: lane's result is sum lane / (32 / NV); NV 4, 8 or 16.
template <int NV, typename Sum>
__device__ __forceinline__ double warp_reduce_scatter(Sum (&v)[NV], int lane) {
  constexpr int LG = NV == 16 ? 4 : (NV == 8 ? 3 : 2);
#pragma unroll
  for (int r = 0; r < LG; ++r) {
    const bool up = (lane & (16 >> r)) != 0;
#pragma unroll
    for (int i = 0; i < NV / 2; ++i) {
      if (i < (NV >> (r + 1))) {
        const int o = NV >> (r + 1);
        const Sum send = up ? v[i] : v[i + o], keep = up ? v[i + o] : v[i];
        v[i] = add_sums(keep, shfl_sum(send, 16 >> r));
      }
    }
  }
  Sum x = v[0];
#pragma unroll
  for (int mask = 16 >> LG; mask > 0; mask >>= 1) x = add_sums(x, shfl_sum(x, mask));
  return value_of(x);
}

// One pack of a vector: four FP32 or two FP64 entries (one 16-byte access), or one entry.
template <typename T, int PK>
__device__ __forceinline__ void ld_pack(const T* p, long long e, T (&v)[PK]) {
  if constexpr (PK == 1) v[0] = p[e];
  else if constexpr (sizeof(T) == 4) {
    const float4 q = reinterpret_cast<const float4*>(p)[e];
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  } else {
    const double2 q = reinterpret_cast<const double2*>(p)[e];
    v[0] = q.x; v[1] = q.y;
  }
}
template <typename T, int PK>
__device__ __forceinline__ void st_pack(T* p, long long e, const T (&v)[PK]) {
  if constexpr (PK == 1) p[e] = v[0];
  else if constexpr (sizeof(T) == 4) reinterpret_cast<float4*>(p)[e] = make_float4(v[0], v[1], v[2], v[3]);
  else reinterpret_cast<double2*>(p)[e] = make_double2(v[0], v[1]);
}

// Pass b of step j: subtract block b (nu vectors, none in pass -1), form the inner products with block b + 1
// (nd vectors), or ||W||^2 after the last.
struct GsPass {
  int j, b, nu, nd;
  bool lastu, lastd;
  __device__ __forceinline__ GsPass(int j_, int b_) : j(j_), b(b_) {
    const int nblk = j / kGB + 1;
    nu = b >= 0 ? min(kGB, j + 1 - kGB * b) : 0;
    nd = b + 1 < nblk ? min(kGB, j + 1 - kGB * (b + 1)) : 0;
    lastu = b + 1 == nblk;
    lastd = b + 2 == nblk;
  }
};

// The coefficients h of block b from the previous pass's sums Pin[sum * ldp + c], c0 <= c < c1, by every CTA
// alike; the one with `writes` also keeps them (H column j) and V_j's Gram row.  VB: the most vectors of a block.
template <typename T, int VB>
__device__ __forceinline__ void gs_coefficients(const GsPass& g, const double* __restrict__ Pin, long long ldp, int c0,
                                                int c1, double* gram, double* Hj, bool writes, T (&h)[VB]) {
  if (!g.nu) {
#pragma unroll
    for (int q = 0; q < VB; ++q) h[q] = T(0);
    return;
  }
  __shared__ double sd[kGsSums], sh[kGB];
  const int t = threadIdx.x, lane = t & 31, wp = t >> 5, nw = blockDim.x >> 5;
  double* G = gram + (size_t)(kGB * g.b) * kGB;
  double row[kGB - 1];
  if (wp == 0) {
#pragma unroll
    for (int l = 0; l < kGB - 1; ++l)   // rows of earlier steps; V_j's is among the sums
      row[l] = lane < g.nu && l < lane && kGB * g.b + lane < g.j ? G[lane * kGB + l] : 0.0;
  }
  for (int q = wp; q < kGsSums; q += nw) {
    if (!(q < kGB ? q < g.nu : (g.lastu && q - kGB < g.nu - 1))) continue;
    double x = 0.0;
    for (int c = c0 + lane; c < c1; c += 32) x += Pin[q * ldp + c];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
    if (lane == 0) sd[q] = x;
  }
  __syncthreads();
  if (wp == 0) {
    double x = lane < g.nu ? sd[lane] : 0.0;
    if (g.lastu && lane == g.nu - 1) {
#pragma unroll
      for (int l = 0; l < kGB - 1; ++l) row[l] = l < lane ? sd[kGB + l] : 0.0;
      if (writes) {
#pragma unroll
        for (int l = 0; l < kGB - 1; ++l)
          if (l < lane) G[lane * kGB + l] = row[l];
      }
    }
    x = gs_forward(x, row, g.nu, lane);
    if (lane < g.nu) {
      sh[lane] = x;
      if (writes) Hj[kGB * g.b + lane] = x;
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < VB; ++q) h[q] = q < g.nu ? (T)sh[q] : T(0);
}

// A thread's sums of a pass.
template <typename T, int VB>
struct GsSums {
  using Sum = typename std::conditional<sizeof(T) == 8, double, Triple>::type;
  Sum v[2 * VB];
  double norm = 0.0;
  __device__ __forceinline__ GsSums() {
#pragma unroll
    for (int q = 0; q < 2 * VB; ++q) v[q] = Sum{};
  }
};

// One thread's packs of W, first, first + stride, ... < NP, of a pass.
// FP32 vectors: a pack's four products are summed in FP32 and such sums in Triples; a conversion and an FP64
// addition per eight products took half of the pass's time, and reducing FP64 sums over the block most of a
// batch's.  (Two FP32 parts, rounding in the second one, and groups of eight held 48 bits: n = s = 1024, p = 16
// BF16 solve 19.31 -> 19.36 ms, 64 uneven instances 20.43 -> 20.45; two sums to an f32x2 instruction 19.52 and
// 20.91.)  VB = 4 (the first steps) keeps twice the packs in flight.
template <typename T, int PK, int VB>
__device__ __forceinline__ void gs_stream(const GsPass& g, T* __restrict__ W, const T* __restrict__ V, long long ldv,
                                          long long first, long long NP, long long stride, const T (&h)[VB],
                                          GsSums<T, VB>& sums) {
  const int nu = g.nu, nd = g.nd;
  const bool lastd = g.lastd;
  const T *Vu = V + (long long)(kGB * max(g.b, 0)) * ldv, *Vd = V + (long long)(kGB * (g.b + 1)) * ldv;
  // packs in flight of each vector, and per round of the loop
  constexpr int UN = sizeof(T) == 4 ? 2 : 1, GR = VB == 4 ? 2 * UN : 1, NI = VB == 4 ? GR : UN;
  for (long long p0 = first; p0 < NP; p0 += NI * stride) {
#pragma unroll
    for (int u0 = 0; u0 < NI; u0 += GR) {
      T w[GR][PK], v[VB][GR][PK];
      bool in[GR];
#pragma unroll
      for (int u = 0; u < GR; ++u) {
        in[u] = p0 + (u0 + u) * stride < NP;
#pragma unroll
        for (int c = 0; c < PK; ++c) w[u][c] = T(0);
        if (in[u]) ld_pack<T, PK>(W, p0 + (u0 + u) * stride, w[u]);
      }
      const auto load = [&](const T* base, int count) {
#pragma unroll
        for (int q = 0; q < VB; ++q)
#pragma unroll
          for (int u = 0; u < GR; ++u) {
#pragma unroll
            for (int c = 0; c < PK; ++c) v[q][u][c] = T(0);
            if (q < count && in[u]) ld_pack<T, PK>(base + q * ldv, p0 + (u0 + u) * stride, v[q][u]);
          }
      };
      if (nu) {
        load(Vu, nu);
#pragma unroll
        for (int u = 0; u < GR; ++u) {
#pragma unroll
          for (int q = 0; q < VB; ++q)
            if (q < nu) {
#pragma unroll
              for (int c = 0; c < PK; ++c) w[u][c] = w[u][c] - h[q] * v[q][u][c];
            }
          if (in[u]) st_pack<T, PK>(W, p0 + (u0 + u) * stride, w[u]);
        }
      }
      if (nd) load(Vd, nd);
#pragma unroll
      for (int u = 0; u < GR; ++u) {
        if (nd) {
          T vj[PK];   // V_j where the block holds it, for its Gram row (again, from L1)
#pragma unroll
          for (int c = 0; c < PK; ++c) vj[c] = T(0);
          if (lastd && nd > 1 && in[u])
            ld_pack<T, PK>(Vd + (long long)(nd - 1) * ldv, p0 + (u0 + u) * stride, vj);
#pragma unroll
          for (int q = 0; q < VB; ++q)
            if (q < nd) add_products(sums.v[q], v[q][u], w[u]);
          if (lastd) {
#pragma unroll
            for (int q = 0; q < VB - 1; ++q)
              if (q < nd - 1) add_products(sums.v[VB + q], v[q][u], vj);
          }
        } else if constexpr (sizeof(T) == 8 || PK == 1) {
#pragma unroll
          for (int c = 0; c < PK; ++c) sums.norm = fma((double)w[u][c], (double)w[u][c], sums.norm);
        } else {   // no sum of squares beyond FP32's range
          sums.norm += (double)pack_dot(w[u], w[u]);
        }
      }
    }
  }
}

// The CTA's sums to Pout[sum * ldp + at].  blockDim.x <= 512.
template <typename T, int VB>
__device__ __forceinline__ void gs_store(const GsPass& g, GsSums<T, VB>& sums, double* __restrict__ Pout, long long ldp,
                                         long long at) {
  __shared__ double red[16][kGsSums];
  const int t = threadIdx.x, lane = t & 31, wp = t >> 5, nw = blockDim.x >> 5;
  if (!g.nd) {
    const double tot = block_sum(sums.norm);
    if (t == 0) Pout[at] = tot;
    return;
  }
  if (g.lastd) {
    const double x = warp_reduce_scatter<2 * VB>(sums.v, lane);
    if (lane % (16 / VB) == 0) red[wp][lane / (16 / VB)] = x;
  } else {
    typename GsSums<T, VB>::Sum a[VB];
#pragma unroll
    for (int q = 0; q < VB; ++q) a[q] = sums.v[q];
    const double x = warp_reduce_scatter<VB>(a, lane);
    if (lane % (32 / VB) == 0) red[wp][lane / (32 / VB)] = x;
  }
  __syncthreads();
  if (t < (g.lastd ? 2 * VB : VB)) {
    double x = 0.0;
    for (int q = 0; q < nw; ++q) x += red[q][t];
    Pout[(t < VB ? t : kGB + t - VB) * ldp + at] = x;
  }
}

}  // namespace ts
