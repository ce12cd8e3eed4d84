// Register-resident radix-2 FFT of a compile-time power-of-two length P <= 32, used for the DFT
// along mode 3 (one tube per thread).  The direct DFT costs P(P/2+1) complex multiply-adds per
// tube; this costs (P/2) log2 P butterflies, which moves the mode-3 transforms from instruction
// bound to HBM bound for the tube lengths of the workloads (p = 4 .. 32).
//
// A real tube of length P >= 4 is transformed as one complex tube of length M = P/2 (even samples
// as real parts, odd samples as imaginary parts) plus one combining pass (the standard two-for-one
// real FFT), about 40% fewer arithmetic instructions than a complex length-P FFT with zero
// imaginary parts.  That matters for FP64 tubes, which GB300's FP64 rate makes instruction bound.
//
// Convention (MATLAB's fft): forward X_k = sum_t x_t e^{-2 pi i k t / P}; the inverse is the sum with
// e^{+2 pi i k t / P}, times 1/P in FP64 and unnormalised in FP32 (the caller applies kIrfftScale).
//
// The twiddles are constants (cos and sin of multiples of pi/16).  As a table that every block computed with
// sincospi they cost 1.3 us at the start of a block, in FP64 instructions of one warp, whatever the tube
// type.  In FP64, whose instructions these kernels are bound by, the butterflies with twiddle (1 -+ i)/sqrt 2
// multiply sums of the two parts (6 instructions instead of 8) and the scale 1/P rides on constants and
// multiply-adds that are there anyway: 16 fewer instructions of ~115 for an inverse of 16 points.  FP64,
// 1024 x 1024 x 16: forward 208 -> 185 us, inverse 233 -> 186; 64 uneven instances: FP32 49 -> 31 and 48 -> 26.
#pragma once
#include <cuda_runtime.h>

namespace ts {

__host__ __device__ constexpr int ilog2c(int p) { return p <= 1 ? 0 : 1 + ilog2c(p / 2); }
__host__ __device__ constexpr int bitrevc(int x, int bits) {
  int r = 0;
  for (int b = 0; b < bits; ++b) r = (r << 1) | ((x >> b) & 1);
  return r;
}

// cos(2 pi r / 32) and sin(2 pi r / 32), correctly rounded; 32 r / P for the P-th roots of unity.
__host__ __device__ constexpr double cos32(int r) {
  const double t[9] = {1.0, 0.98078528040323044913, 0.92387953251128675613, 0.83146961230254523708,
                       0.70710678118654752440, 0.55557023301960222474, 0.38268343236508977173,
                       0.19509032201612826785, 0.0};
  r &= 31;
  if (r > 16) r = 32 - r;
  return r > 8 ? -t[16 - r] : t[r];
}
__host__ __device__ constexpr double sin32(int r) { return cos32(r + 24); }
template <typename Real, int P>
__host__ __device__ constexpr Real kIrfftScale() { return sizeof(Real) == 8 ? Real(1) : Real(1) / Real(P); }
// Roots of unity for direct sums, cos and sin of 2 pi r / p for r < p, by threads t < nt of a block (a multiple
// of 64).  Even warps take the cosines and odd ones the sines: one warp's sincospi is twice the chain of FP64
// instructions (64 clocks each), and every block waits for it.
template <typename Real>
__device__ __forceinline__ void fill_roots(Real* c, Real* s, int p, int t, int nt) {
  for (int r = (t >> 6) * 32 + (t & 31); r < p; r += nt / 2) {
    if (t & 32) s[r] = (Real)sinpi(2.0 * r / p);
    else c[r] = (Real)cospi(2.0 * r / p);
  }
}

// a b + c d and a b - c d with the rounding written out: the second product is rounded, the first is not.
// Left to the compiler the choice changes with what it knows about the constants, and an FP32 transform that
// feeds BF16 operands has to give the same bits everywhere.
template <typename Real>
__device__ __forceinline__ Real mul2_add(Real a, Real b, Real c, Real d) {
  if constexpr (sizeof(Real) == 8) return __fma_rn(a, b, __dmul_rn(c, d));
  else return __fmaf_rn(a, b, __fmul_rn(c, d));
}
template <typename Real>
__device__ __forceinline__ Real mul2_sub(Real a, Real b, Real c, Real d) {
  if constexpr (sizeof(Real) == 8) return __fma_rn(a, b, -__dmul_rn(c, d));
  else return __fmaf_rn(a, b, -__fmul_rn(c, d));
}

// One radix-2 stage of span LEN, then the next; LEN is a template argument so that every register
// index is a compile-time constant (a runtime stage loop leaves the arrays in local memory).
template <typename Real, int P, bool INVERSE, int LEN>
struct FftStages {
  template <int Q, int START>
  static __device__ __forceinline__ void butterfly(Real (&xr)[P], Real (&xi)[P]) {
    constexpr int half = LEN / 2, a = START + Q, b = START + Q + half, root = Q * (32 / LEN);
    Real vr, vi;
    if constexpr (Q == 0) {                       // twiddle 1
      vr = xr[b];
      vi = xi[b];
    } else if constexpr (4 * Q == LEN) {          // twiddle -+i
      vr = INVERSE ? -xi[b] : xi[b];
      vi = INVERSE ? xr[b] : -xr[b];
    } else if constexpr (sizeof(Real) == 8 && (8 * Q == LEN || 8 * Q == 3 * LEN)) {   // (+-1 -+ i) / sqrt 2
      // forward: v = h (sum, dif), then h (dif, -sum); inverse: h (dif, sum), then h (-sum, dif)
      constexpr bool q1 = 8 * Q == LEN;
      constexpr Real h = Real(cos32(4)), cr = INVERSE && !q1 ? -h : h, ci = !INVERSE && !q1 ? -h : h;
      const Real sum = xr[b] + xi[b], dif = INVERSE ? xr[b] - xi[b] : xi[b] - xr[b];
      const Real pr = q1 != INVERSE ? sum : dif, pi = q1 != INVERSE ? dif : sum;
      xr[b] = fma(-cr, pr, xr[a]);
      xi[b] = fma(-ci, pi, xi[a]);
      xr[a] = fma(cr, pr, xr[a]);
      xi[a] = fma(ci, pi, xi[a]);
      return;
    } else {
      constexpr Real wr = Real(cos32(root)), si = Real(sin32(root));
      vr = INVERSE ? mul2_sub(xr[b], wr, xi[b], si) : mul2_add(xr[b], wr, xi[b], si);
      vi = INVERSE ? mul2_add(xr[b], si, xi[b], wr) : mul2_sub(xi[b], wr, xr[b], si);
    }
    xr[b] = xr[a] - vr;
    xi[b] = xi[a] - vi;
    xr[a] = xr[a] + vr;
    xi[a] = xi[a] + vi;
  }
  template <int I>   // butterflies I .. P/2 - 1: group by group
  static __device__ __forceinline__ void all(Real (&xr)[P], Real (&xi)[P]) {
    if constexpr (I < P / 2) {
      butterfly<I % (LEN / 2), (I / (LEN / 2)) * LEN>(xr, xi);
      all<I + 1>(xr, xi);
    }
  }
  static __device__ __forceinline__ void run(Real (&xr)[P], Real (&xi)[P]) {
    all<0>(xr, xi);
    FftStages<Real, P, INVERSE, 2 * LEN>::run(xr, xi);
  }
};
template <typename Real, int P, bool INVERSE>
struct FftStages<Real, P, INVERSE, 2 * P> {
  static __device__ __forceinline__ void run(Real (&)[P], Real (&)[P]) {}
};

// In-place decimation-in-time FFT; the inputs must already sit in bit-reversed order.
template <typename Real, int P, bool INVERSE>
__device__ __forceinline__ void fft_bitrev_inplace(Real (&xr)[P], Real (&xi)[P]) {
  FftStages<Real, P, INVERSE, 2>::run(xr, xi);
}

// Forward transform of P real samples read by `load(t)`; writes the P/2+1 non-redundant outputs
// through `store(k, re, im)`.
//
// Two-for-one (P >= 4): z_t = x_2t + i x_2t+1, Z = DFT_M(z).  With E_k, O_k the length-M DFTs of the
// even and odd samples, Z_k = E_k + i O_k and conj(Z_M-k) = E_k - i O_k, so
// E_k = (Z_k + conj Z_M-k)/2, O_k = (Z_k - conj Z_M-k)/(2i) and X_k = E_k + w^k O_k,
// X_M-k = conj(E_k) - conj(w^k O_k), w = e^{-2 pi i/P}; X_0 = Re Z_0 + Im Z_0, X_M = Re Z_0 - Im Z_0
// and X_M/2 = conj Z_M/2.
template <typename Real, int P, typename Load, typename Store>
__device__ __forceinline__ void rfft_reg(Load load, Store store) {
  if constexpr (P < 4) {
    constexpr int LB = ilog2c(P);
    Real xr[P], xi[P];
#pragma unroll
    for (int t = 0; t < P; ++t) {
      xr[bitrevc(t, LB)] = load(t);
      xi[bitrevc(t, LB)] = Real(0);
    }
    fft_bitrev_inplace<Real, P, false>(xr, xi);
#pragma unroll
    for (int k = 0; k <= P / 2; ++k) store(k, xr[k], (k == 0 || k == P / 2) ? Real(0) : xi[k]);
  } else {
    constexpr int M = P / 2, LB = ilog2c(M);
    Real zr[M], zi[M];
#pragma unroll
    for (int t = 0; t < M; ++t) {
      zr[bitrevc(t, LB)] = load(2 * t);
      zi[bitrevc(t, LB)] = load(2 * t + 1);
    }
    FftStages<Real, M, false, 2>::run(zr, zi);
    store(0, zr[0] + zi[0], Real(0));
    store(M, zr[0] - zi[0], Real(0));
#pragma unroll
    for (int k = 1; 2 * k <= M; ++k) {
      if (2 * k == M) {
        store(k, zr[k], -zi[k]);
      } else {
        const Real s1 = zr[k] + zr[M - k], s2 = zi[k] - zi[M - k];
        const Real s3 = zi[k] + zi[M - k], s4 = zr[M - k] - zr[k];
        const Real hc = Real(0.5) * Real(cos32(k * (32 / P))), hs = Real(0.5) * Real(sin32(k * (32 / P)));
        const Real u = mul2_add(hc, s3, hs, s4), v = mul2_sub(hc, s4, hs, s3);
        store(k, Real(0.5) * s1 + u, Real(0.5) * s2 + v);
        store(M - k, Real(0.5) * s1 - u, v - Real(0.5) * s2);
      }
    }
  }
}

// Inverse of a Hermitian half spectrum c_0..c_{P/2} read by `load(k, re, im)`: writes the P real
// samples (FP32: times P) through `store(t, value)`.  Imaginary parts of c_0 and c_{P/2}
// are ignored (they are zero for the spectrum of a real tensor).
//
// Two-for-one (P >= 4), the forward steps reversed: Z'_k = (c_k + conj c_M-k) +
// i (c_k - conj c_M-k) w^-k (= 2 Z_k), and the unnormalised inverse DFT_M of Z' is P z, so
// x_2t = Re and x_2t+1 = Im of its entry t.
template <typename Real, int P, typename Load, typename Store>
__device__ __forceinline__ void irfft_reg(Load load, Store store) {
  constexpr Real scale = Real(1) / (kIrfftScale<Real, P>() * Real(P));   // FP64: 1/P; FP32: 1
  if constexpr (P < 4) {
    constexpr int LB = ilog2c(P);
    Real xr[P], xi[P];
#pragma unroll
    for (int k = 0; k <= P / 2; ++k) {
      Real re, im;
      load(k, re, im);
      if (k == 0 || k == P / 2) im = Real(0);
      xr[bitrevc(k, LB)] = re;
      xi[bitrevc(k, LB)] = im;
      if (k > 0 && k < P / 2) {
        xr[bitrevc(P - k, LB)] = re;
        xi[bitrevc(P - k, LB)] = -im;
      }
    }
    fft_bitrev_inplace<Real, P, true>(xr, xi);
#pragma unroll
    for (int t = 0; t < P; ++t) store(t, sizeof(Real) == 8 ? scale * xr[t] : xr[t]);
  } else {
    constexpr int M = P / 2, LB = ilog2c(M);
    Real zr[M], zi[M];
    {
      Real a, b, c, d;
      load(0, a, b);
      load(M, c, d);
      zr[0] = a + c;
      zi[0] = a - c;
      if (sizeof(Real) == 8) {
        zr[0] *= scale;
        zi[0] *= scale;
      }
    }
#pragma unroll
    for (int k = 1; 2 * k <= M; ++k) {
      Real a, b;
      load(k, a, b);
      if (2 * k == M) {
        zr[bitrevc(k, LB)] = Real(2) * scale * a;
        zi[bitrevc(k, LB)] = Real(-2) * scale * b;
      } else {
        Real c, d;
        load(M - k, c, d);
        const Real s1 = a + c, s2 = b - d, s3 = b + d, s4 = c - a;
        const Real co = scale * Real(cos32(k * (32 / P))), si = scale * Real(sin32(k * (32 / P)));
        const Real pp = -mul2_add(s4, co, s3, si), qq = mul2_sub(s3, co, s4, si);
        if constexpr (sizeof(Real) == 8) {
          zr[bitrevc(k, LB)] = fma(scale, s1, -qq);
          zi[bitrevc(k, LB)] = fma(scale, s2, pp);
          zr[bitrevc(M - k, LB)] = fma(scale, s1, qq);
          zi[bitrevc(M - k, LB)] = fma(-scale, s2, pp);
        } else {
          zr[bitrevc(k, LB)] = s1 - qq;
          zi[bitrevc(k, LB)] = s2 + pp;
          zr[bitrevc(M - k, LB)] = s1 + qq;
          zi[bitrevc(M - k, LB)] = pp - s2;
        }
      }
    }
    FftStages<Real, M, true, 2>::run(zr, zi);
#pragma unroll
    for (int t = 0; t < M; ++t) {
      store(2 * t, zr[t]);
      store(2 * t + 1, zi[t]);
    }
  }
}

// Direct DFT of p <= PMAX real samples, p any: the outputs k0, k0 + ks, ... of the p/2+1 non-redundant ones.
// x_t and x_p-t meet the same cosine and opposite sines, so their sum and difference are formed once and a
// multiply-add serves both: half of a term-by-term sum's.  c(r), s(r): cos and sin of 2 pi r / p.
template <typename Real, int PMAX, typename Load, typename Store, typename Cos, typename Sin>
__device__ __forceinline__ void rfft_direct(Load load, Store store, int p, int k0, int ks, Cos c, Sin s) {
  constexpr int H = PMAX / 2;
  const int K = p / 2 + 1, h = (p - 1) / 2;
  Real sum[H + 1], dif[H + 1];
  const Real x0 = load(0), xm = p % 2 == 0 ? load(p / 2) : Real(0);
#pragma unroll
  for (int t = 1; t <= H; ++t) {
    const Real a = t <= h ? load(t) : Real(0), b = t <= h ? load(p - t) : Real(0);
    sum[t] = a + b;
    dif[t] = b - a;
  }
#pragma unroll 1
  for (int k = k0; k < K; k += ks) {
    Real re = k & 1 ? x0 - xm : x0 + xm, im = 0;
    int r = 0;
#pragma unroll
    for (int t = 1; t <= H; ++t) {
      if (t <= h) {
        r += k;
        if (r >= p) r -= p;
        re = fma(sum[t], c(r), re);
        im = fma(dif[t], s(r), im);
      }
    }
    store(k, re, im);
  }
}

// The inverse from p/2+1 coefficients, times p: the outputs t and p - t of t0 <= t < t0 + NO, t <= p/2.
template <typename Real, int NO, typename Load, typename Store, typename Cos, typename Sin>
__device__ __forceinline__ void irfft_direct(Load load, Store store, int p, int t0, Cos c, Sin s) {
  const int K = p / 2 + 1, nyq = p % 2 == 0 ? p / 2 : -1;
  Real a[NO], b[NO];
#pragma unroll
  for (int u = 0; u < NO; ++u) a[u] = b[u] = Real(0);
  Real next_re, next_im;
  load(0, next_re, next_im);
  int r0 = 0;   // k t0 mod p
#pragma unroll 1
  for (int k = 0; k < K; ++k) {
    const Real re = next_re, im = next_im;
    if (k + 1 < K) load(k + 1, next_re, next_im);   // one coefficient ahead
    const bool real = k == 0 || k == nyq;
    const Real cr = real ? re : Real(2) * re, ci = real ? Real(0) : Real(2) * im;
    int r = r0;
#pragma unroll
    for (int u = 0; u < NO; ++u) {
      if (t0 + u < K) {
        a[u] = fma(cr, c(r), a[u]);
        b[u] = fma(ci, s(r), b[u]);
        r += k;
        if (r >= p) r -= p;
      }
    }
    r0 += t0;
    if (r0 >= p) r0 -= p;
  }
#pragma unroll
  for (int u = 0; u < NO; ++u) {
    const int t = t0 + u;
    if (t < K) {
      if (t == 0 || 2 * t == p) {
        store(t, a[u]);
      } else {
        store(t, a[u] - b[u]);
        store(p - t, a[u] + b[u]);
      }
    }
  }
}

}  // namespace ts
