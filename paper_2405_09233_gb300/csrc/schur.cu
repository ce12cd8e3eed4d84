// Complex Schur form B_k = Q T Q^H of the small s x s Fourier slices of B (t-Bartels-Stewart,
// Algorithm 4 read with a complex Schur form per slice; and the projected equation of TBAS): one CTA
// per slice, Householder reduction to upper Hessenberg form, then implicitly shifted single-shift QR
// with Wilkinson shifts and deflation, T and Q in shared memory while they fit.
//
// What bounds it: a chain of dependent FP64 instructions.  GB300 spends 64 clocks on an FP64
// instruction of one warp, however few of its lanes are active, so a QR sweep costs its rotations
// times the instructions between one rotation and the next.  Two things follow:
//  * the chase belongs to one warp whose lanes each form one real scalar of the 3 x 2 window around
//    the bulge (three instructions for the row rotation, three for the column rotation, then the next
//    Givens rotation from one reciprocal square root): ~18 dependent instructions per rotation, where
//    a thread forming the window's complex numbers one after the other issues ~150;
//  * everything else a rotation touches (the rest of its two rows, of its two columns, and Q) goes to
//    the warps of the other three sub-partitions in the same interval, one element pair per lane, so
//    that one barrier per rotation is the only wait.
// Dependences of interval i (rotation i known at its start): the window rows i..i+2 x columns i, i+1
// is the chase's; the row rotation on columns >= i+2 and the column rotation on rows < i touch
// disjoint entries, which interval i-1 has finished.  The chase needs T(i, i+1) after row rotation
// i-1, which interval i-1 applied to columns >= i+1.
// Measured: s = 64, 5 slices 54.0 -> 9.6 ms (one warp on global memory before, Givens reduction to Hessenberg
// form, every modulus by hypot).
#include <cfloat>
#include "internal.cuh"
#include "complex_ops.cuh"
#include "tba.cuh"

namespace ts {
namespace {

constexpr int kSchurThreads = 256;
constexpr int kSchurWorkers = 192;   // warps 1-3 and 5-7: sub-partition 0 is left to the chase (warp 0)

// Givens rotation G = [[c, s], [-conj(s), c]] (c real) with G [a; b] = [r; 0], for entries whose
// squares leave the FP64 range (the chase forms the others from one reciprocal square root).
__device__ __noinline__ void givens_safe(double2 a, double2 b, double& c, double2& s, double2& r) {
  const double na = cabs2(a), nb = cabs2(b);
  if (nb == 0.0) {
    c = 1.0;
    s = make_double2(0.0, 0.0);
    r = a;
    return;
  }
  if (na == 0.0) {
    c = 0.0;
    s = make_double2(b.x / nb, -b.y / nb);   // G [0; b] = [s b; c b] = [|b|; 0]
    r = make_double2(nb, 0.0);
    return;
  }
  // quotients, not reciprocals: the reciprocal of a subnormal modulus overflows
  const double nr = hypot(na, nb);
  c = na / nr;
  const double2 ua = make_double2(a.x / na, a.y / na);
  s = cmul(ua, make_double2(b.x / nr, -b.y / nr));
  r = cscale(ua, nr);
}

// Principal square root of z with |z| = r > 0: the smaller component as Im z / (2 larger), no cancellation.
__device__ __forceinline__ double2 principal_root(double2 z, double r) {
  const double t = sqrt(0.5 * (r + fabs(z.x))), o = z.y / (2.0 * t);
  return z.x >= 0.0 ? make_double2(t, o) : make_double2(fabs(o), z.y < 0.0 ? -t : t);
}

// The Wilkinson shift of [[a, b], [cc, d]] (see the sweep) when squares of its entries leave the FP64 range: the
// block is scaled by a power of two first, moduli are taken by hypot and the quotient by Smith's division.
__device__ __noinline__ double2 shift_safe(double2 a, double2 b, double2 cc, double2 d) {
  double2 half = csub(a, d);
  const double m = fmax(fmax(fmax(fabs(half.x), fabs(half.y)), fmax(fabs(b.x), fabs(b.y))),
                        fmax(fabs(cc.x), fabs(cc.y)));
  if (!(m > 0.0 && m <= DBL_MAX)) return d;
  const int e = ilogb(m);
  auto scaled = [](double2 z, int q) { return make_double2(scalbn(z.x, q), scalbn(z.y, q)); };
  half = scaled(half, -e - 1);
  const double2 bc = cmul(scaled(b, -e), scaled(cc, -e)), z = cadd(cmul(half, half), bc);
  const double r = cabs2(z);
  double2 sq = r > 0.0 ? principal_root(z, r) : make_double2(0.0, 0.0);
  if (fma(half.y, sq.y, half.x * sq.x) < 0.0) sq = make_double2(-sq.x, -sq.y);
  const double2 den = cadd(half, sq);
  if (den.x == 0.0 && den.y == 0.0) return d;
  return csub(d, scaled(cdiv(bc, den), e));
}

__device__ __forceinline__ double shfl_d(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }

// One rotation: c, s and the value r it leaves on the subdiagonal.
struct Rot {
  double c, sr, si, rr, ri;
};

// The rotation that maps (x, y) to (r, 0), by all lanes of a warp; every lane holds x and y and gets
// the whole result.  With f2 = |x|^2, h2 = f2 + |y|^2 and d = 1 / sqrt(f2 h2): c = f2 d,
// s = x conj(y) d, r = h2 d x.  Lane roles: 0 c, 1 and 2 s, 3 and 4 r.
__device__ __forceinline__ Rot make_rot(double2 x, double2 y, int lane) {
  const bool odd = lane & 1;
  const double vr = odd ? y.x : x.x, vi = odd ? y.y : x.y;
  const double n2 = fma(vi, vi, vr * vr);
  const double h2 = n2 + __shfl_xor_sync(0xffffffffu, n2, 1);
  const double f2 = shfl_d(n2, 0);
  const double prod = f2 * h2;
  Rot q;
  if (prod >= 1e-280 && prod <= 1e280) {   // uniform: every lane holds the same f2 and h2
    const double d = rsqrt(prod);
    const double u = lane == 0 ? f2 : (lane == 2 ? x.y : (lane == 4 ? x.y : x.x));
    const double v = lane == 0 ? 1.0 : (lane <= 2 ? y.x : h2);
    const double a = lane == 1 ? x.y : (lane == 2 ? -x.x : 0.0);
    const double m = fma(a, y.y, u * v) * d;
    q.c = shfl_d(m, 0);
    q.sr = shfl_d(m, 1);
    q.si = shfl_d(m, 2);
    q.rr = shfl_d(m, 3);
    q.ri = shfl_d(m, 4);
  } else {
    double c;
    double2 s, r;
    givens_safe(x, y, c, s, r);
    q = Rot{c, s.x, s.y, r.x, r.y};
  }
  return q;
}

// Rows: (p, q) -> (c p + s q, c q - conj(s) p).
__device__ __forceinline__ void rot_row(double2& p, double2& q, double c, double sr, double si) {
  const double2 a = p, b = q;
  p.x = fma(-si, b.y, fma(sr, b.x, c * a.x));
  p.y = fma(si, b.x, fma(sr, b.y, c * a.y));
  q.x = fma(-si, a.y, fma(-sr, a.x, c * b.x));
  q.y = fma(si, a.x, fma(-sr, a.y, c * b.y));
}
// Columns (right multiplication by G^H): (p, q) -> (c p + conj(s) q, c q - s p).
__device__ __forceinline__ void rot_col(double2& p, double2& q, double c, double sr, double si) {
  rot_row(p, q, c, sr, -si);
}

__device__ __forceinline__ double cabs1(double2 z) { return fabs(z.x) + fabs(z.y); }

// B (s x s, column-major, in Tall) = Q T Q^H, one CTA per matrix.  ts_in / qs_in: keep T / Q in shared
// memory (leading dimension s + 1); otherwise they are worked on in global memory.  err bit 1 on
// failure to converge.
__global__ void __launch_bounds__(kSchurThreads)
    k_schur_small(double2* __restrict__ Tall, double2* __restrict__ Qall, int s, int* err, int ts_in, int qs_in) {
  extern __shared__ double2 sch_smem[];
  double2* Tg = Tall + (long long)blockIdx.x * s * s;
  double2* Qg = Qall + (long long)blockIdx.x * s * s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long lt = ts_in ? s + 1 : s, lq = qs_in ? s + 1 : s;
  double2* T = ts_in ? sch_smem : Tg;
  double2* Q = qs_in ? sch_smem + (ts_in ? (long long)s * lt : 0) : Qg;
  __shared__ Rot rot[2];
  __shared__ double sred[kSchurThreads / 32];
  __shared__ double2 sbc[2];     // Householder: leading entry of v; sweep: shift
  __shared__ int sint[2];        // window [lo, hi] of the sweep
  // The matrix is scaled by a power of two to max(|Re|, |Im|) in [1/2, 1), so that squares of the
  // entries that matter stay in range; exact, and undone at the end.
  double mx = 0.0;
  int bad = 0;
  for (long long e = tid; e < (long long)s * s; e += kSchurThreads) {
    const double2 v = Tg[e];
    mx = fmax(mx, fmax(fabs(v.x), fabs(v.y)));
    bad |= !(fabs(v.x) <= DBL_MAX && fabs(v.y) <= DBL_MAX);
  }
  if (__syncthreads_or(bad) && s > 1) {   // NaN or Inf: no Schur form
    if (tid == 0) atomicOr(err, 1);
    return;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) sred[warp] = mx;
  __syncthreads();
  mx = 0.0;
  for (int w = 0; w < kSchurThreads / 32; ++w) mx = fmax(mx, sred[w]);
  const int ex = (mx > 0.0 && mx <= DBL_MAX) ? ilogb(mx) + 1 : 0;
  for (long long e = tid; e < (long long)s * s; e += kSchurThreads) {
    const int r = (int)(e % s);
    const long long q = e / s;
    const double2 v = Tg[e];
    T[r + lt * q] = make_double2(scalbn(v.x, -ex), scalbn(v.y, -ex));
    Q[r + lq * q] = make_double2(r == q ? 1.0 : 0.0, 0.0);
  }
  __syncthreads();

  // Upper Hessenberg form: for column c the reflection I - tau v v^H (tau real) maps
  // x = T(c+1.., c) to -e^{i arg x_0} ||x|| e_1, v = x + e^{i arg x_0} ||x|| e_1,
  // tau = 1 / (||x||^2 + |x_0| ||x||).  Four lanes share a column (left) or a row (right).
  for (int c = 0; c + 2 < s; ++c) {
    double2* xc = T + lt * c;
    double n2 = 0.0;   // below the leading entry
    if (warp == 0) {
      for (int r = c + 2 + lane; r < s; r += 32) n2 = fma(xc[r].y, xc[r].y, fma(xc[r].x, xc[r].x, n2));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, o);
      if (lane == 0) {
        const double2 x0 = xc[c + 1];
        const double a2 = fma(x0.y, x0.y, x0.x * x0.x), nx = sqrt(n2 + a2), ax = sqrt(a2);
        const double2 ph = ax > 0.0 ? make_double2(x0.x / ax, x0.y / ax) : make_double2(1.0, 0.0);
        sbc[0] = make_double2(fma(ph.x, nx, x0.x), fma(ph.y, nx, x0.y));   // v_0
        sbc[1] = make_double2(-ph.x * nx, -ph.y * nx);                     // the new T(c+1, c)
        sred[0] = n2;
        sred[1] = n2 > 0.0 ? 1.0 / (n2 + a2 + ax * nx) : 0.0;              // tau
      }
    }
    __syncthreads();
    const double tau = sred[1];
    const bool skip = !(sred[0] > 0.0) || !(tau <= DBL_MAX);   // already Hessenberg here (or below FP64's range)
    const double2 v0 = sbc[0], b0 = sbc[1];
    if (!skip) {   // uniform over the CTA
      const int sub = tid & 3;
      auto vat = [&](int r) { return r == c + 1 ? v0 : xc[r]; };
      for (int q0 = c + 1 + (tid >> 2); q0 < ((s - c - 1 + 63) / 64) * 64 + c + 1; q0 += kSchurThreads / 4) {   // T <- H T
        const bool live = q0 < s;
        double2* col = T + lt * (live ? q0 : c + 1);
        double2 w = make_double2(0.0, 0.0);
        for (int r = c + 1 + sub; live && r < s; r += 4) {
          const double2 v = vat(r), t = col[r];
          w.x = fma(v.y, t.y, fma(v.x, t.x, w.x));
          w.y = fma(-v.y, t.x, fma(v.x, t.y, w.y));
        }
#pragma unroll
        for (int o = 1; o <= 2; o <<= 1) {
          w.x += __shfl_xor_sync(0xffffffffu, w.x, o);
          w.y += __shfl_xor_sync(0xffffffffu, w.y, o);
        }
        w.x *= tau;
        w.y *= tau;
        for (int r = c + 1 + sub; live && r < s; r += 4) {
          const double2 v = vat(r), t = col[r];
          col[r] = make_double2(fma(v.y, w.y, fma(-v.x, w.x, t.x)), fma(-v.y, w.x, fma(-v.x, w.y, t.y)));
        }
      }
      __syncthreads();
      for (int r0 = tid >> 2; r0 < ((2 * s + 63) / 64) * 64; r0 += kSchurThreads / 4) {   // T <- T H, Q <- Q H
        const bool live = r0 < 2 * s;
        double2* M = r0 < s ? T : Q;
        const long long ld = r0 < s ? lt : lq;
        const int r = live ? (r0 < s ? r0 : r0 - s) : 0;
        double2 u = make_double2(0.0, 0.0);
        for (int q = c + 1 + sub; live && q < s; q += 4) {
          const double2 v = vat(q), t = M[r + ld * q];
          u.x = fma(-t.y, v.y, fma(t.x, v.x, u.x));
          u.y = fma(t.y, v.x, fma(t.x, v.y, u.y));
        }
#pragma unroll
        for (int o = 1; o <= 2; o <<= 1) {
          u.x += __shfl_xor_sync(0xffffffffu, u.x, o);
          u.y += __shfl_xor_sync(0xffffffffu, u.y, o);
        }
        u.x *= tau;
        u.y *= tau;
        for (int q = c + 1 + sub; live && q < s; q += 4) {
          const double2 v = vat(q), t = M[r + ld * q];   // t - u conj(v)
          M[r + ld * q] =
              make_double2(fma(-u.y, v.y, fma(-u.x, v.x, t.x)), fma(u.x, v.y, fma(-u.y, v.x, t.y)));
        }
      }
      __syncthreads();
      for (int r = c + 1 + tid; r < s; r += kSchurThreads) xc[r] = r == c + 1 ? b0 : make_double2(0.0, 0.0);
    } else {
      __syncthreads();   // sred and sbc are rewritten by the next column
      for (int r = c + 2 + tid; r < s; r += kSchurThreads) xc[r] = make_double2(0.0, 0.0);
    }
    __syncthreads();
  }

  // Shifted QR on the active window [lo, hi].
  const double eps = 2.220446049250313e-16;
  int hi = s - 1, iter = 0, since = 0;
  const int max_iter = 60 * s + 60;
  while (hi > 0) {
    if (warp == 0) {
      // lo: the highest l <= hi whose subdiagonal entry T(l, l-1) is negligible (0 when there is none)
      int lo = 0;
      for (int base = hi; base > 0; base -= 32) {
        const int l = base - lane;
        bool small = false;
        if (l > 0) {
          const double2 sub = T[l + lt * (l - 1)];
          double scale = cabs1(T[l + lt * l]) + cabs1(T[l - 1 + lt * (l - 1)]);
          if (scale == 0.0) scale = 1.0;
          small = cabs1(sub) <= eps * scale;
        }
        const unsigned hit = __ballot_sync(0xffffffffu, small);
        if (hit) {
          lo = base - (__ffs(hit) - 1);
          break;
        }
      }
      if (lane == 0) {
        if (lo > 0) T[lo + lt * (lo - 1)] = make_double2(0.0, 0.0);
        sint[0] = lo;
      }
      __syncwarp();
      if (lo < hi) {
        // Wilkinson shift: the eigenvalue of the trailing 2 x 2 block of the window closer to its
        // last entry, mu = d - bc / (half +- sqrt(half^2 + bc)) with the sign of the larger denominator
        const double2 a = T[hi - 1 + lt * (hi - 1)], b = T[hi - 1 + lt * hi];
        const double2 cc = T[hi + lt * (hi - 1)], d = T[hi + lt * hi];
        double2 mu;
        if ((since + 1) % 11 == 10) {   // exceptional shift
          mu = cadd(d, make_double2(cabs2(cc), 0.0));
        } else {
          const double2 half = cscale(csub(a, d), 0.5), bc = cmul(b, cc);
          const double2 z = cadd(cmul(half, half), bc);
          const double r2 = fma(z.y, z.y, z.x * z.x);
          if (r2 >= 1e-280) {   // |sq| >= 1e-70, and |den| >= |sq|
            double2 sq = principal_root(z, sqrt(r2));
            if (fma(half.y, sq.y, half.x * sq.x) < 0.0) sq = make_double2(-sq.x, -sq.y);
            const double2 den = cadd(half, sq);
            mu = csub(d, cscale(cmul(bc, cconj(den)), 1.0 / fma(den.y, den.y, den.x * den.x)));
          } else {
            mu = shift_safe(a, b, cc, d);
          }
        }
        const double2 x = csub(T[lo + lt * lo], mu), y = T[lo + 1 + lt * lo];
        const Rot q = make_rot(x, y, lane);
        if (lane == 0) rot[lo & 1] = q;
      }
    }
    __syncthreads();
    const int lo = sint[0];
    __syncthreads();   // sint is rewritten by warp 0 of the next pass
    if (lo == hi) {
      --hi;
      since = 0;
      continue;
    }
    if (iter++ > max_iter) {
      if (tid == 0) atomicOr(err, 1);
      break;
    }
    ++since;
    for (int i = lo; i < hi; ++i) {
      const Rot g = rot[i & 1];
      if (warp == 0) {
        const bool has2 = i + 2 <= hi;      // row i+2 is in the window
        // row rotation on columns i, i+1: lane 2o + part forms entry o (0: (i,i), 1: (i+1,i), 2: (i,i+1),
        // 3: (i+1,i+1))
        const int part = lane & 1, o = (lane >> 1) & 3;
        const double2 p = T[i + lt * (i + (o >> 1))], q = T[i + 1 + lt * (i + (o >> 1))];
        const bool top = !(o & 1);
        const double2 A = top ? p : q, B = top ? q : p;
        const double sgr = top ? g.sr : -g.sr;
        const double sgi = part ? g.si : -g.si;
        const double v = fma(sgi, part ? B.x : B.y, fma(sgr, part ? B.y : B.x, g.c * (part ? A.y : A.x)));
        // column rotation on rows i, i+1, i+2: lane 4 row + 2 col + part; row i+2 is (0, T(i+2, i+1))
        const int row = min(lane >> 2, 2), cl = (lane >> 1) & 1;
        const int e0 = 2 * min(row, 1), e1 = e0 + 4;   // lanes of (row, column i) and (row, column i+1), Re parts
        double2 P, R;
        P.x = shfl_d(v, e0);
        P.y = shfl_d(v, e0 + 1);
        R.x = shfl_d(v, e1);
        R.y = shfl_d(v, e1 + 1);
        if (row == 2) {
          P = make_double2(0.0, 0.0);
          R = has2 ? T[i + 2 + lt * (i + 1)] : make_double2(0.0, 0.0);
        }
        // column i: c P + conj(s) R; column i+1: c R - s P
        const double2 A2 = cl ? R : P, B2 = cl ? P : R;
        const double tsr = cl ? -g.sr : g.sr;
        const double tsi = part ? -g.si : g.si;
        const double w = fma(tsi, part ? B2.x : B2.y, fma(tsr, part ? B2.y : B2.x, g.c * (part ? A2.y : A2.x)));
        // (i+1, i) and (i+2, i) become the next rotation's x and y; the rest of the window is stored
        const double2 x = make_double2(shfl_d(w, 4), shfl_d(w, 5)), y = make_double2(shfl_d(w, 8), shfl_d(w, 9));
        if (lane < 12 && (row < 2 || has2)) {
          double* dst = reinterpret_cast<double*>(T + (i + row) + lt * (i + cl)) + part;
          if (!(row == 2 && cl == 0)) *dst = w;
        }
        if (lane == 12 && i > lo) {   // what rotation i left in column i-1
          T[i + lt * (i - 1)] = make_double2(g.rr, g.ri);
        }
        if (i + 1 < hi) {
          const Rot nx = make_rot(x, y, lane);
          if (lane == 0) rot[(i + 1) & 1] = nx;
        }
      } else if (warp != 4) {
        const int id = tid - (warp > 4 ? 64 : 32);
        const int nR = max(0, s - (i + 2)), nC = i, tot = nR + nC + s;
        for (int e = id; e < tot; e += kSchurWorkers) {
          if (e < nR) {
            double2* a = T + i + lt * (i + 2 + e);
            double2 p = a[0], q = a[1];
            rot_row(p, q, g.c, g.sr, g.si);
            a[0] = p;
            a[1] = q;
          } else {
            const int r = e - nR;
            double2* a = r < nC ? T + r + lt * i : Q + (r - nC) + lq * i;
            const long long ld = r < nC ? lt : lq;
            double2 p = a[0], q = a[ld];
            rot_col(p, q, g.c, g.sr, g.si);
            a[0] = p;
            a[ld] = q;
          }
        }
      }
      __syncthreads();
    }
  }
  __syncthreads();
  for (long long e = tid; e < (long long)s * s; e += kSchurThreads) {
    const int r = (int)(e % s);
    const long long q = e / s;
    const double2 t = T[r + lt * q];
    Tg[e] = r > q ? make_double2(0.0, 0.0) : make_double2(scalbn(t.x, ex), scalbn(t.y, ex));
    if (qs_in) Qg[e] = Q[r + lq * q];
  }
}

}  // namespace

void schur_small(double2* T, double2* Q, int s, int count, int* err, cudaStream_t st) {
  // T and Q share the 227 KB up to s = 84, T alone fits up to s = 119; larger matrices stay in global memory
  constexpr size_t kMax = 226 * 1024;
  const size_t one = sizeof(double2) * (size_t)s * (s + 1);
  const int ts_in = one <= kMax, qs_in = 2 * one <= kMax;
  const size_t smem = one * (ts_in + qs_in);
  set_max_dynamic_smem((const void*)k_schur_small, (int)kMax);
  k_schur_small<<<count, kSchurThreads, smem, st>>>(T, Q, s, err, ts_in, qs_in);
  count_launch();
  TS_CUDA(cudaGetLastError());
}

}  // namespace ts
