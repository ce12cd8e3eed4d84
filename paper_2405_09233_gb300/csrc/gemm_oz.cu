// Emulated FP64 per-slice products on the tcgen05 tensor cores (Ozaki scheme):
//     Y_k = A_k X_k - X_k B_k      (Eq. (2) in the Fourier domain, Algorithm 1 step 2)
// from FP64 inputs, with a result at the accuracy level of an FP64 product, computed from BF16
// products that the tensor cores form and sum without rounding.  GB300 issues FP64 at ~1.26
// TFLOP/s but BF16 at ~2 PFLOP/s, so the ~21 digit-pair products cost far less than one DFMA GEMM.
//
// Method: Ozaki, Ogita, Oishi and Rump, "Error-free transformations of matrix multiplication by
// using fast routines of matrix multiplication and its applications", Numer. Algorithms 59 (2012),
// arranged for tensor memory:
//  * Every FP64 slice Z (A_k and B_k share one exponent E_op[k]; X_k has E_x[k], both with
//    max |Re|, |Im| < 2^(E-1)) is written as Z = 2^E sum_{t=1..S} d_t 256^-t + r, |r| <= 2^E 256^-S / 2,
//    with integer digits |d_t| <= 128: the balanced base-256 expansion of round(Z 2^(8S-E)), taken
//    with integer arithmetic from the FP64 bit pattern.  Such digits are exact in BF16.
//  * A digit product is an integer of magnitude <= 2^14.  One accumulator run adds at most 512 of them
//    into a TMEM FP32 accumulator (8 pairs over a k-block of 32, or 4 over 64, Re of Ar Xr and of -Ai Xi);
//    every partial sum is an integer of at most 2^23, so the tensor core sums them exactly.
//  * Digit pairs (u, v) with u + v = g share the scale 2^(E_op + E_x - 8g); the pairs with
//    g <= S + 1 are kept (the dropped ones are below the truncation error of the digits).  Each
//    accumulator run ("unit": every pair of one g over one k-block of 32) is read from TMEM, converted to
//    int32 and added into per-thread int64 accumulators at the common fixed point
//    2^(E_op + E_x - F), F = 63 - ceil(log2(2 (n + s))), which keeps every partial sum below 2^62.
//    Units with 8g > F are added with a rounded right shift.
//  * Y = double(acc) 2^(E_op + E_x - F): one rounding.
//
// What bounds the product and why it walks the digits this way.  A 128 x 128 x 16 MMA reads 8 KB of
// shared memory in 64 clocks, all the 128 bytes per clock an SM has, and every operand byte TMA writes
// competes with it.  Walking one digit pair over 8 k-blocks at a time (the first form) loaded 56 KB per 8
// MMAs, another 110 bytes per clock, and held the tensor pipe near a half.  Now a k-block's S digits of A and
// X are loaded once, stay in shared memory for all S (S + 1) / 2 pairs, and leave digit by digit (the
// pairs run from g = S + 1 down to 2; digit d is last used at g = d + 1), so operand traffic falls to 168 KB
// per 84 MMAs (S = 6).  The k-block is 32 deep so that 8 digit slots of 28 KB fit: six in use and the next
// k-block's first ones arriving.  Pairs of g = S + 1 start with the middle digits, the first to arrive.
// A real slice (k = 0 or p/2) multiplies the real planes of 128 columns instead of Re and Im of 64.
// Measured (6 digits): n = s = 1024, p = 16 2.80 -> 2.15 ms (1.26 PFLOP/s of digit products); n = 4096, s = 256,
// p = 8 3.46 -> 2.40 ms; n = 256, s = 128, p = 8 94 -> 74 us.  Left: MMAs and operand writes together ask for 160
// bytes of shared memory per clock (1.58 ms), and the drains are hidden only in part.
//
// One CTA computes a 128 x 64 (real slices: 128 x 128) output tile of one slice.  Warp roles (320 threads):
//   warps 0-7  epilogue: warp w reads TMEM lanes 32 (w mod 4) .. +31 (output rows) and columns
//              32 (w div 4) .. +31 of each half of the accumulator; holds 2 x 32 int64 per thread
//   warp 8     TMA producer
//   warp 9     TMEM allocator and MMA issuer (all lanes converged, one elected lane executes)
// Four TMEM accumulators (Re 64 + Im 64 columns each) alternate between units and are drained two at a time,
// so that the MMAs run on meanwhile.  Every wait is bounded.
#include <cuda_bf16.h>
#include <climits>
#include <cfloat>
#include <cstdlib>
#include <algorithm>
#include <vector>
#include "internal.cuh"
#include "apply.cuh"
#include "tcgen05.cuh"
#include "oz.cuh"

namespace ts {
namespace {
using namespace tcg;

constexpr int kOzM = 128;                               // tile rows (TMEM lanes)
constexpr int kOzN = 64;                                // tile columns (complex slices)
constexpr int kOzKB = 32;                               // k-block: BF16 elements per 64-byte row
constexpr int kOzSlots = 8;                             // digit slots (the most digits a value has)
constexpr int kOzTileA = kOzM * 2 * kOzKB;              // bytes of one A-operand plane tile
constexpr int kOzTileB = kOzN * 2 * kOzKB;              // bytes of one 64-row B-operand block
constexpr int kOzSlot = 2 * kOzTileA + 3 * kOzTileB;    // A Re, A Im; B blocks [P; Q; R]
constexpr int kOzSmem = kOzSlots * kOzSlot + 1024 + 256;
constexpr int kOzAccs = 4;                              // TMEM accumulators
constexpr int kOzTmemCols = kOzAccs * 2 * kOzN;
constexpr int kOzEpi = 8;                               // epilogue warps
constexpr int kOzCols = kOzN / (kOzEpi / 4);            // columns of each half per epilogue warp
constexpr int kOzThreads = 32 * (kOzEpi + 2);
static_assert(kOzTmemCols == 512 && kOzSmem <= 227 * 1024, "tensor and shared memory");

struct OzMaps {
  CUtensorMap a_re, a_im;     // A digits  [S*K][n][ldn]  row-major A_k         (A operand of A X)
  CUtensorMap xc_re, xc_im;   // X digits  [S*K][s][ldn]  column-major X_k      (B operand of A X)
  CUtensorMap xc_nim;         //   and the digits of -Im X_k
  CUtensorMap xr_re, xr_im;   // X digits  [S*K][n][lds]  row-major X_k         (A operand of X B)
  CUtensorMap b_re, b_im;     // B digits  [S*K][s][lds]  column-major B_k      (B operand of X B)
  CUtensorMap b_nre;          //   and the digits of -Re B_k
};

// The output and sizes of one product; mx_op, mx_x: per-slice maxima of (A_k, B_k) and of X_k.
struct OzOut {
  double2* Y;
  const unsigned long long* mx_op;
  const unsigned long long* mx_x;
  int n, s, K, nyq, S, F;
  int stall;   // test aid: load the first k-block only, so the MMA warp's next wait expires
};

// Exponent of a slice from its maximum: max < 2^(E-1): ilogb(max) + 2 (0 for an all-zero slice); false when
// not finite.
__device__ __forceinline__ bool oz_exponent(unsigned long long mx, int& E) {
  const double m = __longlong_as_double((long long)mx);
  E = m == 0.0 ? 0 : ilogb(m) + 2;
  if (m <= DBL_MAX) return true;
  E = 0;
  return false;
}

// The order of one k-block's units and pairs: g from S + 1 down to 2, and inside g = S + 1 the pairs from the
// middle digits outwards (the order in which the digits arrive: S first).
__device__ __forceinline__ constexpr int oz_pair_u(int S, int g, int t) {
  if (g <= S) return t + 1;
  const int m = (S + 1) / 2 - (S % 2 ? (t + 1) / 2 : t / 2);     // min(u, v) of the t-th pair
  const bool first = S % 2 ? (t % 2 == 0 ? false : true) : t % 2 == 0;
  return S % 2 && t == 0 ? m : (first ? m : g - m);
}

// Shared-memory matrix descriptor: K-major operand tile with 64-byte rows and the 64-byte swizzle TMA
// applied (8-row atoms of 512 bytes).
__device__ __forceinline__ uint64_t smem_desc_sw64(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFFu);   // start address
  d |= (uint64_t)1 << 16;                   // leading byte offset (unused with this swizzle)
  d |= (uint64_t)(512 >> 4) << 32;          // stride byte offset
  d |= (uint64_t)1 << 46;                   // descriptor version
  d |= (uint64_t)4 << 61;                   // 64-byte swizzle
  return d;
}

// 8 consecutive TMEM columns of this warp's 32 lanes (one value per column per thread).
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}

// 32-deep blocks per unit: with few digits two fit the slots, and a unit of few MMAs would leave the epilogue
// behind (4 pairs x 128 products of 2^14 stay below 2^24).
__host__ __device__ constexpr int oz_sub(int S) { return 2 * S <= kOzSlots ? 2 : 1; }

// Units are drained two at a time, g + 1 (values b) and g (values a), 256 apart in scale (an odd S leaves its
// top unit alone, as a b without a): t = a' ca + b' in 32 bits, then acc += t m in one 32 x 32 + 64
// multiply-add, so that the accumulators see half the updates.  a' is converted (2 clocks of the SM per
// warp, on a pipe of its own); b' is read off the bit pattern of b + M, M = 1.5 2^(23 + e), which is that of M
// plus round(b / 2^e) while |b| <= 2^(22 + e).  M's pattern goes into the accumulators with the value and
// comes out at the end (arithmetic modulo 2^64).  e = 0 needs at most 4 pairs (4 x 64 products of 2^14).  More occur
// at e = 0 where F leaves all of the lowest units' bits: with 5 digits or fewer, and for n + s <= 64 (oz_forms's
// conditions).  There b is converted like a (kOzConvert), and beyond a factor of 2^30 the sum is shifted instead of
// multiplied more than twice (kOzShift).
// |t| < 2^31: M's pattern, 1.26e9, plus 256 times 3 x 2^20 (e = 0) or 2^7 times 6 x 2^20 (e > 0), plus 2^23; without
// M, 256 times 7 x 2^20 plus 2^23.
// The epilogue sets the pace together with the MMAs, so it exists once per set of forms: with all of them in one,
// n = s = 1024, p = 16 and 6 digits took 2.72 to 2.82 ms, not 2.69.
// There, before the lowest bits were kept and now: 5 digits 2.40 / 2.43 ms, 4 digits 1.69 / 1.69, 3 digits 1.33 / 1.32.
constexpr uint32_t kOzMagic = 0x4B400000u;   // pattern of 1.5 2^23; 2^e times it: + e 2^23
enum { kOzPattern, kOzConvert, kOzShift };
// The last form that some unit of a product takes.
__device__ __forceinline__ int oz_forms(int F, int S) {
  return F < 8 * (S + 1) && F <= 55 ? kOzPattern : (F <= 54 ? kOzConvert : kOzShift);
}
struct OzScale {
  int mode;
  float M, fa;        // b' from b + M; a' = round(a fa)
  int ca, m, reps;    // acc += (a' ca + pattern) m, reps times
  int sh;             // kOzShift: acc += (a' ca + b') << sh
  long long offset;   // what M's pattern adds
};
template <int FORMS>
__device__ __forceinline__ OzScale oz_scale(int F, int S, int gb, bool lone) {
  const int sb = F - 8 * gb, sa = sb + 8;
  const uint32_t pat = kOzMagic + (sb < 0 ? (uint32_t)-sb << 23 : 0u);
  OzScale q;
  if (FORMS == kOzPattern) q.mode = kOzPattern;
  else if (FORMS == kOzShift && sb > 30) q.mode = kOzShift;
  else q.mode = sb >= 0 && (gb - 1) * oz_sub(S) > 4 ? kOzConvert : kOzPattern;
  q.M = __uint_as_float(pat);
  q.fa = sa < 0 ? __uint_as_float((uint32_t)(127 + sa) << 23) : 1.f;
  q.ca = FORMS == kOzPattern && lone ? 0 : (sb >= 0 ? 256 : (sa > 0 ? 1 << sa : 1));
  q.m = sb <= 0 ? 1 : 1 << (sb > 30 ? 30 : sb);
  q.reps = sb > 30 ? 1 << (sb - 30) : 1;
  q.sh = sb;
  q.offset = q.mode == kOzPattern ? (long long)pat * q.m * q.reps : 0ll;
  return q;
}
// Columns C0 .. C0 + 7 of the units at ta (a) and tb (b).
template <int MODE, int C0>
__device__ __forceinline__ void acc_add8(long long (&acc)[kOzCols], uint32_t ta, uint32_t tb, const OzScale& q) {
  uint32_t va[8], vb[8];
  tmem_ld8(ta + C0, va);
  tmem_ld8(tb + C0, vb);
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const float fb = __uint_as_float(vb[c]);
    const int b = MODE == kOzPattern ? __float_as_int(fb + q.M) : __float2int_rn(fb);
    const int t = __float2int_rn(__uint_as_float(va[c]) * q.fa) * q.ca + b;
    if (MODE == kOzShift) acc[C0 + c] += (long long)t << q.sh;
    else asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc[C0 + c]) : "r"(t), "r"(q.m));
  }
}
// The lone unit at tb.
template <int MODE, int C0>
__device__ __forceinline__ void acc_add8_lone(long long (&acc)[kOzCols], uint32_t tb, const OzScale& q) {
  uint32_t vb[8];
  tmem_ld8(tb + C0, vb);
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const float fb = __uint_as_float(vb[c]);
    const int t = MODE == kOzPattern ? __float_as_int(fb + q.M) : __float2int_rn(fb);
    if (MODE == kOzShift) acc[C0 + c] += (long long)t << q.sh;
    else asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc[C0 + c]) : "r"(t), "r"(q.m));
  }
}
template <int MODE, int C0 = 0>
__device__ __forceinline__ void acc_add(long long (&acc)[kOzCols], uint32_t ta, uint32_t tb, const OzScale& q) {
  acc_add8<MODE, C0>(acc, ta, tb, q);
  if constexpr (C0 + 8 < kOzCols) acc_add<MODE, C0 + 8>(acc, ta, tb, q);
}
template <int MODE, int C0 = 0>
__device__ __forceinline__ void acc_add_lone(long long (&acc)[kOzCols], uint32_t tb, const OzScale& q) {
  acc_add8_lone<MODE, C0>(acc, tb, q);
  if constexpr (C0 + 8 < kOzCols) acc_add_lone<MODE, C0 + 8>(acc, tb, q);
}
// Fixed point 2^(E_op + E_x - F): |partial sums| < 2 (n + s) 2^(E_op + E_x - 2) <= 2^(E_op + E_x + 62 - F).
int oz_fixed_point(int n, int s) {
  int lg = 0;
  while ((1ll << lg) < 2ll * ((long long)n + s)) ++lg;
  return 63 - lg;
}

// The MMA issuer's walk of a tile with S digits (one converged warp).  Everything but the slots is known at
// compile time and the operands are uniform, so that between two MMAs (64 clocks) it executes a handful of
// instructions: with the pairs and slots computed in a loop the issuing thread, not the tensor pipe, set the
// pace (206 clocks per MMA).
// KIND 0: complex slice, A X: D += Ar [Xr | Xi] + Ai [-Xi | Xr]   (B blocks [P; Q; R], Q-R then P-Q)
//      1: complex slice, X B: D += -Xr [Br | Bi] + Xi [Bi | -Br]  (P-Q then Q-R)
//      2, 3: real slice, A X and X B, 128 real columns: D += Ar [Xr], D += -Xr [Br]  (P-Q)
// Returns false when a wait expired; oz_mma_walk has then committed the MMAs it issued to the `done` barrier (a
// commit covers its own thread's MMAs only, and the elected lane is known here).
template <int S, int KIND>
__device__ __forceinline__ bool oz_mma_block(uint32_t one, uint32_t bar_full, uint32_t bar_empty, uint32_t bar_acc, uint32_t bar_free,
                                             uint64_t desc0, uint32_t tmem, int first, int& q, int* err) {
  constexpr uint32_t idp = make_idesc(1, kOzM, 2 * kOzN, false);
  constexpr uint32_t idn = make_idesc(1, kOzM, 2 * kOzN, true);
  constexpr uint32_t oAi = kOzTileA >> 4, oP = 2 * kOzTileA >> 4, oQ = oP + (kOzTileB >> 4);
  constexpr int U = oz_sub(S);
  uint64_t desc[S * U];   // digit d of sub-block b at (S - d) U + b
#pragma unroll
  for (int i = 0; i < S * U; ++i) desc[i] = desc0 + (uint32_t)((first + i) % kOzSlots) * (kOzSlot >> 4);
#pragma unroll
  for (int g = S + 1; g >= 2; --g, ++q) {
    const int b = q % kOzAccs;   // its accumulator has been drained
    if (q >= kOzAccs && !mbar_wait_warp(bar_free + 8 * b, (uint32_t)(q / kOzAccs - 1) & 1u, err, 12)) return false;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t d = tmem + (uint32_t)(b * 2 * kOzN);
#pragma unroll
    for (int tb = 0; tb < (g - 1) * U; ++tb) {
      const int t = tb / U, sub = tb % U;
      const int u = oz_pair_u(S, g, t), v = g - u, iu = (S - u) * U + sub, iv = (S - v) * U + sub;
      if (g == S + 1) {   // every digit is met once in this unit: the wait for its arrival
        if (!mbar_wait_warp(bar_full + 8 * ((first + iu) % kOzSlots), (uint32_t)((first + iu) / kOzSlots) & 1u, err, 13))
          return false;
        if (u != v &&
            !mbar_wait_warp(bar_full + 8 * ((first + iv) % kOzSlots), (uint32_t)((first + iv) / kOzSlots) & 1u, err, 13))
          return false;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      }
      const uint64_t dA = desc[iu], dB = desc[iv];
#pragma unroll
      for (int kk = 0; kk < 2; ++kk) {
        const uint64_t f = (uint64_t)(kk * 2);   // 32 bytes >> 4
        const uint32_t acc = tb == 0 && kk == 0 ? 0u : 1u;
        if (KIND >= 2) {
          mma_issue_one(one, d, dA + f, dB + oP + f, KIND == 2 ? idp : idn, acc, 0);
        } else if (KIND == 0) {
          mma_issue_one(one, d, dA + f, dB + oQ + f, idp, acc, 0);
          mma_issue_one(one, d, dA + oAi + f, dB + oP + f, idp, 1u, 0);
        } else {
          mma_issue_one(one, d, dA + f, dB + oP + f, idn, acc, 0);
          mma_issue_one(one, d, dA + oAi + f, dB + oQ + f, idp, 1u, 0);
        }
      }
    }
#pragma unroll
    for (int sub = 0; sub < U; ++sub)
      mma_commit_one(one, bar_empty + 8 * ((first + (S - (g - 1)) * U + sub) % kOzSlots));   // digit g - 1 is done with
    mma_commit_one(one, bar_acc + 8 * b);
  }
  return true;
}
template <int S>
__device__ __noinline__ bool oz_mma_walk(uint32_t bars, uint32_t base, uint32_t tmem_, int real_, int kbA_, int kbs_,
                                         int* err) {
  const uint32_t bar_full = warp_uniform(bars), bar_empty = bar_full + 8 * kOzSlots;
  const uint32_t bar_acc = bar_empty + 8 * kOzSlots, bar_free = bar_acc + 8 * kOzAccs;
  const uint64_t desc0 = smem_desc_sw64(warp_uniform(base));
  const uint32_t tmem = warp_uniform(tmem_), one = elect_one();
  const bool real = warp_uniform(real_) != 0;
  const int kbA = (int)warp_uniform(kbA_), kbs = (int)warp_uniform(kbs_);
  int q = 0;   // unit
  for (int kb = 0; kb < kbs; ++kb) {
    bool ok;
    if (real) {
      ok = kb < kbA ? oz_mma_block<S, 2>(one, bar_full, bar_empty, bar_acc, bar_free, desc0, tmem, kb * S * oz_sub(S), q, err)
                    : oz_mma_block<S, 3>(one, bar_full, bar_empty, bar_acc, bar_free, desc0, tmem, kb * S * oz_sub(S), q, err);
    } else {
      ok = kb < kbA ? oz_mma_block<S, 0>(one, bar_full, bar_empty, bar_acc, bar_free, desc0, tmem, kb * S * oz_sub(S), q, err)
                    : oz_mma_block<S, 1>(one, bar_full, bar_empty, bar_acc, bar_free, desc0, tmem, kb * S * oz_sub(S), q, err);
    }
    if (!ok) {
      mma_commit_one(one, bar_free + 8 * kOzAccs);
      return false;
    }
  }
  return true;
}

// The epilogue warps' part of a tile: every unit into the accumulators, then Y.  Out of line (as the issue
// walks are), so that its registers are allocated for it alone.
template <int FORMS>   // oz_forms(F, S)
__device__ __noinline__ void oz_drain(const OzOut& o, uint32_t tmem, uint32_t bar_acc, uint32_t bar_free, int k, int i0,
                                      int j0, int* err) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n = o.n, s = o.s, S = o.S, F = o.F;
  const bool real = (k == 0) || (k == o.nyq);
  const int depth = kOzKB * oz_sub(S), kbs = (n + depth - 1) / depth + (s + depth - 1) / depth;
  // Rows i0 + 32 (warp mod 4) + lane; columns kOzCols (warp div 4) + c of both halves.
  const int quad = warp & 3, part = warp >> 2;
  const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(part * kOzCols);
  long long ar[kOzCols], ai[kOzCols];
#pragma unroll
  for (int c = 0; c < kOzCols; ++c) ar[c] = ai[c] = 0;
  long long magic = 0;
  bool ok = true;
  int q = 0;   // units drained
  for (int kb = 0; kb < kbs && ok; ++kb) {
    for (int g = S + 1; g >= 2;) {   // units g (b) and g - 1 (a)
      const bool lone = g == S + 1 && S % 2 != 0;
      const OzScale sc = oz_scale<FORMS>(F, S, g, lone);
      const int qa = lone ? q : q + 1, bb = q % kOzAccs, ba = qa % kOzAccs;
      if (!mbar_wait(bar_acc + 8 * ba, (uint32_t)(qa / kOzAccs) & 1u, err, 14)) {   // then b is complete too
        ok = false;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t tb = lane_base + (uint32_t)(bb * 2 * kOzN), ta = lane_base + (uint32_t)(ba * 2 * kOzN);
      // 8 columns at a time: little room beside the accumulators
      if (FORMS != kOzPattern && lone) {
        if (sc.mode == kOzPattern) {
          acc_add_lone<kOzPattern>(ar, tb, sc);
          acc_add_lone<kOzPattern>(ai, tb + kOzN, sc);
        } else if (FORMS == kOzConvert || sc.mode == kOzConvert) {
          acc_add_lone<kOzConvert>(ar, tb, sc);
          acc_add_lone<kOzConvert>(ai, tb + kOzN, sc);
        } else {
          acc_add_lone<kOzShift>(ar, tb, sc);
          acc_add_lone<kOzShift>(ai, tb + kOzN, sc);
        }
      } else if (FORMS == kOzPattern || sc.mode == kOzPattern) {
        for (int r = 0; r < sc.reps; ++r) {
          acc_add<kOzPattern>(ar, ta, tb, sc);
          acc_add<kOzPattern>(ai, ta + kOzN, tb + kOzN, sc);
        }
      } else if (FORMS == kOzConvert || sc.mode == kOzConvert) {
        acc_add<kOzConvert>(ar, ta, tb, sc);
        acc_add<kOzConvert>(ai, ta + kOzN, tb + kOzN, sc);
      } else {
        acc_add<kOzShift>(ar, ta, tb, sc);
        acc_add<kOzShift>(ai, ta + kOzN, tb + kOzN, sc);
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(bar_free + 8 * bb);
        if (!lone) mbar_arrive(bar_free + 8 * ba);
      }
      magic += sc.offset;
      g -= lone ? 1 : 2;
      q = qa + 1;
    }
  }
  const int row = i0 + quad * 32 + lane;
  if (ok && row < n) {
    int ea, ex;
    const bool fa = oz_exponent(o.mx_op[k], ea), fx = oz_exponent(o.mx_x[k], ex);
    const bool bad = !fa || !fx;
    const double scale = bad ? __longlong_as_double(0x7ff8000000000000ll) : ldexp(1.0, ea + ex - F);
    double2* Yk = o.Y + (long long)k * n * s + row;
#pragma unroll
    for (int c = 0; c < kOzCols; ++c) {
      const int j = j0 + part * kOzCols + c;
      const double re = (double)(ar[c] - magic) * scale, im = (double)(ai[c] - magic) * scale;
      if (!real) {
        if (j < s) Yk[(long long)j * n] = make_double2(re, im);
      } else {
        if (j < s) Yk[(long long)j * n] = make_double2(re, bad ? scale : 0.0);
        if (j + kOzN < s) Yk[(long long)(j + kOzN) * n] = make_double2(im, bad ? scale : 0.0);
      }
    }
  }
}

// One output tile (rows i0.., columns j0..) of slice k; blockDim.x == kOzThreads.
__device__ __noinline__ void oz_tile(const OzMaps* maps, const OzOut& o, int k, int i0, int j0, int* err) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base - raw);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kOzSlots * kOzSlot);
  // bars: full[kOzSlots], empty[kOzSlots], acc[kOzAccs], free[kOzAccs], done; then the TMEM address slot
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kOzSlots + 2 * kOzAccs + 1);
  const uint32_t bar_full = smem_u32(bars), bar_empty = smem_u32(bars + kOzSlots);
  const uint32_t bar_acc = smem_u32(bars + 2 * kOzSlots), bar_free = smem_u32(bars + 2 * kOzSlots + kOzAccs);
  const uint32_t bar_done = smem_u32(bars + 2 * kOzSlots + 2 * kOzAccs);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n = o.n, s = o.s, K = o.K, S = o.S;
  const bool real = (k == 0) || (k == o.nyq);
  const int sub = oz_sub(S), depth = kOzKB * sub;
  const int kbA = (n + depth - 1) / depth, kbs = kbA + (s + depth - 1) / depth;   // k-blocks of A X, of both

  if (threadIdx.x == 0) {
    for (int q = 0; q < kOzSlots; ++q) {
      mbar_init(bar_full + 8 * q, 1);
      mbar_init(bar_empty + 8 * q, 1);
    }
    for (int b = 0; b < kOzAccs; ++b) {
      mbar_init(bar_acc + 8 * b, 1);
      mbar_init(bar_free + 8 * b, kOzEpi);   // one arrival per epilogue warp
    }
    mbar_init(bar_done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kOzEpi + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(kOzTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  if (warp == kOzEpi) {
    if (lane == 0) {
      int it = 0, issued = 0;   // slots visited / slots whose loads were issued
      bool ok = true;
      for (int kb = 0; kb < (o.stall ? 1 : kbs) && ok; ++kb) {
        const bool ax = kb < kbA;
        for (int i = 0; i < S * sub; ++i, ++it) {
          const int d = S - i / sub, l0 = (ax ? kb : kb - kbA) * depth + i % sub * kOzKB;
          const int slot = it % kOzSlots;
          const uint32_t phase = (uint32_t)(it / kOzSlots) & 1u;
          if (!mbar_wait(bar_empty + 8 * slot, phase ^ 1u, err, 11)) {
            ok = false;
            break;
          }
          const uint32_t full = bar_full + 8 * slot;
          // a real slice uses the real A tile and two B blocks (columns j0.. and j0 + 64..)
          mbar_expect_tx(full, real ? kOzTileA + 2 * kOzTileB : kOzSlot);
          const uint32_t sA = base + slot * kOzSlot;
          const uint32_t sAi = sA + kOzTileA, sP = sA + 2 * kOzTileA, sQ = sP + kOzTileB, sR = sQ + kOzTileB;
          const int pl = (d - 1) * K + k;
          if (real) {
            const CUtensorMap* mb = ax ? &maps->xc_re : &maps->b_re;
            tma_load_3d(sA, ax ? &maps->a_re : &maps->xr_re, l0, i0, pl, full);
            tma_load_3d(sP, mb, l0, j0, pl, full);
            tma_load_3d(sQ, mb, l0, j0 + kOzN, pl, full);
          } else if (ax) {   // [P; Q; R] = [-Xi; Xr; Xi]
            tma_load_3d(sA, &maps->a_re, l0, i0, pl, full);
            tma_load_3d(sAi, &maps->a_im, l0, i0, pl, full);
            tma_load_3d(sP, &maps->xc_nim, l0, j0, pl, full);
            tma_load_3d(sQ, &maps->xc_re, l0, j0, pl, full);
            tma_load_3d(sR, &maps->xc_im, l0, j0, pl, full);
          } else {           // [P; Q; R] = [Br; Bi; -Br]
            tma_load_3d(sA, &maps->xr_re, l0, i0, pl, full);
            tma_load_3d(sAi, &maps->xr_im, l0, i0, pl, full);
            tma_load_3d(sP, &maps->b_re, l0, j0, pl, full);
            tma_load_3d(sQ, &maps->b_im, l0, j0, pl, full);
            tma_load_3d(sR, &maps->b_nre, l0, j0, pl, full);
          }
          issued = it + 1;
        }
      }
      // Every slot this warp loaded lands before the CTA exits, also when an error stopped the MMA
      // warp from consuming it: bounded waits on the last kOzSlots loads (immediate when all were used).
      for (int i = issued > kOzSlots ? issued - kOzSlots : 0; i < issued; ++i)
        mbar_wait(bar_full + 8 * (i % kOzSlots), (uint32_t)(i / kOzSlots) & 1u, err, 15);
      // ... and so do the commits that free the last slots (nobody else waits for them).
      for (int i = issued > kOzSlots ? issued - kOzSlots : 0; ok && i < issued; ++i)
        ok = mbar_wait(bar_empty + 8 * (i % kOzSlots), (uint32_t)(i / kOzSlots) & 1u, err, 17);
    }
  } else if (warp == kOzEpi + 1) {
    bool ok = true;
    switch (S) {
#define TS_OZ_WALK(D) \
  case D: ok = oz_mma_walk<D>(bar_full, base, tmem, real, kbA, kbs, err); break;
      TS_OZ_WALK(3) TS_OZ_WALK(4) TS_OZ_WALK(5) TS_OZ_WALK(6) TS_OZ_WALK(7) TS_OZ_WALK(8)
#undef TS_OZ_WALK
    }
    // after an error the MMAs already issued still complete before TMEM is freed
    if (!ok) mbar_wait(bar_done, 0u, err, 16);
    __syncwarp();
  } else {
    const int forms = oz_forms(o.F, S);
    if (forms == kOzPattern) oz_drain<kOzPattern>(o, tmem, bar_acc, bar_free, k, i0, j0, err);
    else if (forms == kOzConvert) oz_drain<kOzConvert>(o, tmem, bar_acc, bar_free, k, i0, j0, err);
    else oz_drain<kOzShift>(o, tmem, bar_acc, bar_free, k, i0, j0, err);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == kOzEpi + 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kOzTmemCols));
  }
}

// Columns of an output tile of slice k.
__host__ __device__ __forceinline__ int oz_tile_cols(int k, int nyq) { return k == 0 || k == nyq ? 2 * kOzN : kOzN; }

// Batched form: one CTA per (instance, slice, tile) work item; gate holds a flag per instance.
struct OzInstance {
  OzMaps maps;
  OzOut out;
  // the digit planes of X_k (see oz_split) and the spectrum they come from
  const double2* Xh;
  __nv_bfloat16 *xc_re, *xc_im, *xc_nim, *xr_re, *xr_im;
  unsigned long long* mx_x;
  int ldn, lds;
};
// The product kernel.  One instance (items null): blocks run over the complex slices' tiles, then the real
// ones' (half the work each, they fill the end of the launch); inside a slice, rows first.  A batch: one
// block per work item.
__global__ void __launch_bounds__(kOzThreads, 1)
    k_oz_sylv(const __grid_constant__ OzMaps maps, const __grid_constant__ OzOut out, const OzInstance* __restrict__ inst,
              const int4* __restrict__ items, const int* __restrict__ gate, int* err) {
  if (items) {
    const int4 it = items[blockIdx.x];
    if (gate[it.x] == 0) return;   // instance that has left the current cycle
    oz_tile(&inst[it.x].maps, inst[it.x].out, it.y, it.z, it.w, err);
    return;
  }
  const int mt = (out.n + kOzM - 1) / kOzM, ntc = (out.s + kOzN - 1) / kOzN;
  const int ntr = (out.s + 2 * kOzN - 1) / (2 * kOzN), kc = out.K - 1 - (out.nyq >= 0 ? 1 : 0);
  int b = blockIdx.x, k;
  if (b < kc * mt * ntc) {
    k = 1 + b / (mt * ntc);
    b %= mt * ntc;
  } else {
    b -= kc * mt * ntc;
    k = b / (mt * ntr) == 0 ? 0 : out.nyq;
    b %= mt * ntr;
  }
  oz_tile(&maps, out, k, b % mt * kOzM, b / mt * oz_tile_cols(k, out.nyq), err);
}

// ------------------------------------------------------------------------------------------------
// Exponents and digits
// ------------------------------------------------------------------------------------------------
// Per-slice max(|Re|, |Im|) of complex slices of T entries, as FP64 bit patterns (monotone for
// non-negative values) combined with atomicMax; a non-finite entry makes the slice's value +inf.
__device__ __forceinline__ void oz_maxabs(const double2* __restrict__ Zk, long long e0, long long e1, long long step,
                                          unsigned long long* __restrict__ out) {
  // Non-negative doubles order like their bit patterns read as unsigned integers (and every
  // non-finite pattern lies above that of +Inf), so the maximum is taken on integer ALUs: FP64
  // compares would make this pass FP64-pipe bound on GB300.
  constexpr unsigned long long kAbs = 0x7FFFFFFFFFFFFFFFull, kInf = 0x7FF0000000000000ull;
  unsigned long long m = 0;
#pragma unroll 4
  for (long long e = e0; e < e1; e += step) {
    const double2 v = Zk[e];
    const unsigned long long a = (unsigned long long)__double_as_longlong(v.x) & kAbs;
    const unsigned long long b = (unsigned long long)__double_as_longlong(v.y) & kAbs;
    m = max(m, max(a, b));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  __shared__ unsigned long long wm[32];
  if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long t = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t = max(t, wm[w]);
    atomicMax(out, t >= kInf ? kInf : t);   // any non-finite entry reads as +Inf
  }
}
__global__ void k_oz_maxabs(const double2* __restrict__ Z, long long T, unsigned long long* __restrict__ out) {
  oz_maxabs(Z + blockIdx.y * T, (long long)blockIdx.x * blockDim.x + threadIdx.x, T, (long long)gridDim.x * blockDim.x,
            out + blockIdx.y);
}
// Batched form: items (instance, slice, first column, end column).
__global__ void k_b_oz_maxabs(const OzInstance* __restrict__ inst, const int4* __restrict__ items,
                              const int* __restrict__ gate) {
  const int4 it = items[blockIdx.x];
  if (gate[it.x] == 0) return;
  const OzInstance& q = inst[it.x];
  const long long n = q.out.n;
  oz_maxabs(q.Xh + it.y * n * q.out.s, it.z * n + threadIdx.x, it.w * n, blockDim.x, q.mx_x + it.y);
}

// round(v 2^(8S - E)) as an integer from the FP64 bit pattern (|v| < 2^(E-1), so |q| <= 2^(8S-1)).
__device__ __forceinline__ long long oz_fixed(double v, int E, int S) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
  const int ex = (int)((bits >> 52) & 0x7FF);
  long long m = (long long)(bits & 0xFFFFFFFFFFFFFull);
  int e2;
  if (ex == 0) {
    e2 = 1 - 1075;            // subnormal: no implicit bit
  } else {
    m |= 1ll << 52;
    e2 = ex - 1075;
  }
  const int sh = e2 + 8 * S - E;
  long long q;
  if (m == 0 || sh <= -54) q = 0;
  else if (sh >= 0) q = m << sh;
  else q = (m + (1ll << (-sh - 1))) >> (-sh);
  return (bits >> 63) ? -q : q;
}

// Digit planes of one 64 x 32 tile of a complex slice: Sk is a column-major R x C matrix (entry (r, c) at
// Sk[c*R + r]).  COLS: planes with contiguous index r (rows c, pitch ldc), with the digits of -Re (NEG 1) or
// -Im (NEG 2) in cn; ROWS: planes with contiguous index c (rows r, pitch ldr).  Digit t (0 = most
// significant) of slice k lands in plane t*K + k.  Entries beyond R or C are not written, except one zero
// beside an odd edge (the tensor maps read them as zero); real slices have no Im planes.
//
// What bounds it: HBM (16 bytes read, 2 S bytes written per plane and entry).  Both layouts come from one read
// (a pass per layout read the spectrum twice), in runs of 128
// (COLS) and 64 (ROWS) bytes, two digits per lane.  The balanced digits are
// the bytes of q + 128 (1 + 256 + ..): one 64-bit addition, then a byte permute and an addition per digit
// make the exact FP32 value whose upper half is the BF16 digit.
// Measured, both layouts and 6 digits of n = s = 1024, p = 16: 222 -> 128 us.
struct OzPlanes {
  __nv_bfloat16 *c_re, *c_im, *c_neg, *r_re, *r_im;
  int ldc, ldr;
  long long plane_c, plane_r;   // entries of a plane
};
constexpr int kOzSplitR = 64, kOzSplitC = 32, kOzSplitPitch = kOzSplitC + 2, kOzSplitThreads = 256;
constexpr int oz_split_smem(int S) { return S * 2 * kOzSplitR * kOzSplitPitch * 2; }

template <bool COLS, bool ROWS, int NEG>
__device__ __forceinline__ void oz_split_tile(const double2* __restrict__ Sk, int R, int C, int K, int k, bool real,
                                              int r0, int c0, int E, int S, const OzPlanes& P) {
  extern __shared__ uint16_t split_smem[];   // ROWS: [S][2][64 r][34 c] digits
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int r = r0 + 2 * tx;
  const int parts = real ? 1 : 2;
  // q = top 256^(S-1) + low: the bytes of low + bias are the balanced digits + 128, its carry goes to the top
  const int top = 8 * (S - 1);
  const unsigned long long mask = (1ull << top) - 1, bias = 0x0080808080808080ull & mask;
  #pragma unroll 2
  for (int cc = ty; cc < kOzSplitC; cc += kOzSplitThreads / 32) {
    const int c = c0 + cc;
    double2 z0 = make_double2(0.0, 0.0), z1 = z0;
    if (c < C) {
      if (r < R) z0 = Sk[(long long)c * R + r];
      if (r + 1 < R) z1 = Sk[(long long)c * R + r + 1];
    }
#pragma unroll
    for (int part = 0; part < 2; ++part) {
      if (part >= parts) break;
      const long long q0 = oz_fixed(part ? z0.y : z0.x, E, S), q1 = oz_fixed(part ? z1.y : z1.x, E, S);
      const unsigned long long l0 = ((unsigned long long)q0 & mask) + bias, l1 = ((unsigned long long)q1 & mask) + bias;
      __nv_bfloat16* dst = part ? P.c_im : P.c_re;
      for (int t = 0; t < S; ++t) {
        const int sh = top - 8 * t;
        float f0, f1;
        if (t == 0) {   // signed, |d| <= 128
          f0 = (float)((int)(q0 >> top) + (int)(l0 >> top));
          f1 = (float)((int)(q1 >> top) + (int)(l1 >> top));
        } else {        // 8388608 + byte, exactly, minus 8388608 + 128
          f0 = __uint_as_float(0x4B000000u | ((uint32_t)(l0 >> sh) & 255u)) - 8388736.f;
          f1 = __uint_as_float(0x4B000000u | ((uint32_t)(l1 >> sh) & 255u)) - 8388736.f;
        }
        const uint32_t both = __byte_perm(__float_as_uint(f0), __float_as_uint(f1), 0x7632);
        if (COLS && c < C && r < R) {
          const long long o = ((long long)t * K + k) * P.plane_c + (long long)c * P.ldc + r;
          *reinterpret_cast<uint32_t*>(dst + o) = both;
          if (NEG == part + 1) *reinterpret_cast<uint32_t*>(P.c_neg + o) = both ^ 0x80008000u;
        }
        if (ROWS) {
          uint16_t* d = split_smem + ((t * 2 + part) * kOzSplitR + 2 * tx) * kOzSplitPitch + cc;
          d[0] = (uint16_t)both;
          d[kOzSplitPitch] = (uint16_t)(both >> 16);
        }
      }
    }
  }
  if (!ROWS) return;
  __syncthreads();
  const int c = c0 + 2 * (tx % 16), rl = 2 * ty + tx / 16;   // a half warp per row
  for (int t = 0; t < S; ++t)
    for (int part = 0; part < parts; ++part)
#pragma unroll
      for (int rr = rl; rr < kOzSplitR; rr += kOzSplitThreads / 16) {
        const int row = r0 + rr;
        if (row < R && c < C) {
          const uint32_t both = *reinterpret_cast<const uint32_t*>(
              split_smem + ((t * 2 + part) * kOzSplitR + rr) * kOzSplitPitch + 2 * (tx % 16));
          const long long o = ((long long)t * K + k) * P.plane_r + (long long)row * P.ldr + c;
          *reinterpret_cast<uint32_t*>((part ? P.r_im : P.r_re) + o) = both;
        }
      }
}

template <bool COLS, bool ROWS, int NEG>
__global__ void __launch_bounds__(kOzSplitThreads)
    k_oz_split(const double2* __restrict__ src, int R, int C, int K, int nyq, const unsigned long long* __restrict__ mx,
               int S, OzPlanes P) {
  const int k = blockIdx.z;
  int E;
  oz_exponent(mx[k], E);
  oz_split_tile<COLS, ROWS, NEG>(src + (long long)k * R * C, R, C, K, k, k == 0 || k == nyq, blockIdx.x * kOzSplitR,
                                 blockIdx.y * kOzSplitC, E, S, P);
}
// Batched form: items (instance, slice, first row, first column).
__global__ void __launch_bounds__(kOzSplitThreads)
    k_b_oz_split(const OzInstance* __restrict__ inst, const int4* __restrict__ items, const int* __restrict__ gate) {
  const int4 it = items[blockIdx.x];
  if (gate[it.x] == 0) return;
  const OzInstance& q = inst[it.x];
  const int n = q.out.n, s = q.out.s, K = q.out.K, k = it.y;
  int E;
  oz_exponent(q.mx_x[k], E);
  const OzPlanes P{q.xc_re, q.xc_im, q.xc_nim, q.xr_re, q.xr_im, q.ldn, q.lds, (long long)s * q.ldn, (long long)n * q.lds};
  oz_split_tile<true, true, 2>(q.Xh + (long long)k * n * s, n, s, K, k, k == 0 || k == q.out.nyq, it.z, it.w, E, q.out.S,
                               P);
}

inline int round_up(int v, int m) { return (v + m - 1) / m * m; }

void slice_maxabs(const double2* Z, long long T, int K, unsigned long long* out, cudaStream_t st) {
  long long b = (T + 1023) / 1024;
  if (b > 128) b = 128;
  k_oz_maxabs<<<dim3((unsigned)b, K), 256, 0, st>>>(Z, T, out);
  count_launch();
  TS_CUDA(cudaGetLastError());
}

template <bool COLS, bool ROWS, int NEG>
void split(const double2* src, int R, int C, int K, int nyq, const unsigned long long* mx, int S, const OzPlanes& P,
           cudaStream_t st) {
  const int smem = ROWS ? oz_split_smem(S) : 0;
  set_max_dynamic_smem((const void*)k_oz_split<COLS, ROWS, NEG>, oz_split_smem(8));
  k_oz_split<COLS, ROWS, NEG>
      <<<dim3((R + kOzSplitR - 1) / kOzSplitR, (C + kOzSplitC - 1) / kOzSplitC, K), kOzSplitThreads, smem,
         st>>>(src, R, C, K, nyq, mx, S, P);
  count_launch();
  TS_CUDA(cudaGetLastError());
}

// Tensor maps of one product: the operator's planes (all t.S digits exist; digit u of slice k is plane
// u K + k, the kernel reads u < S) and the S digits of X.
void oz_maps(OzMaps* m, const ts_op* op, int S, const OzBuffers& b) {
  const OzOperands& t = *op->oz;
  const int n = op->n, s = op->s, K = op->K;
  auto map = [](CUtensorMap* q, const void* base, int ld, int cols, int rows, int planes, int box_rows) {
    make_map(q, base, 2, ld, cols, rows, planes, box_rows, 64);
  };
  map(&m->a_re, t.a_re, t.ldn, n, n, t.S * K, kOzM);
  map(&m->a_im, t.a_im, t.ldn, n, n, t.S * K, kOzM);
  map(&m->xc_nim, b.xc_nim, t.ldn, n, s, S * K, kOzN);
  map(&m->xc_re, b.xc_re, t.ldn, n, s, S * K, kOzN);
  map(&m->xc_im, b.xc_im, t.ldn, n, s, S * K, kOzN);
  map(&m->xr_re, b.xr_re, t.lds, s, n, S * K, kOzM);
  map(&m->xr_im, b.xr_im, t.lds, s, n, S * K, kOzM);
  map(&m->b_re, t.b_re, t.lds, s, s, t.S * K, kOzN);
  map(&m->b_im, t.b_im, t.lds, s, s, t.S * K, kOzN);
  map(&m->b_nre, t.b_nre, t.lds, s, s, t.S * K, kOzN);
}

OzOut oz_out(const ts_op* op, double2* Yh, int S, const OzBuffers& b) {
  return OzOut{Yh, op->oz->mx, b.mx, op->n, op->s, op->K, nyquist_index(op->p), S,
               oz_fixed_point(op->n, op->s), 0};
}

}  // namespace

void OzOperands::release() {
  op_free(a_re);
  op_free(a_im);
  op_free(b_re);
  op_free(b_im);
  op_free(b_nre);
  op_free(mx);
  a_re = a_im = b_re = b_im = b_nre = nullptr;
  mx = nullptr;
  S = 0;
}

void oz_prepare(ts_op* op, int S, cudaStream_t st) {
  if (op->oz && op->oz->S == S) return;
  OzOperands* t = op->oz ? op->oz : new OzOperands();
  op->oz = t;
  t->release();
  const int n = op->n, s = op->s, K = op->K;
  t->ldn = round_up(n, 64);
  t->lds = round_up(s, 64);
  const size_t na = (size_t)S * K * n * t->ldn * 2, nb = (size_t)S * K * s * t->lds * 2;
  op_alloc_on(t->a_re, na, st);
  op_alloc_on(t->a_im, na, st);
  op_alloc_on(t->b_re, nb, st);
  op_alloc_on(t->b_im, nb, st);
  op_alloc_on(t->b_nre, nb, st);
  op_alloc_on(t->mx, sizeof(unsigned long long) * K, st);
  // A_k and B_k share one exponent per slice, so both products of Eq. (2) land on one fixed point.
  unsigned long long* mxb = t->mx;
  TS_CUDA(cudaMemsetAsync(mxb, 0, sizeof(unsigned long long) * K, st));
  slice_maxabs(op->Ah, (long long)n * n, K, mxb, st);
  slice_maxabs(op->Bh, (long long)s * s, K, mxb, st);
  const int nyq = nyquist_index(op->p);
  OzPlanes pa{};
  pa.r_re = static_cast<__nv_bfloat16*>(t->a_re);
  pa.r_im = static_cast<__nv_bfloat16*>(t->a_im);
  pa.ldr = t->ldn;
  pa.plane_r = (long long)n * t->ldn;
  split<false, true, 0>(op->Ah, n, n, K, nyq, mxb, S, pa, st);
  OzPlanes pb{};
  pb.c_re = static_cast<__nv_bfloat16*>(t->b_re);
  pb.c_im = static_cast<__nv_bfloat16*>(t->b_im);
  pb.c_neg = static_cast<__nv_bfloat16*>(t->b_nre);
  pb.ldc = t->lds;
  pb.plane_c = (long long)s * t->lds;
  split<true, false, 1>(op->Bh, s, s, K, nyq, mxb, S, pb, st);
  t->S = S;
}

double oz_bf16_flops(int n, int s, int K, int nyq, int S) {
  const int nreal = 1 + (nyq >= 0 ? 1 : 0);
  const double pairs = 0.5 * S * (S + 1);
  const double per = (double)n * s * ((double)n + s);
  return pairs * per * (8.0 * (K - nreal) + 2.0 * nreal);
}

void oz_preload() {
  const void* fns[] = {(const void*)k_oz_maxabs, (const void*)k_oz_split<true, true, 2>, (const void*)k_oz_sylv,
                       (const void*)k_b_oz_maxabs, (const void*)k_b_oz_split};
  for (const void* f : fns) {
    cudaFuncAttributes fa;
    TS_CUDA(cudaFuncGetAttributes(&fa, f));
  }
  set_max_dynamic_smem((const void*)k_oz_sylv, kOzSmem);
  set_max_dynamic_smem((const void*)k_oz_split<true, true, 2>, oz_split_smem(8));
  set_max_dynamic_smem((const void*)k_b_oz_split, oz_split_smem(8));
}

OzBufferSizes oz_buffer_sizes(int n, int s, int K, int S) {
  OzBufferSizes z;
  z.xc = (size_t)S * K * s * round_up(n, 64) * 2;
  z.xr = (size_t)S * K * n * round_up(s, 64) * 2;
  z.K = K;
  return z;
}

void oz_products(const ts_op* op, const double2* Xh, double2* Yh, int S, const OzBuffers& b, int* err,
                 cudaStream_t st) {
  const OzOperands& t = *op->oz;
  TS_REQUIRE(S >= 3 && S <= kOzSlots && t.S >= S, "oz_products: operator digits not prepared");
  const int n = op->n, s = op->s, K = op->K, nyq = nyquist_index(op->p);
  TS_CUDA(cudaMemsetAsync(b.mx, 0, sizeof(unsigned long long) * K, st));
  slice_maxabs(Xh, (long long)n * s, K, b.mx, st);
  const OzPlanes P{static_cast<__nv_bfloat16*>(b.xc_re),  static_cast<__nv_bfloat16*>(b.xc_im),
                   static_cast<__nv_bfloat16*>(b.xc_nim), static_cast<__nv_bfloat16*>(b.xr_re),
                   static_cast<__nv_bfloat16*>(b.xr_im),  t.ldn, t.lds, (long long)s * t.ldn, (long long)n * t.lds};
  split<true, true, 2>(Xh, n, s, K, nyq, b.mx, S, P, st);
  OzMaps maps;
  oz_maps(&maps, op, S, b);
  const long long mt = (n + kOzM - 1) / kOzM, kr = 1 + (nyq >= 0 ? 1 : 0);
  const long long blocks = mt * ((K - kr) * ((s + kOzN - 1) / kOzN) + kr * ((s + 2 * kOzN - 1) / (2 * kOzN)));
  TS_REQUIRE(blocks <= INT_MAX, "emulated product: grid too large");
  OzOut out = oz_out(op, Yh, S, b);
  // Test aid for the failure path (see tc_apply): with TSTAR_TEST_STALL_TMA=1 the producer stops after the first
  // k-block, with that block's MMAs issued.
  const char* stall_env = std::getenv("TSTAR_TEST_STALL_TMA");
  out.stall = stall_env && stall_env[0] == '1';
  k_oz_sylv<<<(unsigned)blocks, kOzThreads, kOzSmem, st>>>(maps, out, nullptr, nullptr, nullptr, err);
  count_launch();
  TS_CUDA(cudaGetLastError());
}

// --- batches ---
size_t oz_batch_instance_bytes() { return sizeof(OzInstance); }

size_t oz_batch_plane_bytes(const ts_op* op, int S) {
  const OzBufferSizes z = oz_buffer_sizes(op->n, op->s, op->K, S);
  auto up = [](size_t b) { return (b + 255) / 256 * 256; };
  return 3 * up(z.xc) + 2 * up(z.xr);
}

void oz_batch_instance(const ts_op* op, const double2* Xh, double2* Yh, int S, void* planes, unsigned long long* mx,
                       void* out) {
  const OzBufferSizes z = oz_buffer_sizes(op->n, op->s, op->K, S);
  auto up = [](size_t b) { return (b + 255) / 256 * 256; };
  char* q = static_cast<char*>(planes);
  OzBuffers b;
  b.xc_re = q; q += up(z.xc);
  b.xc_im = q; q += up(z.xc);
  b.xc_nim = q; q += up(z.xc);
  b.xr_re = q; q += up(z.xr);
  b.xr_im = q;
  b.mx = mx;
  OzInstance* o = static_cast<OzInstance*>(out);
  oz_maps(&o->maps, op, S, b);
  o->out = oz_out(op, Yh, S, b);
  o->Xh = Xh;
  o->xc_re = static_cast<__nv_bfloat16*>(b.xc_re);
  o->xc_im = static_cast<__nv_bfloat16*>(b.xc_im);
  o->xc_nim = static_cast<__nv_bfloat16*>(b.xc_nim);
  o->xr_re = static_cast<__nv_bfloat16*>(b.xr_re);
  o->xr_im = static_cast<__nv_bfloat16*>(b.xr_im);
  o->mx_x = mx;
  o->ldn = op->oz->ldn;
  o->lds = op->oz->lds;
}

void oz_batch_items(const std::vector<const ts_op*>& ops, int first, int end, std::vector<int4>* products,
                    std::vector<int4>* splits, std::vector<int4>* maxima) {
  const size_t sorted = products->size();
  for (int i = first; i < end; ++i) {
    const int n = ops[i]->n, s = ops[i]->s, K = ops[i]->K, nyq = nyquist_index(ops[i]->p);
    for (int k = 0; k < K; ++k) {
      const int tn = oz_tile_cols(k, nyq);
      for (int j0 = 0; j0 < s; j0 += tn)
        for (int i0 = 0; i0 < n; i0 += kOzM) products->push_back(make_int4(i, k, i0, j0));
      for (int c0 = 0; c0 < s; c0 += kOzSplitC)
        for (int r0 = 0; r0 < n; r0 += kOzSplitR) splits->push_back(make_int4(i, k, r0, c0));
      const int cols = std::max(1, 8192 / n);   // columns per block of the maxima
      for (int c0 = 0; c0 < s; c0 += cols) maxima->push_back(make_int4(i, k, c0, std::min(s, c0 + cols)));
    }
  }
  // largest first (a complex tile is twice a real one)
  std::stable_sort(products->begin() + sorted, products->end(), [&](const int4& a, const int4& b) {
    auto cost = [&](const int4& q) {
      const ts_op* op = ops[q.x];
      return (oz_tile_cols(q.y, nyquist_index(op->p)) == kOzN ? 2.0 : 1.0) * (op->n + op->s);
    };
    return cost(a) > cost(b);
  });
}

void oz_batch_products(const void* inst, const std::vector<OzBatchLists>& groups, unsigned long long* mx,
                       size_t mx_count, int S, const int* gate, int* err, cudaStream_t st) {
  const OzInstance* q = static_cast<const OzInstance*>(inst);
  TS_CUDA(cudaMemsetAsync(mx, 0, sizeof(unsigned long long) * mx_count, st));
  for (const OzBatchLists& l : groups) {
    k_b_oz_maxabs<<<l.n_maxima, 256, 0, st>>>(q, l.maxima, gate);
    k_b_oz_split<<<l.n_splits, kOzSplitThreads, oz_split_smem(S), st>>>(q, l.splits, gate);
    k_oz_sylv<<<l.n_products, kOzThreads, kOzSmem, st>>>(OzMaps{}, OzOut{}, q, l.products, gate, err);
    count_launch(3);
  }
  TS_CUDA(cudaGetLastError());
}

// The emulated products on spectral tensors: Yh = A_k Xh_k - Xh_k B_k (workspace digit planes of Xh).
void oz_apply_spectral(ts_ctx* ctx, const ts_op* cop, const double2* Xh, double2* Yh, int S, int S_op,
                       cudaStream_t st) {
  ts_op* op = const_cast<ts_op*>(cop);   // the digit planes are cached on first use
  oz_prepare(op, S_op, st);
  oz_preload();
  const int n = op->n, s = op->s, p = op->p, K = op->K;
  const OzBufferSizes z = oz_buffer_sizes(n, s, K, S);
  OzBuffers b;
  b.xc_re = ctx->ws.get("oz_xc_re", z.xc);
  b.xc_im = ctx->ws.get("oz_xc_im", z.xc);
  b.xc_nim = ctx->ws.get("oz_xc_nim", z.xc);
  b.xr_re = ctx->ws.get("oz_xr_re", z.xr);
  b.xr_im = ctx->ws.get("oz_xr_im", z.xr);
  b.mx = static_cast<unsigned long long*>(ctx->ws.get("oz_mx", sizeof(unsigned long long) * K));
  int* err = static_cast<int*>(ctx->ws.get("tc_err", sizeof(int) * 4));
  KernelTimer& tm = ctx->timer;
  tm.begin(st, 3, gemm_flops(n, s, n, s, K, nyquist_index(p)));
  if (tm.enabled) tm.oz_pair_flops += oz_bf16_flops(n, s, K, nyquist_index(p), S);
  oz_products(op, Xh, Yh, S, b, err, st);
  tm.end(st);
}

void apply_f64_oz(ts_ctx* ctx, const ts_op* cop, const double* X, double* Y, int mode, const double* C,
                  double* partials, int S, int S_op, cudaStream_t st) {
  ts_op* op = const_cast<ts_op*>(cop);   // the digit planes are cached on first use
  oz_prepare(op, S_op, st);
  oz_preload();
  const int n = op->n, s = op->s, p = op->p, K = op->K;
  const long long T = (long long)n * s;
  double2* Xh = static_cast<double2*>(ctx->ws.get("apply_Xh", sizeof(double2) * (size_t)K * T));
  double2* Yh = static_cast<double2*>(ctx->ws.get("apply_Yh", sizeof(double2) * (size_t)K * T));
  const OzBufferSizes z = oz_buffer_sizes(n, s, K, S);
  OzBuffers b;
  b.xc_re = ctx->ws.get("oz_xc_re", z.xc);
  b.xc_im = ctx->ws.get("oz_xc_im", z.xc);
  b.xc_nim = ctx->ws.get("oz_xc_nim", z.xc);
  b.xr_re = ctx->ws.get("oz_xr_re", z.xr);
  b.xr_im = ctx->ws.get("oz_xr_im", z.xr);
  b.mx = static_cast<unsigned long long*>(ctx->ws.get("oz_mx", sizeof(unsigned long long) * K));
  int* err = static_cast<int*>(ctx->ws.get("tc_err", sizeof(int) * 4));
  KernelTimer& tm = ctx->timer;
  tm.begin(st, 1, 8.0 * T * p + 16.0 * K * T);
  rfft_tube<double, double2>(X, Xh, T, p, st);
  tm.end(st);
  tm.begin(st, 3, gemm_flops(n, s, n, s, K, nyquist_index(p)));
  if (tm.enabled) tm.oz_pair_flops += oz_bf16_flops(n, s, K, nyquist_index(p), S);
  oz_products(op, Xh, Yh, S, b, err, st);
  tm.end(st);
  tm.begin(st, 1, 16.0 * K * T + 8.0 * T * p * (mode == IRFFT_RESIDUAL ? 2 : 1));
  irfft_tube<double, double2>(Yh, Y, T, p, mode, C, partials, st);
  tm.end(st);
}

}  // namespace ts
