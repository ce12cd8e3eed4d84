// Per-Fourier-slice complex products on CUDA cores, FP64 and FP32 (Algorithm 1 step 2; inside M
// it is the fused Y_k = A_k X_k - X_k B_k of Eq. (2) in the Fourier domain).
//
// GB300 runs FP64 at ~1 TFLOP/s on CUDA cores (DFMA and the m8n8k4 DMMA measure within 4% of
// each other), so the FP64 product is FP64-pipe bound by a wide margin and its tiles are free to
// follow the problem's shape (gemm_tile.cuh; launch_cheapest picks them).  What matters is the number of
// FP64 operations: the complex product uses three real products (Gauss):
//   T1 = sum ar*br, T2 = sum ai*bi, T3 = sum (ar+ai)(br+bi);  re = T1 - T2, im = T3 - T1 - T2,
// 3 DFMA per complex multiply-add instead of 4.  The sums ar+ai, br+bi are formed once per
// shared-memory tile element.  Slices k = 0 and k = p/2 are real (their imaginary parts are
// exactly zero) and take a single real product.
#include <type_traits>
#include "internal.cuh"
#include "gemm_tile.cuh"

namespace ts {
namespace {

// Slices in the order of their cost: the complex ones (k = 1 ..), then the real ones (k = 0, k = p/2).
__device__ __forceinline__ int slice_by_cost(int z, int K, int nyq) {
  const int kc = K - 1 - (nyq >= 0 ? 1 : 0);
  return z < kc ? z + 1 : (z == kc ? 0 : nyq);
}

template <int NT, int BN, int TM>
__global__ void __launch_bounds__(NT, (TM > 2 ? 3 : 4) * (256 / NT)) k_gemm_f64(ZGemmArgs a, int mt, int nt) {
  const int per = mt * nt, z = blockIdx.x / per, t = blockIdx.x % per;
  gemm_tile_f64<NT, BN, TM>(a, slice_by_cost(z, a.K, a.nyq), t % mt * F64Tile<NT, BN, TM>::BM, t / mt * BN);
}

template <int BM, int BN, int G>
__global__ void __launch_bounds__((F32Tile<BM, BN, G>::NT), G > 1 ? 3 : 2) k_gemm_f32(CGemmArgs a, int mt, int nt) {
  const int per = mt * nt, z = blockIdx.x / per, t = blockIdx.x % per;
  gemm_tile_f32<BM, BN, G>(a, slice_by_cost(z, a.K, a.nyq), t % mt * BM, t / mt * BN);
}

template <typename Real>
__global__ void __launch_bounds__(kTinyThreads) k_gemm_tiny(GemmArgs<typename CplxOf<Real>::T> a) {
  gemm_tiny_tile<Real>(a, blockIdx.z, blockIdx.x * kTinyBM, blockIdx.y * kTinyBN);
}

int sm_count() {
  static int cached[64] = {0};
  int dev = 0;
  TS_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return 152;
  if (!cached[dev]) TS_CUDA(cudaDeviceGetAttribute(&cached[dev], cudaDevAttrMultiProcessorCount, dev));
  return cached[dev];
}

// Estimated time of the product on bm x bn tiles, in output entries of a real slice per SM: the padded
// products (three real ones per complex entry) and `stage` extra operations per staged row or column,
// spread over the SMs, plus part of one tile for the uneven end of the launch.
double tile_cost(int M, int N, int K, int nyq, int bm, int bn, double stage, double tail) {
  const double kr = 1 + (nyq >= 0 ? 1 : 0), kc = K - kr;
  const double mt = (M + bm - 1) / bm, nt = (N + bn - 1) / bn, area = (double)bm * bn;
  const double one = 3.0 * area + stage * (bm + bn);   // a complex tile
  return mt * nt * (kc * one + kr * area) / sm_count() + tail * (kc > 0 ? one : area);
}

template <int NT, int BN, int TM>
void launch_f64(const ZGemmArgs& a, cudaStream_t st) {
  constexpr int BM = F64Tile<NT, BN, TM>::BM;
  const int mt = (a.M + BM - 1) / BM, nt = (a.N + BN - 1) / BN;
  const long long blocks = (long long)mt * nt * a.K;
  TS_REQUIRE((long long)mt * nt <= INT32_MAX && blocks <= INT32_MAX, "slice GEMM grid too large");
  k_gemm_f64<NT, BN, TM><<<(unsigned)blocks, NT, 0, st>>>(a, mt, nt);
}

template <int BM, int BN, int G>
void launch_f32(const CGemmArgs& a, cudaStream_t st) {
  using Cfg = F32Tile<BM, BN, G>;
  const int mt = (a.M + BM - 1) / BM, nt = (a.N + BN - 1) / BN;
  const long long blocks = (long long)mt * nt * a.K;
  TS_REQUIRE((long long)mt * nt <= INT32_MAX && blocks <= INT32_MAX, "slice GEMM grid too large");
  k_gemm_f32<BM, BN, G><<<(unsigned)blocks, Cfg::NT, Cfg::kSmem, st>>>(a, mt, nt);
}

// The cheapest tile by tile_cost.  `stage`, `tail` and `slow` were fitted to launches forced onto every shape:
//   FP64: at 1024 x 1024 x 16 (no padding, no uneven end) the shapes' rates follow the additions of their
//   factor sums, 0.96 of the pipe at 32 x 32 down to 0.87 at 32 x 4; the 64-thread 16 x 4 tile runs lower, 0.83.
//   FP32: 0.56, 0.47 and 0.39 of the FP32 rate for the three shapes at that size (fewer products per
//   barrier and per read); 512 x 128 x 16 takes 65, 72 and 74 us, 256 x 256 x 8 takes 52, 46 and 41 us.
template <typename Args>
struct TileShape {
  int bm, bn;
  double stage, tail, slow;
  void (*run)(const Args&, cudaStream_t);
};
template <typename Args, size_t N>
void launch_cheapest(const TileShape<Args> (&shapes)[N], const Args& a, cudaStream_t st) {
  const TileShape<Args>* best = nullptr;
  double cost = 0.0;
  for (const auto& s : shapes) {
    const double c = s.slow * tile_cost(a.M, a.N, a.K, a.nyq, s.bm, s.bn, s.stage, s.tail);
    if (!best || c < cost) {
      best = &s;
      cost = c;
    }
  }
  best->run(a, st);
}
void launch_tiles(const ZGemmArgs& a, cudaStream_t st) {
  static const TileShape<ZGemmArgs> shapes[] = {
      {64, 16, 1.3, 0.6, 1.0, launch_f64<256, 16, 4>}, {32, 32, 1.3, 0.6, 1.0, launch_f64<256, 32, 4>},
      {128, 8, 1.3, 0.6, 1.0, launch_f64<256, 8, 4>},  {32, 16, 1.3, 0.6, 1.0, launch_f64<256, 16, 2>},
      {64, 8, 1.3, 0.6, 1.0, launch_f64<256, 8, 2>},   {16, 16, 1.3, 0.6, 1.0, launch_f64<256, 16, 1>},
      {32, 8, 1.3, 0.6, 1.0, launch_f64<256, 8, 1>},   {64, 4, 1.3, 0.6, 1.0, launch_f64<256, 4, 1>},
      {16, 8, 1.3, 0.6, 1.0, launch_f64<128, 8, 1>},   {32, 4, 1.3, 0.6, 1.0, launch_f64<128, 4, 1>},
      {16, 4, 1.8, 0.6, 1.0, launch_f64<64, 4, 1>}};
  launch_cheapest(shapes, a, st);
}
void launch_tiles(const CGemmArgs& a, cudaStream_t st) {
  static const TileShape<CGemmArgs> shapes[] = {{64, 64, 0.0, 0.4, 1.0, launch_f32<64, 64, 1>},
                                                {64, 32, 0.0, 0.4, 1.2, launch_f32<64, 32, 2>},
                                                {32, 32, 0.0, 0.4, 1.4, launch_f32<32, 32, 4>}};
  launch_cheapest(shapes, a, st);
}

// Products whose reductions are at most kTinyL long run one 8 x 4 tile per CTA (see gemm_tiny_tile).
template <typename Real>
void launch_slices(const GemmArgs<typename CplxOf<Real>::T>& a, cudaStream_t st) {
  if (a.M <= 0 || a.N <= 0 || a.K <= 0) return;
  if (a.L1 <= kTinyL && a.L2 <= kTinyL) {
    dim3 grid((a.M + kTinyBM - 1) / kTinyBM, (a.N + kTinyBN - 1) / kTinyBN, a.K);
    TS_REQUIRE(grid.y <= 65535 && grid.z <= 65535, "slice GEMM grid too large");
    k_gemm_tiny<Real><<<grid, kTinyThreads, 0, st>>>(a);
  } else {
    launch_tiles(a, st);
  }
  count_launch();
  TS_CUDA(cudaGetLastError());
}

}  // namespace

void zgemm_slices_f64(const ZGemmArgs& a, cudaStream_t st) { launch_slices<double>(a, st); }

void cgemm_slices_f32(const CGemmArgs& a, cudaStream_t st) { launch_slices<float>(a, st); }

}  // namespace ts
