// Device-side building blocks of the tcgen05 kernels (gemm_tc.cu, gemm_oz.cu): mbarriers with
// bounded waits, TMA tensor loads, shared-memory matrix descriptors for 128-byte-swizzled K-major
// tiles, MMA issue / commit and tensor-memory loads; and the host-side tensor-map encoder.
#pragma once
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cstdint>
#include "internal.cuh"

namespace ts {
namespace tcg {

// Every mbarrier wait is bounded by elapsed time (the %globaltimer nanosecond clock): a stage of a
// healthy pipeline completes in microseconds, so a wait that lasts kWaitNs means a stalled pipeline.
constexpr unsigned long long kWaitNs = 1000000000ull;   // 1 s

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Bounded wait: returns false (and records `code` in *err unless an earlier code is there) when
// the phase has not completed within limit_ns nanoseconds.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int* err, int code,
                                          unsigned long long limit_ns = kWaitNs) {
  for (int i = 0; i < 64; ++i)
    if (mbar_try(bar, parity)) return true;
  const unsigned long long t0 = globaltimer_ns();
  for (;;) {
    if (mbar_try(bar, parity)) return true;
    __nanosleep(128);
    if (globaltimer_ns() - t0 > limit_ns) break;
  }
  atomicCAS(err, 0, code);
  return false;
}
// For a warp that issues MMAs with all its lanes converged (see mma_issue_one): the wait of every lane, and a
// result the compiler knows to be the same in all of them.  The part after the first look is out of line,
// so that an unrolled issue loop has a few instructions per wait.
static __device__ __noinline__ bool mbar_wait_call(uint32_t bar, uint32_t parity, int* err, int code,
                                                   unsigned long long limit_ns = kWaitNs) {
  return mbar_wait(bar, parity, err, code, limit_ns);
}
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, int* err, int code,
                                               unsigned long long limit_ns = kWaitNs) {
  const bool ok = mbar_try(bar, parity) || mbar_wait_call(bar, parity, err, code, limit_ns);
  return __all_sync(0xffffffffu, ok);
}
// A value that is the same in every lane, as one the compiler can keep in a uniform register.
__device__ __forceinline__ uint32_t warp_uniform(uint32_t v) { return __shfl_sync(0xffffffffu, v, 0); }
// True in one lane of the (converged) warp.
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t r;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(r));
  return r;
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* tm, int c0, int c1, int c2,
                                            uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(tm)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
      : "memory");
}

// Shared-memory matrix descriptor: K-major operand tile with 128-byte rows and the 128-byte
// swizzle TMA applied (8-row atoms of 1024 bytes; stride between atoms 1024 bytes).
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFFu);   // start address
  d |= (uint64_t)1 << 16;                   // leading byte offset (unused with this swizzle)
  d |= (uint64_t)(1024 >> 4) << 32;         // stride byte offset
  d |= (uint64_t)1 << 46;                   // descriptor version
  d |= (uint64_t)2 << 61;                   // 128-byte swizzle
  return d;
}

// The MMA and the commit as a converged warp issues them: every lane passes here with the same operands, the
// lane with `one` set (elect_one) executes.  The operands then stay in uniform registers, where the
// instruction wants them; from inside an `if (lane == 0)` each one is moved there again for every MMA.
__device__ __forceinline__ void mma_issue_one(uint32_t one, uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                              uint32_t acc, int kind_tf32) {
  if (kind_tf32) {
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
        " @q tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc), "r"(one));
  } else {
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc), "r"(one));
  }
}
__device__ __forceinline__ void mma_commit_one(uint32_t one, uint32_t bar) {
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.b32 q, %1, 0;\n"
      " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(bar),
      "r"(one)
      : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// Instruction descriptor (kind::f16 / kind::tf32): FP32 accumulator, both operands K-major.
__host__ __device__ constexpr uint32_t make_idesc(int fmt, int M, int N, bool negA) {
  return (1u << 4)                        // accumulator format: F32
         | ((uint32_t)fmt << 7)           // A format (1 = BF16, 2 = TF32)
         | ((uint32_t)fmt << 10)          // B format
         | ((negA ? 1u : 0u) << 13)       // negate A
         | ((uint32_t)(N >> 3) << 17)     // N / 8
         | ((uint32_t)(M >> 4) << 24);    // M / 16
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

}  // namespace tcg

// 3-D TMA map over planes [planes][rows][ld] of esz-byte elements (BF16 for esz 2, FP32 for 4):
// logical extent cols x rows x planes (elements beyond cols or rows read as zero), box = box_bytes (128 or
// 64) of the contiguous index x box_rows x 1, swizzle of the same width.
void make_map(CUtensorMap* m, const void* base, int esz, int ld, int cols, int rows, int planes, int box_rows,
              int box_bytes = 128);

}  // namespace ts
