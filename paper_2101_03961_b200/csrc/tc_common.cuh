// Building blocks shared by the tensor-core kernels (expert GEMMs and the bfloat16-split router): inline-PTX wrappers
// for mbarrier, TMA (cp.async.bulk.tensor, never multicast), tcgen05 (alloc, mma, commit, ld, fences), the 128-byte
// swizzle shared-memory matrix descriptor, and the time-bounded barrier wait.
#pragma once

#include <cuda.h>

#include "switch_common.cuh"

namespace swmoe {
namespace tc {

constexpr int kBN = 256, kBK = 64, kStages = 4, kUmmaK = 16;
constexpr int kABytes = kTileM * kBK * 2;            // 16 KB
constexpr int kBBytes = kBN * kBK * 2;               // 32 KB
constexpr int kStageBytes = kABytes + kBBytes;       // 48 KB
constexpr int kAtomBytes = 64 * kBK * 2;             // one 64(MN) x 64(K) MN-major box: 8 KB
constexpr int kTmemCols = 512;
constexpr long long kWaitLimitCycles = 4000000000ll;          // about 2 s of SM clock per wait

// ---------------------------------------------------------------------------------------------- PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Non-blocking poll: cheaper than try_wait when the phase has already completed (the common case for a pipeline
// that is running ahead).
__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Bounded wait.  Returns false (after recording `code`) if the barrier did not flip within the limit or another
// thread of the CTA already gave up.  The common case -- the phase is complete, or completes within a few polls --
// is inline: producer and MMA loops must stay small and call-free, because a lone warp that jumps to far code pays an
// instruction-cache miss per iteration while the epilogue warps stream through the cache.
// kProgress: the limit starts anew whenever the word behind the abort flag has changed (long finite work elsewhere in the block).
template <bool kProgress = false>
static __device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status,
                                                   int code) {
  long long t0 = clock64();
  int seen = kProgress ? abort_flag[1] : 0;
  for (uint32_t spin = 1;; ++spin) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((spin & 255u) == 0) {
      if (*abort_flag != 0) return false;
      if (kProgress && abort_flag[1] != seen) {
        seen = abort_flag[1];
        t0 = clock64();
      }
      if (clock64() - t0 > kWaitLimitCycles) {
        *abort_flag = 1;
        if (atomicCAS(status, 0, code) == 0) {
          status[1] = (int)blockIdx.x;
          status[2] = (int)parity;
        }
        __threadfence();
        return false;
      }
    }
  }
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status,
                                          int code) {
  if (mbar_test_wait(bar, parity)) return true;
#pragma unroll 1
  for (int i = 0; i < 32; ++i)
    if (mbar_try_wait(bar, parity)) return true;
  return mbar_wait_slow(bar, parity, abort_flag, status, code);
}

// The same bounded wait for a whole converged warp.  The TMA and MMA warps run their loops with all 32 lanes and elect
// one lane only around the instructions themselves: what they feed to those instructions (descriptors, coordinates,
// barrier addresses) is then warp-uniform for the compiler and stays in uniform registers.  A loop that a single lane
// runs inside a divergent branch has to move every operand of every tcgen05.mma over from vector registers, which cost
// about 1000 cycles per 64-deep k-block of the expert products whatever the loads and the tensor pipe did (GEMM1 at
// 32768 tokens, 768 x 3072, 128 experts: 189 us with single-lane loops, 162 us with these).  The polls sit in one asm
// block so that no divergent branch separates the lanes.
template <bool kProgress = false>
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status,
                                               int code) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t.reg .u32 c;\n\t"
      "mov.u32 c, 0;\n\t"
      "WAIT_LOOP:\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "@p bra WAIT_DONE;\n\t"
      "add.u32 c, c, 1;\n\t"
      "setp.lt.u32 q, c, 64;\n\t"
      "@q bra WAIT_LOOP;\n\t"
      "WAIT_DONE:\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  if (__all_sync(0xffffffffu, ok != 0)) return true;
  return __all_sync(0xffffffffu, mbar_wait_slow<kProgress>(bar, parity, abort_flag, status, code));
}
// True in one lane of a converged warp, always the same one (tcgen05.commit covers the MMAs of its own thread).
__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(pred));
  return pred != 0;
}
// The warp's index within its block, uniform for the compiler.
__device__ __forceinline__ int uniform_warp_id() { return __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0); }

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(tm)), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tc_mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void tc_ld32(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor, 128-byte swizzle.  Offsets are in bytes; the fields hold them divided by 16.
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32;
  d |= 1ull << 46;                                           // descriptor version for this architecture
  d |= 2ull << 61;                                           // layout: 128-byte swizzle
  return d;
}


// bf16 tensor [E][rows][cols] (cols contiguous), box {64 cols, box_rows rows, 1}, 128-byte swizzle, zero OOB fill.
int make_map(CUtensorMap* tm, const void* base, long long E, long long rows, long long cols, int box_rows);
// float32 tensor [E][rows][cols], box {box_cols, box_rows, 1}, zero OOB fill; 128-byte swizzle where a box row is 128 bytes.
int make_map_f32(CUtensorMap* tm, const void* base, long long E, long long rows, long long cols, int box_cols, int box_rows);

}  // namespace tc
}  // namespace swmoe
