// Device pieces shared by the network's tcgen05 kernels: asynchronous copies, bounded
// barrier waits, operand descriptors, tensor-memory loads.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace bfcs {
namespace net {

constexpr int kTcWorkers = 256;                       // staging / epilogue threads (warps 0-7); warp 8 issues MMAs
constexpr unsigned kTcSpinLimit = 1u << 26;           // bound of every mbarrier wait

__device__ __forceinline__ void cp16(unsigned dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int LEFT> __device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(LEFT) : "memory");
}
__device__ __forceinline__ void fence_async() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }
__device__ __forceinline__ void tc_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void tc_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }

__device__ __forceinline__ bool elect_one() {
  unsigned p;
  asm volatile("{\n.reg .pred q;\nelect.sync _|q, 0xffffffff;\nselp.u32 %0, 1, 0, q;\n}\n" : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
// Bounded wait of a whole warp for the phase of the given parity; gives up early once *fail
// is set.  The result is the same in all lanes (an expired limit in one of them counts for
// all): the tensor-memory loads that follow a wait are warp-wide instructions.
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, volatile int* fail) {
  unsigned done = 0, spins = 0;
  bool ok = true;
  while (!done) {
    asm volatile(
        "{\n.reg .pred q;\nmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\nselp.u32 %0, 1, 0, q;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (!done && (++spins > kTcSpinLimit || *fail)) { ok = false; break; }
  }
  return __all_sync(0xffffffffu, ok);
}
// barrier of the worker warps; true when the predicate held in all of them
__device__ __forceinline__ bool workers_all(bool ok) {
  unsigned r;
  asm volatile(
      "{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbarrier.cta.red.and.pred q, 1, %2, p;\nselp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((unsigned)ok), "n"(kTcWorkers)
      : "memory");
  return r != 0;
}

__device__ __forceinline__ uint64_t sdesc(unsigned saddr, unsigned lbo, unsigned sbo) {
  // start address, leading (K) and stride (M/N) byte offsets in 16-byte units,
  // descriptor version 1 (bit 46), no swizzle, base offset 0
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
}
// instruction descriptor of kind::f16: D FP32 (bits 4-5 = 1), A and B BF16
// (bits 7-9 and 10-12 = 1), both K-major, N >> 3 at bit 17, M >> 4 at bit 24
constexpr unsigned idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(N >> 3) << 17) | ((unsigned)(M >> 4) << 24);
}
// operand descriptor of the 64-byte swizzle (layout type 4 at bit 61)
constexpr uint64_t kDescSwizzle64 = (uint64_t)4 << 61;
// both operands MN-major (bits 15 and 16)
constexpr unsigned kIdescMnMajorAB = (1u << 15) | (1u << 16);

// 16-byte copy, or 16 zero bytes
__device__ __forceinline__ void cp16_fill(unsigned dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(valid ? 16u : 0u) : "memory");
}

// 16 columns of this warp's 32 tensor-memory lanes
__device__ __forceinline__ void tmem_ld16(unsigned* v, unsigned taddr) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}

}  // namespace net
}  // namespace bfcs
