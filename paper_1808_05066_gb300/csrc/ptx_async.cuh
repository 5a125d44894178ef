// PTX wrappers for mbarriers and bulk asynchronous copies (cp.async.bulk), shared by the
// kernels that stream operands into shared memory. Every wait is bounded by its caller.
#pragma once
#include <cstdint>

#ifndef HDG_DEVI
#define HDG_DEVI __device__ __forceinline__
#endif

namespace hdg {

HDG_DEVI uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

HDG_DEVI void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
HDG_DEVI bool mbar_try(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
HDG_DEVI unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Waits for the phase of the given parity to complete: `spins` polls, then polls 256 ns apart; gives up after a
// second. The limit is a time because a poll that fails may itself suspend the thread for microseconds (4M polls
// took 4 to 16 s); the number of polls is bounded as well. One loop: with a second one for the timed polls
// k_asm_t5 takes 0.9 ms more (of 103, 82,944 tetrahedra, p = 3). The time is read right after a failed poll, not after the
// sleep: a kernel that was not running meanwhile polls once more.
HDG_DEVI bool mbar_wait(uint64_t* bar, uint32_t parity, int spins = 64) {
  unsigned end = 0;  // in 2^20 ns
  for (int i = 0; i < 1 << 22; ++i) {
    if (mbar_try(bar, parity)) return true;
    if (i > spins) {
      const unsigned t = (unsigned)(global_ns() >> 20);
      if (end == 0) end = t + 1000;
      if ((int)(t - end) > 0) break;
      __nanosleep(256);
    }
  }
  return false;
}
HDG_DEVI void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// Bulk asynchronous copy global -> shared of `bytes` (multiple of 16, both addresses 16-byte
// aligned), completing as transaction bytes on `bar`.
HDG_DEVI void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
HDG_DEVI void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
HDG_DEVI void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

}  // namespace hdg
