// Asynchronous copies into shared memory and their mbarriers, with bounded waits.
#pragma once

#include "common.cuh"

namespace {

DEV uint32_t s_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

DEV unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

DEV void mbar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(s_addr(bar)), "r"(count) : "memory");
}
DEV void mbar_arrive_tx(uint64_t* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(s_addr(bar)), "r"(bytes) : "memory");
}
DEV void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(s_addr(bar)) : "memory");
}
// wait for the phase of parity `par` to complete; false after ~1 s (or once another
// thread of the CTA gave up), with the CTA's abort flag set
DEV bool mbar_wait(uint64_t* bar, unsigned par, volatile int* abort) {
  const uint32_t a = s_addr(bar);
  unsigned long long t0 = 0;  // the clock is read only once a wait is long
  for (unsigned it = 0;; ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(a), "r"(par)
        : "memory");
    if (done) return true;
    if ((it & 255) == 255) {
      if (*abort) return false;
      if (t0 == 0) t0 = now_ns();
      if (now_ns() - t0 > 1000000000ull) {
        *abort = 1;
        return false;
      }
    }
  }
}

// contiguous copy global -> shared: 16-byte aligned addresses, bytes a multiple of 16
DEV void bulk_load(void* dst, const void* src, unsigned bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   s_addr(dst)),
               "l"(__cvta_generic_to_global(src)), "r"(bytes), "r"(s_addr(bar))
               : "memory");
}

}  // namespace
