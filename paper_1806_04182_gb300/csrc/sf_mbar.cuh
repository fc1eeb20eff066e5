// Shared-memory mbarrier operations (PTX mbarrier.*), the bounded wait used by
// every kernel that waits on one, and a bulk L2 prefetch of row segments.  A
// wait that runs past its cycle limit gives up and reports false, so no
// kernel of this library can wait forever; the caller records the failure in
// the status word (ST_TIMEOUT).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace sf {

__device__ __forceinline__ uint32_t saddr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* b, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(b)), "r"(count) : "memory");
}

// Wait for the phase with the given parity, for at most `limit` clock cycles;
// false if it gave up.  (A loop in assembly is shorter code, but keeps every
// lane's result and cost the one-point CCZ4 kernels, which use this wait
// throughout, 1 to 3%: 59 x 46 x 53 step 258 against 251 us.)
__device__ __forceinline__ bool mbar_wait(uint64_t* b, unsigned parity, unsigned limit) {
  auto done = [&] {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n"
        " mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(saddr(b)), "r"(parity)
        : "memory");
    return ok != 0;
  };
  if (done()) return true;
  const long long t0 = clock64();
  while (!done())
    if (clock64() - t0 > limit) return false;
  return true;
}

// The same for a converged warp, without a result: every lane waits, and the
// branches are uniform (on a vote).  A wait that runs past the limit (less than
// 2^31 cycles) sets the shared word *gaveup; once it is set, no wait of the CTA
// spins any more.  The hot path is three instructions: the two-point kernels
// inline some fifty waits each, and their code only just fits the 128 KB from
// which an SM can stream instructions (see sf_z4_pair.cuh).
__device__ __forceinline__ void mbar_wait_warp(uint64_t* b, unsigned parity, unsigned limit,
                                               unsigned* gaveup) {
  asm volatile(
      "{\n .reg .pred p, q;\n .reg .b32 t0, t, g;\n"
      " mov.u32 t0, 0;\n"
      "AGAIN:\n"
      " mbarrier.try_wait.parity.shared::cta.b64 p, [%0], %1;\n"
      " vote.sync.all.pred p, p, 0xffffffff;\n"
      " @p bra.uni DONE;\n"
      " ld.volatile.shared.u32 g, [%3];\n"
      " mov.u32 t, %%clock;\n"
      " setp.eq.u32 q, t0, 0;\n"
      " @q or.b32 t0, t, 1;\n"
      " sub.u32 t, t, t0;\n"
      " setp.gt.s32 q, t, %2;\n"
      " setp.ne.or.u32 q, g, 0, q;\n"
      " vote.sync.any.pred q, q, 0xffffffff;\n"
      " @!q bra.uni AGAIN;\n"
      " st.volatile.shared.u32 [%3], 1;\n"
      "DONE:\n}\n" ::"r"(saddr(b)), "r"(parity), "r"(limit), "r"(saddr(gaveup))
      : "memory");
}

// One lane of a converged warp (the same every time).
__device__ __forceinline__ bool elect_one() {
  unsigned r;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(r));
  return r != 0;
}

// One arrival for a converged warp.
__device__ __forceinline__ void mbar_arrive_warp(uint64_t* b) {
  asm volatile(
      "{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n"
      " @p mbarrier.arrive.shared::cta.b64 _, [%0];\n}\n" ::"r"(saddr(b))
      : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(b)) : "memory");
}

__device__ __forceinline__ void mbar_expect(uint64_t* b, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(saddr(b)), "r"(bytes)
               : "memory");
}

// Bulk L2 prefetch of the 128-byte row segment of every field that the RK
// combination of this stage reads (U^n, the accumulator, the Kahan term):
// those reads come late in the point's computation, one field at a time, and
// would otherwise each wait for DRAM.
template <int kBytes = 144>
__device__ __forceinline__ void prefetch_rows(const float* base, long long F) {
  static_assert(kBytes % 16 == 0, "bulk prefetch size");
#pragma unroll 1
  for (int f = 0; f < 25; ++f)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(base + f * F), "n"(kBytes)
                 : "memory");
}

}  // namespace sf
