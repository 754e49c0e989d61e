// Waits on shared-memory barriers that end: each has a limit in clock cycles, and a block that gives up says so.
#pragma once
#include <cstdint>

namespace dslide {

// About a second at the highest clock.  A count of tries is no limit: how long a try may sleep is the hardware's choice.
constexpr long long WAIT_CYCLES = 2000000000LL;
constexpr long long DRAIN_CYCLES = 20000000LL;       // for what is in flight when a block has given up: copies and multiplications take microseconds

__device__ __forceinline__ uint32_t tc_smem(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// A try may sleep up to 2 us, so that a waiting warp issues little (all-neuron calls of 128 samples x 100,003 neurons x 512 units
// 101.6 us without, 99.8 with; 1,024 x 100,003 x 64 109.3 and 108.3).
// CLUSTER: what the arrivals' threads of the other blocks of the cluster had done is then visible too.
template <bool CLUSTER = false>
__device__ __forceinline__ bool tc_bar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  if (CLUSTER)
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity), "r"(2000u) : "memory");
  else asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(ok) : "r"(bar), "r"(parity), "r"(2000u) : "memory");
  return ok != 0u;
}
// True once the phase of that parity has completed, false when it has not within the limit.
__device__ __forceinline__ bool bar_wait_limited(uint64_t* bar, uint32_t parity) {
  const uint32_t a = tc_smem(bar);
  if (tc_bar_try(a, parity)) return true;
  const long long t0 = clock64();
  while (!tc_bar_try(a, parity))
    if (clock64() - t0 > WAIT_CYCLES) return false;
  return true;
}
// The same by a whole warp: one answer for all lanes, true where all have seen the phase complete.  (Each lane looks at the clock for
// itself; one that gives up must not leave the others to exchange values without it.)
__device__ __forceinline__ bool bar_wait_limited_warp(uint64_t* bar, uint32_t parity) {
  const bool ok = bar_wait_limited(bar, parity);
  return __all_sync(0xffffffffu, ok) != 0;
}
// Sets the flag of this block and, in a pair (PAIR: a cluster of two blocks), of the other one.
template <bool PAIR>
__device__ __forceinline__ void tc_give_up(volatile int* abort) {
  *abort = 1;
  if (PAIR)
    asm volatile("{\n\t.reg .b32 r, a;\n\tmov.u32 r, %%cluster_ctarank;\n\txor.b32 r, r, 1;\n\tmapa.shared::cluster.u32 a, %0, r;\n\t"
                 "st.relaxed.cluster.shared::cluster.b32 [a], %1;\n\t}" ::"r"(tc_smem(const_cast<int*>(abort))), "r"(1) : "memory");
}
// True once the phase of that parity has completed.  False when it has not within the limit -- the flag is then set -- or when
// another wait of the block, or of the pair, has given up: every later wait returns at once.
template <bool PAIR, bool CLUSTER = false>
__device__ __forceinline__ bool tc_bar_wait(uint64_t* bar, uint32_t parity, volatile int* abort) {
  const uint32_t a = tc_smem(bar);
  if (tc_bar_try<CLUSTER>(a, parity)) return true;
  const long long t0 = clock64();
  while (!tc_bar_try<CLUSTER>(a, parity)) {
    if (*abort) return false;
    if (clock64() - t0 > WAIT_CYCLES) { tc_give_up<PAIR>(abort); return false; }
  }
  return true;
}
// The same by a whole warp, one answer for all lanes: true where all of them have seen the phase complete.  A lane that has
// seen the flag, or that a wait has kept longer, is with the others again for what follows: an election, or an instruction that
// takes the whole warp.
template <bool PAIR, bool CLUSTER = false>
__device__ __forceinline__ bool tc_bar_wait_warp(uint64_t* bar, uint32_t parity, volatile int* abort) {
  const bool ok = tc_bar_wait<PAIR, CLUSTER>(bar, parity, abort);
  __syncwarp();
  return __all_sync(0xffffffffu, ok) != 0;
}
// For a block that has given up: it waits until the time `until`, whatever the flag says.
__device__ __forceinline__ void tc_bar_drain(uint64_t* bar, uint32_t parity, long long until) {
  while (!tc_bar_try(tc_smem(bar), parity) && clock64() < until) {}
}

}  // namespace dslide
