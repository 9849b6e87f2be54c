// Barriers between the warps of a group: mbarriers in shared memory, whose waits end.
#pragma once

namespace chasm {
namespace {

__device__ __forceinline__ unsigned sm_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mb_init(unsigned b, int warps) {
  asm volatile("mbarrier.init.shared.b64 [%0], %1;" ::"r"(b), "r"(warps) : "memory");
}
// this warp's arrival: what its lanes did before is visible to whoever waits for the phase
__device__ __forceinline__ void mb_arrive(unsigned b) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0) asm volatile("mbarrier.arrive.shared.b64 _, [%0];" ::"r"(b) : "memory");
  __syncwarp();
}
__device__ __forceinline__ bool mb_try(unsigned b, int parity) {
  unsigned done;
  asm volatile("{\n .reg .pred q;\n mbarrier.try_wait.parity.shared.b64 q, [%1], %2;\n selp.u32 %0, 1, 0, q;\n}"
               : "=r"(done)
               : "r"(b), "r"(parity & 1)
               : "memory");
  return done != 0;
}
// A try that does not succeed returns after 3.9 us (measured, the same with a shorter or a longer
// time hint), so a wait gives up after about a second.
constexpr int kWaitTries = 1 << 18;
// Waits for the end of a phase of this parity.  A wait that runs out sets gone[0] and gone[1] (in shared
// memory); gone[1] stays set and ends every later wait of the block after one try, so that a kernel
// whose partner never comes ends about a second later and not a second per wait.  The words are looked
// at only after a try that failed: carried in a register, the outcome cost the callers spills (double
// precision P(dt) at 24^3 x 16^3 11.07 -> 11.48 ms).  FIRST: the first try stands before the loop.
template <bool FIRST = false>
__device__ __forceinline__ void mb_wait(unsigned b, int parity, volatile int* gone, int tries = kWaitTries) {
  bool done = FIRST && mb_try(b, parity);
  if (!FIRST || !done) {
    int i = 0;
    do done = mb_try(b, parity);
    while (!done && ++i < tries && !gone[1]);
    if (!done) gone[0] = gone[1] = 1;
  }
  __syncwarp();
}

}  // namespace
}  // namespace chasm
