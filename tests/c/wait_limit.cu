// The waits of csrc/group_bar.cuh on the device.  Two warps share a barrier; with `partner` both
// arrive, otherwise only warp 0 does and the phase never ends.  Prints, for both forms of the wait:
// whether a wait ran out, and the nanoseconds of the first wait and of the one after it.
#include <cstdio>
#include <cuda_runtime.h>

#include "../../paper_2205_02380_gb300/csrc/group_bar.cuh"

using namespace chasm;

__device__ long long nanoseconds() {
  long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

template <bool FIRST>
__global__ void k_wait(int partner, int tries, long long* out) {
  __shared__ __align__(8) unsigned long long bar;
  __shared__ int gone[2];
  const unsigned b = sm_addr(&bar);
  if (threadIdx.x == 0) {
    mb_init(b, 2);
    gone[0] = gone[1] = 0;
  }
  __syncthreads();
  if (threadIdx.x < 32 || partner) mb_arrive(b);
  const long long t0 = nanoseconds();
  mb_wait<FIRST>(b, 0, gone, tries);
  const long long t1 = nanoseconds();
  __syncthreads();
  const int ran_out = gone[0] + 2 * gone[1];
  const long long t2 = nanoseconds();
  mb_wait<FIRST>(b, partner ? 0 : 2, gone, tries);
  const long long t3 = nanoseconds();
  if (threadIdx.x == 0) {
    out[0] = ran_out;
    out[1] = t1 - t0;
    out[2] = t3 - t2;
  }
}

template <bool FIRST>
int run(int partner, int tries) {
  long long *d, h[3];
  if (cudaMalloc(&d, sizeof(h)) != cudaSuccess) return 1;
  k_wait<FIRST><<<1, 64>>>(partner, tries, d);
  if (cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
  cudaFree(d);
  std::printf("%d %d %lld %lld %lld\n", partner, tries, h[0], h[1], h[2]);
  return 0;
}

int main() {
  int bad = 0;
  for (int partner = 1; partner >= 0; --partner) bad |= run<false>(partner, 64) | run<true>(partner, 64);
  bad |= run<false>(0, kWaitTries);
  return bad;
}
