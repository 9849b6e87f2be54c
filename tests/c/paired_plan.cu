// For each number of x points given: the launch plan of the packed single-precision kernel with
// N_k = 32 on this device, printed as "x points, CTAs per x point of the last wave, blocks".
#include <cstdio>
#include <cstdlib>

#include "../../paper_2205_02380_gb300/csrc/internal.hpp"

int main(int argc, char** argv) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 1;
  for (int i = 1; i < argc; ++i) {
    chasm::ThetaPlan p;
    chasm::theta_pk_plan(32, std::atoll(argv[i]), sms, &p);
    std::printf("%s %d %d\n", argv[i], p.cluster, p.blocks);
  }
  return 0;
}
