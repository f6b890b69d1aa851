// transport_x32.cu -- FP32 transport with polarization or with the mean-intensity tally (compiled
// like the FP32 production kernels).
#include "transport_x.cuh"

namespace mcrt {
MCRT_TRANSPORT_X(float)

cudaError_t launch_transport_warp_j(const KParams<float>& P, int warps, cudaStream_t st) {
  transport_warp_kernel<false, true><<<warps, 32, 0, st>>>(P);
  return cudaGetLastError();
}

int transport_warps_per_sm_j() {
  int n = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, transport_warp_kernel<false, true>, 32, 0);
  return n;
}
}  // namespace mcrt
