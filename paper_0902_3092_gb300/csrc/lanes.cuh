// lanes.cuh -- the threads that share a sum or a sweep: one (the host), or a warp (the kernels), lane l taking the elements
// l, l + size, ... The same code then serves both, and the host tests run what the kernels run.
#pragma once
#include <cmath>

namespace mcrt {

struct OneLane {
  __host__ __device__ int lane() const { return 0; }
  __host__ __device__ int size() const { return 1; }
  __host__ __device__ double below(double, double carry) const { return carry; }   // the previous lane's x
  __host__ __device__ double upto(double x, double carry) const { return carry + x; }  // carry + the lanes' sum so far
  __host__ __device__ double last(double x) const { return x; }                      // the last lane's x
  __host__ __device__ double sum(double x) const { return x; }
  __host__ __device__ double max(double x) const { return x; }
};

#if defined(__CUDACC__)
struct WarpLanes {
  __device__ int lane() const { return (int)(threadIdx.x & 31u); }
  __device__ int size() const { return 32; }
  __device__ double below(double x, double carry) const {
    const double v = __shfl_up_sync(0xffffffffu, x, 1);
    return lane() == 0 ? carry : v;
  }
  // In the order of the lanes, one addition after another: near the pole the terms of the hydrostatic potential are 1e7
  // times the differences that matter, so another order of the sum has other roundings (1e-9 of the density).
  __device__ double upto(double x, double carry) const {
    double mine = carry;
#pragma unroll
    for (int l = 0; l < 32; ++l) {
      carry += __shfl_sync(0xffffffffu, x, l);
      if (lane() == l) mine = carry;
    }
    return mine;
  }
  __device__ double last(double x) const { return __shfl_sync(0xffffffffu, x, 31); }
  __device__ double sum(double x) const {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
  }
  __device__ double max(double x) const {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = fmax(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
  }
};
#endif

}  // namespace mcrt
