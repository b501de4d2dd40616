// The sweeps' reciprocal over a range of float bit patterns: the largest relative
// error against the FP64 division.
#include "cl_sweep.cuh"

__global__ void k_recip_error(unsigned first, unsigned count, unsigned long long* worst) {
  double e = 0.0;
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
    const float v = __uint_as_float(first + i);
    e = fmax(e, fabs((double)clk::recip(v) * (double)v - 1.0));
  }
  atomicMax(worst, (unsigned long long)__double_as_longlong(e));  // non-negative doubles order like their bits
}

extern "C" int recip_error(unsigned first, unsigned count, unsigned long long* worst) {
  k_recip_error<<<608, 256>>>(first, count, worst);
  return cudaDeviceSynchronize() == cudaSuccess ? 0 : 1;
}
