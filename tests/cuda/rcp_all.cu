// Counts the floats d in [1, 2^125] whose rcp_1_up(d) is not 1.f / d (*worst: one of them, as bits).
#include "rcp.cuh"

__global__ void compare(unsigned first, unsigned last, unsigned long long* bad, unsigned* worst) {
  unsigned long long n = 0;
  for (unsigned long long b = first + blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; b <= last;
       b += (unsigned long long)gridDim.x * blockDim.x) {
    const float d = __uint_as_float((unsigned)b);
    if (__float_as_uint(fhmg::rcp_1_up(d)) != __float_as_uint(1.f / d)) {
      ++n;
      *worst = (unsigned)b;
    }
  }
  if (n) atomicAdd(bad, n);
}

extern "C" int rcp_compare(unsigned first, unsigned last, unsigned long long* bad_dev, unsigned* worst_dev) {
  compare<<<2048, 256>>>(first, last, bad_dev, worst_dev);
  if (cudaGetLastError() != cudaSuccess) return 1;
  return cudaDeviceSynchronize() == cudaSuccess ? 0 : 2;
}
