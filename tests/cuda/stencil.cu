// sp_stencil over n rows of NX + 1 FP64 values (the point, then its neighbours).
#include "split.cuh"

template <int NX>
__global__ void run(const unsigned long long* v, double* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  unsigned long long x[NX];
  for (int k = 0; k < NX; ++k) x[k] = v[i * (NX + 1) + 1 + k];
  out[i] = fhmg::sp_stencil<NX>(v[i * (NX + 1)], x);
}

extern "C" int stencil(int nx, const unsigned long long* v, double* out, int n) {
  if (nx == 2)
    run<2><<<(n + 127) / 128, 128>>>(v, out, n);
  else
    run<4><<<(n + 127) / 128, 128>>>(v, out, n);
  if (cudaGetLastError() != cudaSuccess) return 1;
  return cudaDeviceSynchronize() == cudaSuccess ? 0 : 2;
}
