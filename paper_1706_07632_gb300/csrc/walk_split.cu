// Launcher of the tensor-core defect by digit splitting (split.cuh).
#include <cstdio>
#include <string>

#include "split.cuh"
#include "walk.h"

namespace fhmg {

namespace {
constexpr int kPrepRows = 2;  // grid rows per thread of the pre-pass (2D)
KernelCache g_split_cache;
}

int split_defect_launch(cudaStream_t st, const SplitArgs& a0, std::string* err) {
  if (a0.M % kSplitRows != 0 || a0.M > kSplitMaxM || a0.ld < 1 || !a0.U || !a0.F || !a0.OUT || !a0.fe || !a0.At ||
      !a0.pairs || !a0.rexp) {
    if (err) *err = "split defect: unsupported arguments";
    return 2;
  }
  SplitArgs a = a0;
  a.ntiles = (a.ld + kSpCols - 1) / kSpCols;
  if (a.spin <= 0) a.spin = kSpinLimit;
  const int sms = device_sms();
  // the exponents of u per grid point and B = F - A_h u into OUT
  cudaError_t e = cudaMemsetAsync(a.fe, 0, sizeof(int) * a.ld, st);
  if (e == cudaSuccess) {
    const unsigned bx = (a.N + kPrepThreads - 1) / kPrepThreads, bz = (a.M + kPrepM - 1) / kPrepM;
    if (a.dim == 2)
      split_prep_kernel<2, kPrepRows><<<dim3(bx, (a.N + kPrepRows - 1) / kPrepRows, bz), kPrepThreads, 0, st>>>(
          a.U, a.F, a.OUT, a.fe, a.ld, a.M, a.N, a.inv_h2);
    else
      split_prep_kernel<1, 1><<<dim3(bx, 1, bz), kPrepThreads, 0, st>>>(a.U, a.F, a.OUT, a.fe, a.ld, a.M, a.N, a.inv_h2);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) {
    if (err) *err = std::string("split_prep_kernel: ") + cudaGetErrorString(e);
    return 1;
  }
  a.ns = 5;
  const size_t smem = split_smem(a.ns).total + 1024;  // + the alignment of the swizzled tiles
  int occ = 1;
  e = prepare_launch(split_defect_kernel, kSpBlock, smem, g_split_cache, &occ);
  if (e != cudaSuccess) {
    if (err) *err = std::string("split_defect_kernel attributes: ") + cudaGetErrorString(e);
    return 1;
  }
  const long long grid = std::min<long long>(a.ntiles, (long long)sms * occ);
  split_defect_kernel<<<(unsigned)grid, kSpBlock, smem, st>>>(a);
  e = cudaGetLastError();
  if (e != cudaSuccess) {
    if (err) *err = std::string("split_defect_kernel: ") + cudaGetErrorString(e);
    return 1;
  }
  return 0;
}

}  // namespace fhmg
