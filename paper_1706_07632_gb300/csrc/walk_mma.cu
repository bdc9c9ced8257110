// Launchers of the tensor-core panel walk (FP32 products, leaf 64, column tile 16 or 32).
#include <algorithm>
#include <string>

#include "mma.cuh"
#include "walk.h"

namespace fhmg {
namespace {

constexpr size_t kMmaSmemMax = 227 * 1024;

template <typename T, int TC, int MODE, int XS = 2, bool MEM = MODE == MODE_SMOOTH>
int mma_launch_t(cudaStream_t st, WalkBatch<T, float>& B, std::string* err) {
  auto kern = hmma_kernel<T, TC, MODE, XS, MEM>;
  constexpr int kBlock = mma_threads(TC, MEM);
  constexpr int kRhs = MEM ? sizeof(T) : 0;
  // A short chunk ring leaves the SM's memory to the L1 cache, whose lines the neighbour loads in flight
  // hold: with 2 slots for tile 32 a 255^2 x 1024 FP32 solve takes 117.8 ms (3 slots 119.1, 4 120.1, 8 121.5),
  // with 3 for tile 16, whose chunks are used up twice as fast, a batch of 16 solves of up to 1023 columns x
  // M = 1024 takes 73.1 ms (2 slots 74.0, 4 73.5, 8 73.8)
  constexpr int kSlots = TC == 32 ? 2 : 3;
  const size_t other = mma_smem(TC, XS, B.pool, B.W, B.slot_bytes, 0, kRhs).total + 64;
  int ns = other < kMmaSmemMax ? (int)((kMmaSmemMax - other) / (size_t)B.slot_bytes) : 0;
  ns = std::min(ns, kSlots);
  // many live z values (a high rank) or a wide near field: first tile 32's TF32 pairs give way, then
  // the memory warps' buffers
  if constexpr (TC == 32 && XS == 2) {
    if (ns < 2) return mma_launch_t<T, TC, MODE, 1, MEM>(st, B, err);
  } else if constexpr (MEM) {
    if (ns < 2) return mma_launch_t<T, TC, MODE, XS, false>(st, B, err);
  }
  if (ns < 2) {
    *err = "tensor-core walk: no room for two chunk slots in shared memory";
    return 2;
  }
  B.ns = ns;
  const size_t smem = mma_smem(TC, XS, B.pool, B.W, B.slot_bytes, ns, kRhs).total;
  static KernelCache cache;
  int occ = 1;
  {
    cudaError_t e = prepare_launch(kern, kBlock, smem, cache, &occ);
    if (e != cudaSuccess) {
      *err = std::string("tensor-core walk set-up: ") + cudaGetErrorString(e);
      return 1;
    }
  }
  if (B.ntiles <= 0) return 0;
  const long long grid = std::min<long long>(B.ntiles, (long long)device_sms() * occ);
  cudaError_t e = launch_sized(kern, grid, kBlock, smem, occ, st, B);
  if (e != cudaSuccess) {
    *err = std::string("tensor-core walk launch: ") + cudaGetErrorString(e);
    return 1;
  }
  return 0;
}

template <typename T>
int mma_dispatch(cudaStream_t st, WalkBatch<T, float>& B, int TC, int mode, std::string* err) {
  if (TC == 16) return mode == MODE_SMOOTH ? mma_launch_t<T, 16, MODE_SMOOTH>(st, B, err)
                                           : mma_launch_t<T, 16, MODE_MATVEC>(st, B, err);
  if (TC == 32) return mode == MODE_SMOOTH ? mma_launch_t<T, 32, MODE_SMOOTH>(st, B, err)
                                           : mma_launch_t<T, 32, MODE_MATVEC>(st, B, err);
  *err = "tensor-core walk: column tile must be 16 or 32";
  return 2;
}

}  // namespace

int mma_launch_df(cudaStream_t st, WalkBatch<double, float>& B, int TC, int mode, std::string* err) {
  return mma_dispatch<double>(st, B, TC, mode, err);
}
int mma_launch_ff(cudaStream_t st, WalkBatch<float, float>& B, int TC, int mode, std::string* err) {
  return mma_dispatch<float>(st, B, TC, mode, err);
}

}  // namespace fhmg
