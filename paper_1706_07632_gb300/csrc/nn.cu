// Learned warm start: a small spectral network, trained and run by the kernels of this file.
//
// For a source that is constant in time and a finite sine series, f = sum_pq c_pq s_pq(x, y),
// each spatial eigenmode s_pq of A_h (eigenvalue lam_pq) is carried independently through the
// time discretisation: u = sum_pq c_pq w_pq(t) s_pq with (R + lam_pq I) w_pq = 1.  The network
// predicts y = lam * w(t) in [0, 1) from features of (lam, alpha, t); the warm start projects f
// onto the K x K leading modes, evaluates the network for every (mode, time level) and
// synthesises u0 = sum_pq c_pq w_pq(t_m) s_pq.  Multigrid then solves from u0 and measures
// its error (and is the fallback: u0 = 0).
//
// Network: F = 6 input features -> H -> H -> H -> 1, SiLU activations, FP32 training (Adam), FP32
// or BF16 inference.  Layer l maps width n_l to n_{l+1} with weights W_l (n_{l+1} x n_l,
// row-major) and bias b_l; all parameters live in one FP32 array in layer order (W_0, b_0, W_1,
// b_1, ...).  Kernels: FP32 GEMM (64 x 64 tiles, 8 x 4 per thread, both transposes; bias, SiLU and its
// derivative in the epilogue; weight gradients split over the rows, with the bias gradients), the
// output layer's two passes, MSE loss, Adam; the BF16 network in one tcgen05 kernel (mlp_bf16), a BF16
// tensor-core GEMM per layer for the widths it does not serve; feature build, spectral projection and
// synthesis.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <random>
#include <string>
#include <utility>
#include <vector>

#include "devinfo.h"
#include "rcp.cuh"
#include "umma.cuh"
#include "fhmg.h"

// Kernel launches issued by this file (network training / inference, warm-start projection and
// synthesis), reported by fhmg_wsnet_launches.
static std::atomic<long long> g_nn_launches{0};

int fhmg_internal_fail(int code, const char* msg);

namespace {

constexpr int kFeat = 6;

#define NCK(x)                                                                     \
  do {                                                                             \
    cudaError_t e_ = (x);                                                          \
    if (e_ != cudaSuccess) return fhmg_internal_fail(FHMG_ECUDA, cudaGetErrorString(e_)); \
  } while (0)

__device__ __forceinline__ float sigm(float x) { return 1.f / (1.f + __expf(-x)); }

// the FP64 value of a float by integer operations (the conversion runs on the 1/64-rate FP64 pipe);
// subnormals and non-finite values by the conversion
__device__ __forceinline__ double f2d_exact(float f) {
  const uint32_t b = __float_as_uint(f), m = b & 0x7FFFFFFFu;
  if (m - 0x00800000u >= 0x7F000000u) return m == 0 ? __hiloint2double((int)b, 0) : (double)f;
  return __hiloint2double((int)((b & 0x80000000u) | ((m >> 3) + (896u << 20))), (int)(b << 29));
}

// FP32 GEMM arguments: op(A) (M x K) op(B) (K x N); A stored K x M when transposed, B stored N x K when
// transposed.  Batches and splits run along blockIdx.z.
struct GemmArgs {
  int M, N, K;
  float alpha;
  const float* A;
  const float* B;
  float* C;
  int lda, ldb, ldc;
  long long sA, sB, sC;  // elements between batches
  int kper;              // reduction length per split (a multiple of the K tile), or K
  const float* bias;     // EPI_ACT: bias per column; EPI_ACTB: Z (ldc) of the layer below
  float* out2;           // EPI_ACT: the activations (ldc); EPI_SPLIT: column sums of op(A)^T per split
  int act;               // EPI_ACT: SiLU or none
  double* out64;         // EPI_F64
};
// what is written: alpha C | z = C + bias and its activation | C * SiLU'(Z) | partial sums of a split
// | C widened to FP64 (out64, batch stride sC; thread columns 16 apart, so that a row's stores are contiguous)
enum { EPI_PLAIN = 0, EPI_ACT = 1, EPI_ACTB = 2, EPI_SPLIT = 3, EPI_F64 = 4 };

constexpr int kGB = 64, kGK = 16, kGThreads = 128, kGLd = kGB + 4;

// Tiles of 64 x 64 x 16, 128 threads of 8 x 4 accumulators, the next K tile loaded into registers while
// one is multiplied, shared memory double-buffered, 16-byte global loads where the operand allows them.
// Every sum runs over k in order.  The previous kernel (256 threads of 4 x 4, scalar loads, one
// buffer) took 2.0 ms for the eleven products of a training step at batch 4096 and width 320, most of
// it in the three weight gradients, whose 25 tiles each summed 4096 rows on 25 SMs; the weight
// gradients are now split over the rows (EPI_SPLIT, then reduce_splits_kernel).  Training step with
// bias, activation and their derivatives in the epilogues: 2.52 -> 0.35 ms.
template <bool TA, bool TB, int EPI>
__global__ void __launch_bounds__(kGThreads) gemm_f32(const GemmArgs g) {
  __shared__ __align__(16) float As[2][kGK][kGLd];
  __shared__ __align__(16) float Bs[2][kGK][kGLd];
  const int t = threadIdx.x, tx = t % 16, ty = t / 16;
  const int m0 = blockIdx.y * kGB, n0 = blockIdx.x * kGB;
  const float* A = g.A;
  const float* Bm = g.B;
  float* C = g.C;
  int k0 = 0, k1 = g.K;
  if (EPI == EPI_SPLIT) {
    k0 = blockIdx.z * g.kper;
    k1 = min(g.K, k0 + g.kper);
    C += (long long)blockIdx.z * g.sC;
  } else {
    A += blockIdx.z * g.sA;
    Bm += blockIdx.z * g.sB;
    C += blockIdx.z * g.sC;
  }
  const bool va = (g.lda & 3) == 0 && (reinterpret_cast<uintptr_t>(A) & 15) == 0;
  const bool vb = (g.ldb & 3) == 0 && (reinterpret_cast<uintptr_t>(Bm) & 15) == 0;
  // one 4-vector of a tile: along the rows of the stored matrix, `along` its index there (limit `lim`),
  // `row` the other one
  auto load4 = [](const float* X, int ld, bool vec, int row, int rows, int along, int lim, float (&v)[4]) {
    const float* p = X + (long long)row * ld + along;
    if (row < rows && vec && along + 3 < lim) {
      const float4 q = __ldg(reinterpret_cast<const float4*>(p));
      v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = row < rows && along + e < lim ? __ldg(p + e) : 0.f;
    }
  };
  float ra[2][4], rb[2][4];
  auto fetch = [&](int k) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      if (TA)
        load4(A, g.lda, va, k + t / 16 + 8 * i, k1, m0 + (t % 16) * 4, g.M, ra[i]);
      else
        load4(A, g.lda, va, m0 + t / 4 + 32 * i, g.M, k + (t % 4) * 4, k1, ra[i]);
      if (TB)
        load4(Bm, g.ldb, vb, n0 + t / 4 + 32 * i, g.N, k + (t % 4) * 4, k1, rb[i]);
      else
        load4(Bm, g.ldb, vb, k + t / 16 + 8 * i, k1, n0 + (t % 16) * 4, g.N, rb[i]);
    }
  };
  auto stage = [&](int b) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      if (TA) {
        *reinterpret_cast<float4*>(&As[b][t / 16 + 8 * i][(t % 16) * 4]) = make_float4(ra[i][0], ra[i][1], ra[i][2], ra[i][3]);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) As[b][(t % 4) * 4 + e][t / 4 + 32 * i] = ra[i][e];
      }
      if (TB) {
#pragma unroll
        for (int e = 0; e < 4; ++e) Bs[b][(t % 4) * 4 + e][t / 4 + 32 * i] = rb[i][e];
      } else {
        *reinterpret_cast<float4*>(&Bs[b][t / 16 + 8 * i][(t % 16) * 4]) = make_float4(rb[i][0], rb[i][1], rb[i][2], rb[i][3]);
      }
    }
  };
  float acc[8][4] = {};
  float csum = 0.f;  // EPI_SPLIT: this thread's column of op(A)^T
  fetch(k0);
  stage(0);
  __syncthreads();
  int b = 0;
  for (int k = k0; k < k1; k += kGK, b ^= 1) {
    const bool next = k + kGK < k1;
    if (next) fetch(k + kGK);
#pragma unroll
    for (int kk = 0; kk < kGK; ++kk) {
      const float4 a0 = *reinterpret_cast<const float4*>(&As[b][kk][ty * 8]);
      const float4 a1 = *reinterpret_cast<const float4*>(&As[b][kk][ty * 8 + 4]);
      float4 bb;
      if (EPI == EPI_F64)
        bb = make_float4(Bs[b][kk][tx], Bs[b][kk][tx + 16], Bs[b][kk][tx + 32], Bs[b][kk][tx + 48]);
      else
        bb = *reinterpret_cast<const float4*>(&Bs[b][kk][tx * 4]);
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w}, bv[4] = {bb.x, bb.y, bb.z, bb.w};
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] += av[i] * bv[j];
    }
    if (EPI == EPI_SPLIT && blockIdx.x == 0 && t < kGB) {
#pragma unroll
      for (int kk = 0; kk < kGK; ++kk) csum += As[b][kk][t];
    }
    if (next) stage(b ^ 1);
    __syncthreads();
  }
  if (EPI == EPI_F64) {
    double* D = g.out64 + blockIdx.z * g.sC;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int gm = m0 + ty * 8 + i;
      if (gm >= g.M) break;
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (n0 + tx + 16 * j < g.N) D[(long long)gm * g.ldc + n0 + tx + 16 * j] = f2d_exact(acc[i][j]);
    }
    return;
  }
  const bool v4 = (g.ldc & 3) == 0 && (reinterpret_cast<uintptr_t>(C) & 15) == 0 &&
                  (EPI != EPI_ACT || (reinterpret_cast<uintptr_t>(g.out2) & 15) == 0);
  const int gn = n0 + tx * 4;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int gm = m0 + ty * 8 + i;
    if (gm >= g.M) break;
    const long long o = (long long)gm * g.ldc + gn;
    float c[4], a2[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const bool in = gn + j < g.N;
      c[j] = EPI == EPI_PLAIN ? g.alpha * acc[i][j] : acc[i][j];
      if (EPI == EPI_ACT) {
        c[j] += in ? __ldg(g.bias + gn + j) : 0.f;
        a2[j] = g.act ? c[j] * sigm(c[j]) : c[j];
      } else if (EPI == EPI_ACTB) {
        const float z = in ? __ldg(g.bias + o + j) : 0.f, sg = sigm(z);
        c[j] = c[j] * sg * (1.f + z * (1.f - sg));
      }
    }
    if (v4 && gn + 3 < g.N) {
      *reinterpret_cast<float4*>(C + o) = make_float4(c[0], c[1], c[2], c[3]);
      if (EPI == EPI_ACT) *reinterpret_cast<float4*>(g.out2 + o) = make_float4(a2[0], a2[1], a2[2], a2[3]);
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (gn + j < g.N) {
          C[o + j] = c[j];
          if (EPI == EPI_ACT) g.out2[o + j] = a2[j];
        }
    }
  }
  if (EPI == EPI_SPLIT && blockIdx.x == 0 && t < kGB && m0 + t < g.M)
    g.out2[(long long)blockIdx.z * g.sC + m0 + t] = csum;
}

// g[j] = sum over the splits of part[s][j], j < n
__global__ void reduce_splits_kernel(int splits, long long n, const float* __restrict__ part, float* __restrict__ g) {
  const long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (j >= n) return;
  float s = 0.f;
#pragma unroll 8
  for (int i = 0; i < splits; ++i) s += part[i * n + j];
  g[j] = s;
}

// Output layer of width 1: y = A w + b, a warp per row
__global__ void __launch_bounds__(256) out_layer_fwd(int n, int w, const float* __restrict__ A,
                                                     const float* __restrict__ W, const float* __restrict__ b,
                                                     float* __restrict__ Z, float* __restrict__ Y) {
  const int i = blockIdx.x * 8 + threadIdx.x / 32, lane = threadIdx.x % 32;
  if (i >= n) return;
  float s = 0.f;
  for (int k = lane; k < w; k += 32) s += A[(long long)i * w + k] * __ldg(W + k);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) {
    s += __ldg(b);
    Z[i] = s;
    Y[i] = s;
  }
}

// Backward of the output layer over kOutRows rows per blockIdx.y, thread per column j of the layer
// below: dZ = dy w_j SiLU'(Z), and this block's part of dW (w columns) and db (behind them)
constexpr int kOutRows = 64;
__global__ void __launch_bounds__(128) out_layer_bwd(int n, int w, int act, const float* __restrict__ dy,
                                                     const float* __restrict__ W, const float* __restrict__ A,
                                                     const float* __restrict__ Z, float* __restrict__ dZ,
                                                     float* __restrict__ part) {
  const int j = blockIdx.x * 128 + threadIdx.x, i0 = blockIdx.y * kOutRows, i1 = min(n, i0 + kOutRows);
  if (j > w) return;
  float s = 0.f;
  if (j == w) {
    for (int i = i0; i < i1; ++i) s += __ldg(dy + i);
  } else {
    const float wj = __ldg(W + j);
#pragma unroll 8
    for (int i = i0; i < i1; ++i) {
      const long long o = (long long)i * w + j;
      const float d = __ldg(dy + i);
      s += d * A[o];
      if (act) {
        const float z = Z[o], sg = sigm(z);
        dZ[o] = d * wj * sg * (1.f + z * (1.f - sg));
      }
    }
  }
  part[(long long)blockIdx.y * (w + 1) + j] = s;
}

// BF16 inference GEMM with FP32 accumulation: C (M x N) = A (M x K, row-major bf16) * W^T
// (W: N x K, row-major bf16), one 16 x 8 tensor-core tile (mma.sync m16n8k16) per warp step.
__global__ void __launch_bounds__(128) gemm_bf16_nt(int M, int N, int K, const __nv_bfloat16* A,
                                                    const __nv_bfloat16* W, float* C) {
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int m0 = (blockIdx.y * 4 + warp) * 16;
  const int n0 = blockIdx.x * 8;
  if (m0 >= M) return;
  float c[4] = {0.f, 0.f, 0.f, 0.f};
  const int g = lane / 4, q = lane % 4;
  for (int k0 = 0; k0 < K; k0 += 16) {
    auto ldA = [&](int r, int k) -> __nv_bfloat16 {
      return (r < M && k < K) ? A[(long long)r * K + k] : __float2bfloat16(0.f);
    };
    auto ldW = [&](int n, int k) -> __nv_bfloat16 {
      return (n < N && k < K) ? W[(long long)n * K + k] : __float2bfloat16(0.f);
    };
    // fragment layout of m16n8k16 (row.col): a0..a7, b0..b3 per thread
    __nv_bfloat162 a01 = __halves2bfloat162(ldA(m0 + g, k0 + 2 * q), ldA(m0 + g, k0 + 2 * q + 1));
    __nv_bfloat162 a23 = __halves2bfloat162(ldA(m0 + g + 8, k0 + 2 * q), ldA(m0 + g + 8, k0 + 2 * q + 1));
    __nv_bfloat162 a45 = __halves2bfloat162(ldA(m0 + g, k0 + 2 * q + 8), ldA(m0 + g, k0 + 2 * q + 9));
    __nv_bfloat162 a67 = __halves2bfloat162(ldA(m0 + g + 8, k0 + 2 * q + 8), ldA(m0 + g + 8, k0 + 2 * q + 9));
    __nv_bfloat162 b01 = __halves2bfloat162(ldW(n0 + g, k0 + 2 * q), ldW(n0 + g, k0 + 2 * q + 1));
    __nv_bfloat162 b23 = __halves2bfloat162(ldW(n0 + g, k0 + 2 * q + 8), ldW(n0 + g, k0 + 2 * q + 9));
    const unsigned ra0 = *reinterpret_cast<unsigned*>(&a01), ra1 = *reinterpret_cast<unsigned*>(&a23);
    const unsigned ra2 = *reinterpret_cast<unsigned*>(&a45), ra3 = *reinterpret_cast<unsigned*>(&a67);
    const unsigned rb0 = *reinterpret_cast<unsigned*>(&b01), rb1 = *reinterpret_cast<unsigned*>(&b23);
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(ra0), "r"(ra1), "r"(ra2), "r"(ra3), "r"(rb0), "r"(rb1));
  }
  const int r0 = m0 + g, r1 = m0 + g + 8, cc = n0 + 2 * q;
  if (r0 < M && cc < N) C[(long long)r0 * N + cc] = c[0];
  if (r0 < M && cc + 1 < N) C[(long long)r0 * N + cc + 1] = c[1];
  if (r1 < M && cc < N) C[(long long)r1 * N + cc] = c[2];
  if (r1 < M && cc + 1 < N) C[(long long)r1 * N + cc + 1] = c[3];
}

// BF16 inference layer with the bias and the activation fused: out = SiLU(A W^T + b), A (M x K) and
// W (N x K) row-major BF16 (16-byte aligned rows), b FP32, K % 32 == 0, N % 64 == 0.  Block tile
// 128 x 64; K tiles of 32 double-buffered in shared memory by cp.async (rows padded to 80 bytes:
// the fragment loads below hit 32 distinct banks); 8 warps of 32 x 32, each a 2 x 4 grid of
// mma.sync m16n8k16 tiles with FP32 accumulation, k16 steps in the same order as gemm_bf16_nt; the
// epilogue adds b, applies SiLU and writes BF16 (the same FP32 operations as bias_act_fwd).
__global__ void __launch_bounds__(256) gemm_bf16_silu(int M, int N, int K, const __nv_bfloat16* __restrict__ A,
                                                      const __nv_bfloat16* __restrict__ W,
                                                      const float* __restrict__ bias, __nv_bfloat16* out) {
  constexpr int BM = 128, BN = 64, BK = 32, LDS = BK + 8;
  __shared__ __align__(16) __nv_bfloat16 sA[2][BM * LDS];
  __shared__ __align__(16) __nv_bfloat16 sW[2][BN * LDS];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int wm = warp & 3, wn = warp >> 2;
  const int g = lane >> 2, q = lane & 3;
  const long long m0 = (long long)blockIdx.y * BM;
  const int n0 = blockIdx.x * BN;
  auto load_tile = [&](int buf, int k0) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {  // A: 128 rows x 4 chunks of 16 bytes
      const int c = tid + i * 256;
      const int r = c >> 2, kc = (c & 3) * 8;
      const long long gr = m0 + r;
      const bool ok = gr < M;
      const __nv_bfloat16* src = A + (ok ? gr : 0LL) * K + k0 + kc;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                       (uint32_t)__cvta_generic_to_shared(&sA[buf][r * LDS + kc])),
                   "l"(src), "r"(ok ? 16 : 0)
                   : "memory");
    }
    {  // W: 64 rows x 4 chunks
      const int r = tid >> 2, kc = (tid & 3) * 8;
      const __nv_bfloat16* src = W + (long long)(n0 + r) * K + k0 + kc;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                       (uint32_t)__cvta_generic_to_shared(&sW[buf][r * LDS + kc])),
                   "l"(src)
                   : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  auto lds32 = [](const __nv_bfloat16* p) -> uint32_t { return *reinterpret_cast<const uint32_t*>(p); };
  float acc[2][4][4];
#pragma unroll
  for (int mi = 0; mi < 2; ++mi)
#pragma unroll
    for (int ni = 0; ni < 4; ++ni)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[mi][ni][j] = 0.f;
  const int nk = K / BK;
  load_tile(0, 0);
  for (int kt = 0; kt < nk; ++kt) {
    if (kt + 1 < nk) {
      load_tile((kt + 1) & 1, (kt + 1) * BK);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const __nv_bfloat16* a = sA[kt & 1];
    const __nv_bfloat16* w = sW[kt & 1];
#pragma unroll
    for (int ks = 0; ks < BK; ks += 16) {
      uint32_t af[2][4], bf[4][2];
#pragma unroll
      for (int mi = 0; mi < 2; ++mi) {
        const int r = wm * 32 + mi * 16 + g;
        af[mi][0] = lds32(a + r * LDS + ks + 2 * q);
        af[mi][1] = lds32(a + (r + 8) * LDS + ks + 2 * q);
        af[mi][2] = lds32(a + r * LDS + ks + 2 * q + 8);
        af[mi][3] = lds32(a + (r + 8) * LDS + ks + 2 * q + 8);
      }
#pragma unroll
      for (int ni = 0; ni < 4; ++ni) {
        const int c = wn * 32 + ni * 8 + g;
        bf[ni][0] = lds32(w + c * LDS + ks + 2 * q);
        bf[ni][1] = lds32(w + c * LDS + ks + 2 * q + 8);
      }
#pragma unroll
      for (int mi = 0; mi < 2; ++mi)
#pragma unroll
        for (int ni = 0; ni < 4; ++ni)
          asm volatile(
              "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
              "{%0,%1,%2,%3};"
              : "+f"(acc[mi][ni][0]), "+f"(acc[mi][ni][1]), "+f"(acc[mi][ni][2]), "+f"(acc[mi][ni][3])
              : "r"(af[mi][0]), "r"(af[mi][1]), "r"(af[mi][2]), "r"(af[mi][3]), "r"(bf[ni][0]), "r"(bf[ni][1]));
    }
    __syncthreads();  // this buffer is refilled two tiles on
  }
#pragma unroll
  for (int mi = 0; mi < 2; ++mi)
#pragma unroll
    for (int ni = 0; ni < 4; ++ni) {
      const int c = n0 + wn * 32 + ni * 8 + 2 * q;
      const float b0 = bias[c], b1 = bias[c + 1];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const long long r = m0 + wm * 32 + mi * 16 + g + 8 * h;
        if (r >= M) continue;
        const float z0 = acc[mi][ni][2 * h] + b0, z1 = acc[mi][ni][2 * h + 1] + b1;
        *reinterpret_cast<__nv_bfloat162*>(out + r * N + c) = __floats2bfloat162_rn(z0 * sigm(z0), z1 * sigm(z1));
      }
    }
}

// The whole BF16 network on 128 rows at a time, on the tcgen05 tensor cores: input layer, hidden layers
// of width H and output layer, activations (BF16, SiLU) kept in shared memory between them.  Every
// layer is a batch of MMAs (M = 128 rows, N = the layer's width, FP32 accumulators in tensor memory) by
// one warp, then an epilogue by eight warps (bias, SiLU, rounding, the next layer's A operand in the
// 128-byte swizzle).  The hidden weights pass through a two-stage ring of K tiles of 64 (bulk copies of
// the operand layout, prepared by pack_weights); the input layer's (K = 6, padded to 16), the output
// layer's (one row, padded to 16) and the biases stay in shared memory.  The sums run over k16 steps in
// order and round as mma.sync m16n8k16 does here: the results are those of the one-launch-per-layer path bit
// for bit (tests/test_gpu_network_paths.py).  Bound by the epilogues (two special-function operations per activation).  294912 rows of
// width 320: 1.25 ms over six launches; fused with mma.sync 0.74 ms; 0.34 ms now.
struct MlpArgs {
  int n, layers;                    // rows, hidden layers
  const float* X;                   // n x kFeat
  const unsigned char* W;           // pack_weights
  const float* P;                   // parameters in FP32 (biases)
  long long boff[9];
  float* Y;
  int* err;                         // set if a bounded wait gives up
  long long spin, withhold;         // polls of the MMA and epilogue warps' waits; 1-based tile never loaded (test hook)
};

// kMlpMaxH: the widest multiple of 64 for which every depth the network may have (8 hidden layers) fits in shared
// memory: 200 KB at 320, where 384 would fit up to three layers only (tensor memory would hold 448).
constexpr int kMlpRows = 128, kMlpMaxH = 320, kMlpEpi = 256, kMlpBlock = kMlpEpi + 64;
// bytes of the packed weights: input layer (H x 16), output layer (16 x H), then per hidden layer H / 64
// tiles of H x 64
__host__ __device__ inline size_t mlp_packed(int H, int layers) {
  return (size_t)H * 16 * 2 * 2 + (size_t)(layers - 1) * H * H * 2;
}
struct MlpSmem {
  size_t act, ring, win, wout, xin, bias, bar, total;
};
__host__ __device__ inline MlpSmem mlp_smem(int H, int layers) {
  MlpSmem s;
  s.act = 0;
  s.ring = (size_t)kMlpRows * H * 2;
  s.win = s.ring + 2 * (size_t)H * 128;
  s.wout = s.win + (size_t)H * 32;
  s.xin = s.wout + (size_t)H * 32;
  s.bias = s.xin + (size_t)kMlpRows * 32;
  s.bar = s.bias + (size_t)(layers * H + 4) * 4;
  s.total = s.bar + 8 * 7 + 16;
  return s;
}

// BF16 copies of the weights as MMA operands (W_0: no swizzle, K = 16; W_out and the hidden layers: 64-column
// tiles, 128-byte swizzle), padding zero
__global__ void pack_weights(int H, int layers, const float* __restrict__ P, unsigned char* __restrict__ out) {
  const long long hid = (long long)(layers - 1) * H * H, total = 32LL * H + hid;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    float v = 0.f;
    size_t o;
    if (i < 16LL * H) {
      const int r = (int)(i / 16), k = (int)(i % 16);
      if (k < kFeat) v = P[r * kFeat + k];
      o = fhmg::umma_off(r, k, 16);
    } else if (i < 32LL * H) {
      const int r = (int)((i - 16LL * H) / H), k = (int)((i - 16LL * H) % H);
      if (r == 0) v = P[(long long)(kFeat + 1) * H + (long long)(layers - 1) * (H + 1) * H + k];
      o = (size_t)H * 32 + (size_t)(k / 64) * 16 * 128 + fhmg::sw128_off(r, k % 64);
    } else {
      const long long j = i - 32LL * H;
      const int l = (int)(j / ((long long)H * H)), r = (int)(j % ((long long)H * H) / H), k = (int)(j % H);
      v = P[(long long)(kFeat + 1) * H + (long long)l * (H + 1) * H + (long long)r * H + k];
      o = (size_t)H * 64 + (size_t)l * H * H * 2 + (size_t)(k / 64) * H * 128 + fhmg::sw128_off(r, k % 64);
    }
    *reinterpret_cast<__nv_bfloat16*>(out + o) = __float2bfloat16(v);
  }
}

__global__ void __launch_bounds__(kMlpBlock, 1) mlp_bf16(int H, const __grid_constant__ MlpArgs g) {
  using namespace fhmg;
  extern __shared__ __align__(16) unsigned char smraw[];
  unsigned char* sm = smraw + ((1024u - (smem_u32(smraw) & 1023u)) & 1023u);  // swizzled tiles: 1024-byte aligned
  const MlpSmem lay = mlp_smem(H, g.layers);
  unsigned char* act = sm + lay.act;
  float* bias = reinterpret_cast<float*>(sm + lay.bias);
  uint64_t* wfull = reinterpret_cast<uint64_t*>(sm + lay.bar);  // [2]
  uint64_t* wfree = wfull + 2;                                   // [2]
  uint64_t* aready = wfull + 4;                                  // the A operand of the next batch is complete
  uint64_t* accdone = wfull + 5;                                 // a batch's MMAs are complete
  uint64_t* donebar = wfull + 6;                                 // every MMA issued is complete
  volatile int* abort_flag = reinterpret_cast<volatile int*>(wfull + 7);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(wfull + 7) + 1;
  const int t = threadIdx.x, w = t >> 5, lane = t & 31;
  const int KT = H / 64, nhid = g.layers - 1;
  const uint32_t tcols = H + 16 <= 128 ? 128 : H + 16 <= 256 ? 256 : 512;
  if (t == 0) {
    for (int s = 0; s < 2; ++s) {
      mbar_init(wfull + s, 1);
      mbar_init(wfree + s, 1);
    }
    mbar_init(aready, kMlpEpi / 32);
    mbar_init(accdone, 1);
    mbar_init(donebar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // the resident operands: packed input and output layers, biases, the zero half of the input rows
  for (int i = t; i < H * 64 / 16; i += kMlpBlock)
    reinterpret_cast<uint4*>(sm + lay.win)[i] = __ldg(reinterpret_cast<const uint4*>(g.W) + i);
  for (int i = t; i <= g.layers * H; i += kMlpBlock) bias[i] = __ldg(g.P + g.boff[i / H] + i % H);
  if (t < kMlpRows) *reinterpret_cast<uint4*>(sm + lay.xin + umma_off(t, 8, 16)) = make_uint4(0, 0, 0, 0);
  if (w == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)), "r"(tcols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  async_proxy_fence();
  tc_before_sync();
  __syncthreads();
  tc_after_sync();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tslot, 0);
  const int blocks = (g.n + kMlpRows - 1) / kMlpRows;
  auto raise = [&]() {
    *abort_flag = 1;
    atomicExch(g.err, 1);
  };
  if (w == kMlpEpi / 32) {
    // ---- producer: the hidden layers' K tiles, for every row block ----
    if (lane == 0) {
      const uint32_t bytes = (uint32_t)H * 128;
      int slot = 0;
      uint32_t phase = 1;
      long long k = 0;
      bool ok = true, stop = false;
      for (int blk = blockIdx.x; blk < blocks && ok && !stop; blk += gridDim.x)
        for (int j = 0; j < nhid * KT; ++j, ++k) {
          if (k + 1 == g.withhold) {
            stop = true;
            break;
          }
          if (!mbar_wait_or_abort(wfree + slot, phase, abort_flag)) {
            ok = false;
            break;
          }
          bulk_load(sm + lay.ring + (size_t)slot * bytes, g.W + (size_t)H * 64 + (size_t)j * bytes, bytes, wfull + slot);
          slot ^= 1;
          phase ^= slot ^ 1;
        }
      if (!ok) raise();
      for (int s = 0; s < 2 && s < k; ++s) mbar_wait(wfull + s, (uint32_t)(((k - 1 - s) / 2) & 1));
    }
    __syncwarp();
  } else if (w == kMlpEpi / 32 + 1) {
    // ---- MMA warp (uniform; one elected lane issues) ----
    const bool leader = umma_elect();
    const int N0 = H < 256 ? H : 256, N1 = H - N0;
    int slot = 0;
    uint32_t fphase = 0, aphase = 0;
    bool ok = true;
    auto wait = [&](uint64_t* bar, uint32_t ph) -> bool {
      ok = __all_sync(0xffffffffu, mbar_wait_or_abort(bar, ph, abort_flag, g.spin));
      tc_after_sync();
      return ok;
    };
    auto mma = [&](uint32_t d, uint64_t ad, uint64_t bd, uint32_t idesc, bool accumulate) {
      asm volatile(
          "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
          " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
          "l"(ad), "l"(bd), "r"(idesc), "r"(accumulate ? 1u : 0u)
          : "memory");
    };
    for (int blk = blockIdx.x; blk < blocks && ok; blk += gridDim.x) {
      for (int l = 0; l <= g.layers; ++l) {
        if (!wait(aready, aphase)) break;
        aphase ^= 1;
        if (l == 0) {
          if (leader) {
            umma_product(tmem, smem_u32(sm + lay.xin), smem_u32(sm + lay.win), 16, N0, false);
            if (N1) umma_product(tmem + 256, smem_u32(sm + lay.xin), smem_u32(sm + lay.win) + 256 * 32, 16, N1, false);
          }
        } else if (l <= nhid) {
          for (int kt = 0; kt < KT; ++kt) {
            if (!wait(wfull + slot, fphase)) break;
            const uint64_t ad = sw128_desc(smem_u32(act) + (uint32_t)kt * kMlpRows * 128);
            const uint64_t bd = sw128_desc(smem_u32(sm + lay.ring) + (uint32_t)slot * H * 128);
            if (leader) {
#pragma unroll
              for (int st = 0; st < 4; ++st) mma(tmem, ad + 2 * st, bd + 2 * st, umma_idesc(N0), kt + st > 0);
              if (N1) {
#pragma unroll
                for (int st = 0; st < 4; ++st)
                  mma(tmem + 256, ad + 2 * st, bd + (256 * 128 >> 4) + 2 * st, umma_idesc(N1), kt + st > 0);
              }
              umma_commit(wfree + slot);
            }
            slot ^= 1;
            fphase ^= slot ^ 1;
          }
          if (!ok) break;
        } else {
          if (leader)
            for (int kt = 0; kt < KT; ++kt) {
              const uint64_t ad = sw128_desc(smem_u32(act) + (uint32_t)kt * kMlpRows * 128);
              const uint64_t bd = sw128_desc(smem_u32(sm + lay.wout) + (uint32_t)kt * 16 * 128);
#pragma unroll
              for (int st = 0; st < 4; ++st) mma(tmem + H, ad + 2 * st, bd + 2 * st, umma_idesc(16), kt + st > 0);
            }
        }
        if (leader) umma_commit(accdone);
      }
    }
    if (!ok && leader) raise();
    if (leader) umma_commit(donebar);
    mbar_wait(donebar, 0);
  } else {
    // ---- epilogue warps: lane quarter w % 4 (rows), column half w / 4 ----
    const uint32_t lane_base = (uint32_t)(32 * (w & 3)) << 16;
    const int row = 32 * (w & 3) + lane, c0 = (w >> 2) * (H / 2);
    uint32_t dphase = 0;
    bool failed = false;
    auto ready = [&]() {
      async_proxy_fence();
      tc_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(aready);
    };
    auto put_x = [&](int blk) {  // the block's input rows (BF16) by the first column half
      if (w < 4) {
        const long long r = (long long)blk * kMlpRows + row;
        float2 a = make_float2(0.f, 0.f), b = a, c = a;
        if (r < g.n) {
          const float2* x = reinterpret_cast<const float2*>(g.X + r * kFeat);
          a = __ldg(x), b = __ldg(x + 1), c = __ldg(x + 2);
        }
        *reinterpret_cast<uint4*>(sm + lay.xin + umma_off(row, 0, 16)) =
            make_uint4(pack_bf16(a.x, a.y), pack_bf16(b.x, b.y), pack_bf16(c.x, c.y), 0u);
      }
      ready();
    };
    if ((int)blockIdx.x < blocks) put_x(blockIdx.x);
    for (int blk = blockIdx.x; blk < blocks && !failed; blk += gridDim.x) {
      for (int l = 0; l <= g.layers; ++l) {
        if (!__all_sync(0xffffffffu, mbar_wait_or_abort(accdone, dphase, abort_flag, g.spin))) {
          if (lane == 0) raise();
          failed = true;
          break;
        }
        dphase ^= 1;
        tc_after_sync();
        if (l == g.layers) {  // the output
          float v[16];
          tmem_ld16(tmem + lane_base + H, v);
          const long long r = (long long)blk * kMlpRows + row;
          if (w < 4 && r < g.n) g.Y[r] = v[0] + bias[g.layers * H];
          if (blk + (int)gridDim.x < blocks) put_x(blk + gridDim.x);
          continue;
        }
        for (int c = c0; c < c0 + H / 2; c += 16) {
          float v[16];
          tmem_ld16(tmem + lane_base + c, v);
          const float4* bp = reinterpret_cast<const float4*>(bias + l * H + c);
#pragma unroll
          for (int j = 0; j < 16; j += 4) {
            const float4 b = bp[j / 4];
            v[j] += b.x, v[j + 1] += b.y, v[j + 2] += b.z, v[j + 3] += b.w;
          }
          // SiLU as sigm() computes it, the division only beyond the reciprocal's range
          float d[16], dmax = 0.f;
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            d[j] = 1.f + __expf(-v[j]);
            dmax = fmaxf(dmax, d[j]);
          }
          if (__any_sync(0xffffffffu, dmax > 0x1p125f)) {
#pragma unroll
            for (int j = 0; j < 16; ++j) d[j] = 1.f / d[j];
          } else {
#pragma unroll
            for (int j = 0; j < 16; ++j) d[j] = fhmg::rcp_1_up(d[j]);
          }
#pragma unroll
          for (int j = 0; j < 16; ++j) v[j] = v[j] * d[j];
          unsigned char* dst = act + (size_t)(c / 64) * kMlpRows * 128;
#pragma unroll
          for (int j = 0; j < 16; j += 8)
            *reinterpret_cast<uint4*>(dst + sw128_off(row, c % 64 + j)) =
                make_uint4(pack_bf16(v[j], v[j + 1]), pack_bf16(v[j + 2], v[j + 3]), pack_bf16(v[j + 4], v[j + 5]),
                           pack_bf16(v[j + 6], v[j + 7]));
        }
        ready();
      }
    }
  }
  // every wait above is bounded, so every warp gets here, with the MMAs complete
  tc_before_sync();
  __syncthreads();
  tc_after_sync();
  if (w == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tcols));
  // after a wait gave up: none of this CTA's rows keeps what the array held before (here and not where the
  // epilogue gives up: in its loop the branch cost 14 of 338 us for 294912 rows)
  if (*abort_flag && t < kMlpRows)
    for (int blk = blockIdx.x; blk < blocks; blk += gridDim.x)
      if (t < g.n - blk * kMlpRows) g.Y[blk * kMlpRows + t] = __int_as_float(0x7FC00000);
}

// Z += b (row broadcast); A = SiLU(Z) (act = 1) or Z (act = 0).  Z kept for the backward pass.
__global__ void bias_act_fwd(int n, int w, float* Z, const float* b, float* A, int act, __nv_bfloat16* Abf) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)n * w;
       i += (long long)gridDim.x * blockDim.x) {
    const float z = Z[i] + b[i % w];
    Z[i] = z;
    const float a = act ? z * sigm(z) : z;
    if (A) A[i] = a;
    if (Abf) Abf[i] = __float2bfloat16(a);
  }
}

// loss = mean (y - t)^2 (accumulated into *loss), dY = 2 (y - t) / n
__global__ void mse_fwd_bwd(int n, const float* y, const float* t, float* dy, float* loss) {
  float s = 0.f;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float d = y[i] - t[i];
    if (dy) dy[i] = 2.f * d / n;
    s += d * d;
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(loss, s / n);
}

__global__ void adam_step(long long n, float* p, const float* g, float* m, float* v, float lr, float b1, float b2,
                          float c1, float c2, float eps) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

__global__ void to_bf16(long long n, const float* x, __nv_bfloat16* y) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    y[i] = __float2bfloat16(x[i]);
}

int nblk(long long n) { return fhmg::grid_for(n, 16); }

}  // namespace

// Features of (lam, alpha, t), all O(1): log10(lam)/5, alpha, log10(t)/5 (t > 0), s/(1+s),
// log1p(s)/10 with s = lam t^alpha, t^alpha.  What depends on the mode or the time level alone comes
// from a table (the FP64 pipe runs at 1/64 of the FP32 rate): `loglam` per mode, `ta` = t^alpha and
// `logt` per level.
__device__ __forceinline__ void ws_features(double lam, float loglam, double alpha, double ta, float logt, float* f) {
  const double s = lam * ta;
  f[0] = loglam;
  f[1] = (float)alpha;
  f[2] = logt;
  f[3] = (float)(s / (1.0 + s));
  f[4] = (float)(log1p(s) / 10.0);
  f[5] = (float)ta;
}

__global__ void feature_tables(int nm, const double* lam, int M, const double* t, double alpha, float* loglam, double* ta,
                               float* logt) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < nm) loglam[i] = (float)(log10(lam[i]) / 5.0);
  if (i < M) {
    ta[i] = pow(t[i + 1], alpha);
    logt[i] = (float)(log10(t[i + 1]) / 5.0);
  }
}

struct fhmg_wsnet_s {
  int hidden = 0, layers = 0;     // hidden width, number of hidden layers
  std::vector<int> width;         // n_0 = kFeat, ..., n_L = 1
  std::vector<long long> woff, boff;
  long long nparams = 0;
  float* P = nullptr;             // parameters
  float* G = nullptr;             // gradients
  float* Mo = nullptr;            // Adam moments
  float* Vo = nullptr;
  __nv_bfloat16* Pbf = nullptr;   // BF16 copy of the weights (inference)
  unsigned char* Wpk = nullptr;   // the weights as MMA operands: widths 64, 128, .., kMlpMaxH (mlp_bf16)
  int* err = nullptr;             // set by mlp_bf16 if a bounded wait gave up: [0] in a prediction, [1] in a forward call
  long long inj_spin = 0;         // armed test hook: the next mlp_bf16 withholds a weight tile, waits poll inj_spin times
  long long step = 0;
  // activations for a batch of up to cap rows, owned by act
  int cap = 0;
  std::vector<void*> act;
  std::vector<float*> Z, A, dA;   // per layer
  float* part = nullptr;          // partial sums of split weight gradients (part_n floats, not in allocs): as many as
  size_t part_n = 0;              // the largest batch so far needs
  float* loss = nullptr;
  __nv_bfloat16* Abf[2] = {nullptr, nullptr};
  // scratch of predictions, kept from call to call (the i-th buffer a prediction asks for, grown when it
  // asks for more): every prediction ends synchronised, also one that fails on the way, so no two use it at a
  // time unless the net itself is shared by threads, which its other buffers exclude
  std::vector<std::pair<void*, size_t>> ws;
  std::vector<void*> allocs;
};

namespace {

template <typename T>
int nalloc(std::vector<void*>& owner, T** p, size_t n) {
  cudaError_t e = cudaMalloc((void**)p, (n ? n : 1) * sizeof(T));
  if (e != cudaSuccess) {
    cudaGetLastError();  // not sticky; keep it out of the next launch check
    return fhmg_internal_fail(FHMG_ENOMEM, cudaGetErrorString(e));
  }
  owner.push_back(*p);
  return FHMG_OK;
}

// Activations for batches of n rows.  The smaller ones are freed first (which waits for the device); where the
// larger do not fit, the network is left without any, so that the next call allocates what it needs.
int ensure_cap(fhmg_wsnet net, int n) {
  if (n <= net->cap) return FHMG_OK;
  const int L = (int)net->width.size() - 1;
  for (void* p : net->act) cudaFree(p);
  net->act.clear();
  net->cap = 0;
  net->Z.assign(L, nullptr);
  net->A.assign(L + 1, nullptr);
  net->dA.assign(L + 1, nullptr);
  int maxw = 0;
  for (int w : net->width) maxw = w > maxw ? w : maxw;
  int s = FHMG_OK;
  for (int l = 0; l < L && s == FHMG_OK; ++l) {
    const size_t m = (size_t)n * net->width[l + 1];
    if ((s = nalloc(net->act, &net->Z[l], m)) == FHMG_OK && (s = nalloc(net->act, &net->A[l + 1], m)) == FHMG_OK)
      s = nalloc(net->act, &net->dA[l + 1], m);
  }
  for (int i = 0; i < 2 && s == FHMG_OK; ++i) s = nalloc(net->act, &net->Abf[i], (size_t)n * maxw);
  if (s != FHMG_OK) {
    for (void* p : net->act) cudaFree(p);
    net->act.clear();
    return s;
  }
  net->cap = n;
  return FHMG_OK;
}

template <bool TA, bool TB, int EPI>
int gemm_launch(cudaStream_t st, const GemmArgs& g, int batch) {
  const dim3 grid((g.N + kGB - 1) / kGB, (g.M + kGB - 1) / kGB, batch);
  gemm_f32<TA, TB, EPI><<<grid, kGThreads, 0, st>>>(g);
  ++g_nn_launches;
  NCK(cudaGetLastError());
  return FHMG_OK;
}

// C (M x N, ldc) = alpha op(A) op(B), at most one of them transposed, batched with the given element
// strides
int gemm(cudaStream_t st, int M, int N, int K, float alpha, const float* A, int lda, int ta, const float* B, int ldb,
         int tb, float* C, int ldc, int batch = 1, long long sA = 0, long long sB = 0, long long sC = 0) {
  GemmArgs g{};
  g.M = M, g.N = N, g.K = K, g.alpha = alpha;
  g.A = A, g.B = B, g.C = C, g.lda = lda, g.ldb = ldb, g.ldc = ldc;
  g.sA = sA, g.sB = sB, g.sC = sC;
  if (ta) return gemm_launch<true, false, EPI_PLAIN>(st, g, batch);
  return tb ? gemm_launch<false, true, EPI_PLAIN>(st, g, batch) : gemm_launch<false, false, EPI_PLAIN>(st, g, batch);
}

// out (M x N, ldc; FP64) = op(A) op(B), batched
int gemm_to_f64(cudaStream_t st, int M, int N, int K, const float* A, int lda, const float* B, int ldb, int tb,
                double* out, int ldc, int batch, long long sA, long long sB, long long sC) {
  GemmArgs g{};
  g.M = M, g.N = N, g.K = K;
  g.A = A, g.B = B, g.lda = lda, g.ldb = ldb, g.ldc = ldc, g.out64 = out;
  g.sA = sA, g.sB = sB, g.sC = sC;
  return tb ? gemm_launch<false, true, EPI_F64>(st, g, batch) : gemm_launch<false, false, EPI_F64>(st, g, batch);
}

// Rows per split of the weight gradient of layer l < L - 1 over a batch of n rows (a multiple of the K tile):
// enough splits that the tiles fill every SM twice.
int split_rows(fhmg_wsnet net, int n, int l) {
  const int wi = net->width[l], wo = net->width[l + 1];
  const long long tiles = (long long)((wi + kGB - 1) / kGB) * ((wo + kGB - 1) / kGB);
  const long long want = (2LL * fhmg::device_sms() + tiles - 1) / tiles;
  const int kper = (int)((n + want - 1) / want);
  return (kper + kGK - 1) / kGK * kGK;
}

// Room for the partial sums of every layer, before the backward pass begins (a pass that grew it layer by layer
// held all the smaller ones as well, and stood still at each allocation)
int ensure_part(fhmg_wsnet net, int n) {
  const int L = (int)net->width.size() - 1;
  size_t need = (size_t)((n + kOutRows - 1) / kOutRows) * (net->width[L - 1] + 1);
  for (int l = 0; l < L - 1; ++l) {
    const int kper = split_rows(net, n, l);
    need = std::max(need, (size_t)((n + kper - 1) / kper) * net->width[l + 1] * (net->width[l] + 1));
  }
  if (need <= net->part_n) return FHMG_OK;
  cudaFree(net->part);  // waits for the device
  net->part = nullptr, net->part_n = 0;
  const cudaError_t e = cudaMalloc((void**)&net->part, need * sizeof(float));
  if (e != cudaSuccess) {
    cudaGetLastError();
    net->part = nullptr;
    return fhmg_internal_fail(FHMG_ENOMEM, cudaGetErrorString(e));
  }
  net->part_n = need;
  return FHMG_OK;
}

// FP32 forward of n rows X (n x kFeat) -> output A[L] (n x 1); activations kept.
int forward32(fhmg_wsnet net, cudaStream_t st, const float* X, int n) {
  const int L = (int)net->width.size() - 1;
  int s = ensure_cap(net, n);
  if (s) return s;
  const float* in = X;
  for (int l = 0; l < L - 1; ++l) {
    GemmArgs g{};  // Z = in W^T + b (in: n x wi, W: wo x wi), A = SiLU(Z)
    g.M = n, g.N = net->width[l + 1], g.K = net->width[l];
    g.A = in, g.lda = g.K, g.B = net->P + net->woff[l], g.ldb = g.K;
    g.C = net->Z[l], g.ldc = g.N, g.bias = net->P + net->boff[l], g.out2 = net->A[l + 1], g.act = 1;
    if ((s = gemm_launch<false, true, EPI_ACT>(st, g, 1))) return s;
    in = net->A[l + 1];
  }
  out_layer_fwd<<<(n + 7) / 8, 256, 0, st>>>(n, net->width[L - 1], in, net->P + net->woff[L - 1],
                                             net->P + net->boff[L - 1], net->Z[L - 1], net->A[L]);
  ++g_nn_launches;
  NCK(cudaGetLastError());
  return FHMG_OK;
}

// Backward of the MSE loss against targets Y; gradients into net->G (overwritten).  The gradient of
// layer l (its weights, then its bias, consecutive in G) is summed over splits of the rows into
// partial sums, then over the splits.
int backward32(fhmg_wsnet net, cudaStream_t st, const float* X, const float* Y, int n) {
  const int L = (int)net->width.size() - 1;
  int s = ensure_part(net, n);
  if (s) return s;
  NCK(cudaMemsetAsync(net->loss, 0, sizeof(float), st));
  mse_fwd_bwd<<<nblk(n), 256, 0, st>>>(n, net->A[L], Y, net->dA[L], net->loss);
  ++g_nn_launches;
  NCK(cudaGetLastError());
  auto reduce = [&](int splits, long long m, int l) -> int {
    reduce_splits_kernel<<<(unsigned)((m + 255) / 256), 256, 0, st>>>(splits, m, net->part, net->G + net->woff[l]);
    ++g_nn_launches;
    NCK(cudaGetLastError());
    return FHMG_OK;
  };
  {
    const int l = L - 1, w = net->width[l], nr = (n + kOutRows - 1) / kOutRows;
    out_layer_bwd<<<dim3(w / 128 + 1, nr), 128, 0, st>>>(n, w, l > 0, net->dA[L], net->P + net->woff[l],
                                                         l > 0 ? net->A[l] : X, l > 0 ? net->Z[l - 1] : nullptr,
                                                         net->dA[l], net->part);
    ++g_nn_launches;
    NCK(cudaGetLastError());
    if ((s = reduce(nr, w + 1, l))) return s;
  }
  for (int l = L - 2; l >= 0; --l) {
    const int wi = net->width[l], wo = net->width[l + 1];
    const float* dz = net->dA[l + 1];  // gradient of the layer's pre-activation, n x wo
    const long long m = (long long)wo * wi + wo;
    const int kper = split_rows(net, n, l);
    const int splits = (n + kper - 1) / kper;
    GemmArgs g{};  // dW = dz^T in (wo x wi), db = column sums of dz
    g.M = wo, g.N = wi, g.K = n, g.kper = kper;
    g.A = dz, g.lda = wo, g.B = l == 0 ? X : net->A[l], g.ldb = wi;
    g.C = net->part, g.ldc = wi, g.sC = m, g.out2 = net->part + (long long)wo * wi;
    if ((s = gemm_launch<true, false, EPI_SPLIT>(st, g, splits))) return s;
    if ((s = reduce(splits, m, l))) return s;
    if (l > 0) {
      GemmArgs h{};  // gradient of the pre-activation below: (dz W) * SiLU'(Z)
      h.M = n, h.N = wi, h.K = wo;
      h.A = dz, h.lda = wo, h.B = net->P + net->woff[l], h.ldb = wi;
      h.C = net->dA[l], h.ldc = wi, h.bias = net->Z[l - 1];
      if ((s = gemm_launch<false, false, EPI_ACTB>(st, h, 1))) return s;
    }
  }
  return FHMG_OK;
}

// Y = network(X); err: the word that the one-launch network sets if a wait gives up
int forward_rows(fhmg_wsnet net, const float* X, int n, int bf16, float* Y, cudaStream_t st, int* err);

}  // namespace

extern "C" {

int fhmg_wsnet_create(int hidden, int layers, unsigned long long seed, fhmg_wsnet* out) {
  if (!out || hidden < 8 || hidden > 4096 || layers < 1 || layers > 8)
    return fhmg_internal_fail(FHMG_EINVAL, "wsnet: hidden in [8, 4096], layers in [1, 8]");
  fhmg_wsnet net = new (std::nothrow) fhmg_wsnet_s;
  if (!net) return fhmg_internal_fail(FHMG_ENOMEM, "host allocation failed");
  net->hidden = hidden;
  net->layers = layers;
  net->width.push_back(kFeat);
  for (int l = 0; l < layers; ++l) net->width.push_back(hidden);
  net->width.push_back(1);
  const int L = (int)net->width.size() - 1;
  std::vector<float> host;
  std::mt19937_64 rng(seed);
  for (int l = 0; l < L; ++l) {
    const int wi = net->width[l], wo = net->width[l + 1];
    net->woff.push_back((long long)host.size());
    std::normal_distribution<float> nd(0.f, std::sqrt(2.f / wi));
    for (long long i = 0; i < (long long)wi * wo; ++i) host.push_back(nd(rng) * (l == L - 1 ? 0.1f : 1.f));
    net->boff.push_back((long long)host.size());
    for (int i = 0; i < wo; ++i) host.push_back(0.f);
  }
  net->nparams = (long long)host.size();
  int s = FHMG_OK;
  auto bail = [&](int st) {
    fhmg_wsnet_destroy(net);
    return st;
  };
  if ((s = nalloc(net->allocs, &net->P, host.size())) || (s = nalloc(net->allocs, &net->G, host.size())) ||
      (s = nalloc(net->allocs, &net->Mo, host.size())) || (s = nalloc(net->allocs, &net->Vo, host.size())) ||
      (s = nalloc(net->allocs, &net->Pbf, host.size())) || (s = nalloc(net->allocs, &net->loss, 1)) || (s = nalloc(net->allocs, &net->err, 2)) ||
      (hidden % 64 == 0 && hidden <= kMlpMaxH && (s = nalloc(net->allocs, &net->Wpk, mlp_packed(hidden, layers)))))
    return bail(s);
  if (cudaMemcpy(net->P, host.data(), host.size() * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemset(net->err, 0, 2 * sizeof(int)) != cudaSuccess ||
      cudaMemset(net->Mo, 0, host.size() * 4) != cudaSuccess || cudaMemset(net->Vo, 0, host.size() * 4) != cudaSuccess)
    return bail(fhmg_internal_fail(FHMG_ECUDA, "wsnet upload failed"));
  *out = net;
  return FHMG_OK;
}

int fhmg_wsnet_destroy(fhmg_wsnet net) {
  if (!net) return FHMG_OK;
  for (void* a : net->allocs) cudaFree(a);
  for (void* a : net->act) cudaFree(a);
  cudaFree(net->part);
  for (auto& w : net->ws) cudaFree(w.first);
  delete net;
  return FHMG_OK;
}

int fhmg_wsnet_num_params(fhmg_wsnet net, long long* n) {
  if (!net || !n) return fhmg_internal_fail(FHMG_EINVAL, "null argument");
  *n = net->nparams;
  return FHMG_OK;
}

int fhmg_wsnet_get_params(fhmg_wsnet net, float* host) {
  if (!net || !host) return fhmg_internal_fail(FHMG_EINVAL, "null argument");
  NCK(cudaMemcpy(host, net->P, net->nparams * 4, cudaMemcpyDeviceToHost));
  return FHMG_OK;
}

int fhmg_wsnet_set_params(fhmg_wsnet net, const float* host) {
  if (!net || !host) return fhmg_internal_fail(FHMG_EINVAL, "null argument");
  NCK(cudaMemcpy(net->P, host, net->nparams * 4, cudaMemcpyHostToDevice));
  return FHMG_OK;
}

int fhmg_wsnet_forward(fhmg_wsnet net, const float* X, int n, int bf16, float* Y, void* stream) {
  if (!net || !X || !Y || n < 1) return fhmg_internal_fail(FHMG_EINVAL, "bad arguments");
  return forward_rows(net, X, n, bf16, Y, (cudaStream_t)stream, net->err + 1);
}

int fhmg_wsnet_status(fhmg_wsnet net, void* stream) {
  if (!net) return fhmg_internal_fail(FHMG_EINVAL, "null argument");
  cudaStream_t st = (cudaStream_t)stream;
  int err = 0;
  NCK(cudaMemcpyAsync(&err, net->err + 1, sizeof err, cudaMemcpyDeviceToHost, st));
  NCK(cudaStreamSynchronize(st));
  if (!err) return FHMG_OK;
  NCK(cudaMemsetAsync(net->err + 1, 0, sizeof err, st));
  return fhmg_internal_fail(FHMG_ETIMEOUT, "the network kernel gave up waiting on a shared-memory stage");
}

int fhmg_wsnet_inject_timeout(fhmg_wsnet net, long long consumer_spin) {
  if (!net) return fhmg_internal_fail(FHMG_EINVAL, "null argument");
  if (consumer_spin < 1 || consumer_spin > fhmg::kSpinLimit)
    return fhmg_internal_fail(FHMG_EINVAL, "consumer spin limit must be in 1..2^24");
  if (!net->Wpk || net->layers < 2) return fhmg_internal_fail(FHMG_EINVAL, "the network streams no weight tiles");
  net->inj_spin = consumer_spin;
  return FHMG_OK;
}

int fhmg_wsnet_loss_grad(fhmg_wsnet net, const float* X, const float* Y, int n, float* loss_host, float* grad_host,
                         void* stream) {
  if (!net || !X || !Y || n < 1) return fhmg_internal_fail(FHMG_EINVAL, "bad arguments");
  cudaStream_t st = (cudaStream_t)stream;
  int s = forward32(net, st, X, n);
  if (s || (s = backward32(net, st, X, Y, n))) return s;
  if (loss_host) NCK(cudaMemcpyAsync(loss_host, net->loss, 4, cudaMemcpyDeviceToHost, st));
  if (grad_host) NCK(cudaMemcpyAsync(grad_host, net->G, net->nparams * 4, cudaMemcpyDeviceToHost, st));
  NCK(cudaStreamSynchronize(st));
  return FHMG_OK;
}

}  // extern "C"

namespace {

int forward_rows(fhmg_wsnet net, const float* X, int n, int bf16, float* Y, cudaStream_t st, int* err) {
  const int L = (int)net->width.size() - 1;
  int s;
  if (bf16 && net->Wpk && reinterpret_cast<uintptr_t>(X) % 8 == 0) {
    pack_weights<<<nblk(32LL * net->hidden + (long long)(net->layers - 1) * net->hidden * net->hidden), 256, 0, st>>>(
        net->hidden, net->layers, net->P, net->Wpk);
    ++g_nn_launches;
    NCK(cudaGetLastError());
    MlpArgs a{};
    a.n = n, a.layers = net->layers, a.X = X, a.W = net->Wpk, a.P = net->P, a.Y = Y, a.err = err;
    a.spin = fhmg::kSpinLimit;
    if (net->inj_spin > 0) {
      a.spin = net->inj_spin;
      a.withhold = (net->layers - 1) * (net->hidden / 64) > 1 ? 2 : 1;  // within the first block of rows
      net->inj_spin = 0;
    }
    for (int l = 0; l < L; ++l) a.boff[l] = net->boff[l];
    static fhmg::KernelCache cache;
    const size_t smem = mlp_smem(net->hidden, net->layers).total + 1024;
    int occ = 1;
    NCK(fhmg::prepare_launch(mlp_bf16, kMlpBlock, smem, cache, &occ));
    mlp_bf16<<<std::min((n + kMlpRows - 1) / kMlpRows, fhmg::device_sms()), kMlpBlock, smem, st>>>(net->hidden, a);
    ++g_nn_launches;
    NCK(cudaGetLastError());
    return FHMG_OK;
  }
  if ((s = ensure_cap(net, n))) return s;
  if (!bf16) {
    if ((s = forward32(net, st, X, n))) return s;
    NCK(cudaMemcpyAsync(Y, net->A[L], sizeof(float) * n, cudaMemcpyDeviceToDevice, st));
    return FHMG_OK;
  }
  // BF16 tensor-core inference (FP32 accumulation): weights and activations rounded to BF16
  to_bf16<<<nblk(net->nparams), 256, 0, st>>>(net->nparams, net->P, net->Pbf);
  ++g_nn_launches;
  to_bf16<<<nblk((long long)n * kFeat), 256, 0, st>>>((long long)n * kFeat, X, net->Abf[0]);
  ++g_nn_launches;
  NCK(cudaGetLastError());
  int cur = 0;
  for (int l = 0; l < L; ++l) {
    const int wi = net->width[l], wo = net->width[l + 1];
    const bool last = l == L - 1;
    const __nv_bfloat16* Wl = net->Pbf + net->woff[l];
    if (!last && wi % 32 == 0 && wo % 64 == 0 && reinterpret_cast<uintptr_t>(Wl) % 16 == 0 &&
        reinterpret_cast<uintptr_t>(net->Abf[cur]) % 16 == 0) {
      // hidden layers of the full width: one tiled launch, bias and SiLU fused (Z is not needed:
      // the backward pass runs on the FP32 forward's activations)
      dim3 grid(wo / 64, (n + 127) / 128);
      gemm_bf16_silu<<<grid, 256, 0, st>>>(n, wo, wi, net->Abf[cur], Wl, net->P + net->boff[l], net->Abf[1 - cur]);
      ++g_nn_launches;
      NCK(cudaGetLastError());
      cur = 1 - cur;
      continue;
    }
    dim3 grid((wo + 7) / 8, (n + 63) / 64);
    gemm_bf16_nt<<<grid, 128, 0, st>>>(n, wo, wi, net->Abf[cur], net->Pbf + net->woff[l], net->Z[l]);
    ++g_nn_launches;
    NCK(cudaGetLastError());
    bias_act_fwd<<<nblk((long long)n * wo), 256, 0, st>>>(n, wo, net->Z[l], net->P + net->boff[l],
                                                        last ? Y : nullptr, last ? 0 : 1,
                                                        last ? nullptr : net->Abf[1 - cur]);
    ++g_nn_launches;
    NCK(cudaGetLastError());
    cur = 1 - cur;
  }
  return FHMG_OK;
}

}  // namespace

// ---------------------------------------------------------------- spectral warm start

int fhmg_internal_problem_geom(fhmg_problem p, int* dim, int* N, int* M, double* Lx, void** stream,
                               const double** t_host);

namespace {

// S[n][p] = sin((p+1) pi (n+1) / (N+1)), n < N, p < K  (the discrete sine modes of A_h)
__global__ void sine_basis(int N, int K, float* S) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)N * K;
       i += (long long)gridDim.x * blockDim.x) {
    const int n = (int)(i / K), p = (int)(i % K);
    S[i] = (float)sin((double)(p + 1) * (n + 1) * M_PI / (N + 1));
  }
}

__global__ void d2f(long long n, const double* x, float* y) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    y[i] = (float)x[i];
}
// eigenvalue of mode k (2D: k = p K + q) of the 3-/5-point negative Laplacian
__device__ __forceinline__ double mode_lambda(int dim, int N, double Lx, int K, int k) {
  const double h = Lx / (N + 1);
  const int p = dim == 1 ? k : k / K, q = dim == 1 ? -1 : k % K;
  auto e = [&](int j) {
    const double s = sin((j + 1) * M_PI / (2.0 * (N + 1)));
    return 4.0 / (h * h) * s * s;
  };
  return e(p) + (dim == 2 ? e(q) : 0.0);
}

__global__ void mode_lambdas(int dim, int N, double Lx, int K, int nm, double* lam) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < nm) lam[k] = mode_lambda(dim, N, Lx, K, k);
}

// G[m][k] = c_k * y[k][m] / lam_k  (predicted mode amplitudes per time level)
__global__ void mode_amplitudes(int nm, int M, const float* c, const float* y, const double* lam, float* G) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)nm * M;
       i += (long long)gridDim.x * blockDim.x) {
    const int k = (int)(i / M), m = (int)(i % M);
    G[(long long)m * nm + k] = (float)((double)c[k] * y[i] / lam[k]);
  }
}

// training pairs: y = lam * uhat[m][k] / c[k] for modes with |c_k| >= thr (row order k-major)
__global__ void mode_targets(int nm, int M, const float* c, const float* uhat, const double* lam, float thr,
                             const int* keep, const int* kpos, float* Y) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)nm * M;
       i += (long long)gridDim.x * blockDim.x) {
    const int k = (int)(i / M), m = (int)(i % M);
    if (!keep[k]) continue;
    Y[(long long)kpos[k] * M + m] = (float)(lam[k] * (double)uhat[(long long)m * nm + k] / (double)c[k]);
  }
}

__global__ void build_features_kept(int nm, const double* lam, const float* loglam, int M, const double* ta,
                                    const float* logt, double alpha, const int* keep, const int* kpos, float* X) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)nm * M;
       i += (long long)gridDim.x * blockDim.x) {
    const int k = (int)(i / M), m = (int)(i % M);
    if (!keep || keep[k]) {
      const long long row = (long long)(keep ? kpos[k] : k) * M + m;
      ws_features(lam[k], loglam[k], alpha, ta[m], logt[m], X + row * kFeat);
    }
  }
}

// FP64 projection used for training targets (small sizes; accuracy over speed):
// T[l][p][x] = sum_y S[y][p] u[l][y][x];  out[l][p][q] = sc^2 sum_x T[l][p][x] S[x][q]  (2D)
// out[l][p] = sc sum_x u[l][x] S[x][p]  (1D)
__global__ void sine_basis64(int N, int K, double* S) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)N * K;
       i += (long long)gridDim.x * blockDim.x) {
    const int n = (int)(i / K), p = (int)(i % K);
    S[i] = sin((double)(p + 1) * (n + 1) * M_PI / (N + 1));
  }
}

__global__ void project64_a(int dim, int N, int K, int nl, const double* u, const double* S, double* T) {
  const long long total = dim == 1 ? (long long)nl * K : (long long)nl * K * N;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    if (dim == 1) {
      const int l = (int)(i / K), p = (int)(i % K);
      double s = 0.0;
      for (int x = 0; x < N; ++x) s += u[(long long)l * N + x] * S[(long long)x * K + p];
      T[i] = s;
    } else {
      const int l = (int)(i / ((long long)K * N)), r = (int)(i % ((long long)K * N)), p = r / N, x = r % N;
      double s = 0.0;
      for (int y = 0; y < N; ++y) s += S[(long long)y * K + p] * u[((long long)l * N + y) * N + x];
      T[i] = s;
    }
  }
}
__global__ void project64_b(int dim, int N, int K, int nl, const double* T, const double* S, double sc, float* out) {
  const long long total = dim == 1 ? (long long)nl * K : (long long)nl * K * K;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    if (dim == 1) {
      out[i] = (float)(sc * T[i]);
    } else {
      const int l = (int)(i / ((long long)K * K)), r = (int)(i % ((long long)K * K)), p = r / K, q = r % K;
      double s = 0.0;
      for (int x = 0; x < N; ++x) s += T[((long long)l * K + p) * N + x] * S[(long long)x * K + q];
      out[i] = (float)(sc * sc * s);
    }
  }
}

struct Spectral {
  int dim, N, M, K, nm;
  double Lx;
  cudaStream_t st;
  const double* thost;
  std::vector<void*> mem;  // buffers of its own (no net)
  fhmg_wsnet net = nullptr;  // or the net whose scratch it uses, and the buffers taken so far
  size_t taken = 0;
  bool running = false;      // kernels issued on st may still use the net's scratch
  float* S = nullptr;   // N x K
  double* lam = nullptr;
  double* tdev = nullptr;
  ~Spectral() {
    for (void* p : mem) cudaFree(p);
    if (net && running) {  // a prediction that stops early: its kernels end before the next one takes the scratch
      cudaMemsetAsync(net->err, 0, sizeof(int), st);
      cudaStreamSynchronize(st);
    }
  }
  template <typename T>
  int alloc(T** p, size_t n) {
    const size_t bytes = (n ? n : 1) * sizeof(T);
    if (net && taken < net->ws.size() && net->ws[taken].second >= bytes) {
      *p = (T*)net->ws[taken++].first;
      return FHMG_OK;
    }
    auto give_back = [&](size_t i) {  // (frees wait for the device)
      cudaFree(net->ws[i].first);
      net->ws[i] = {nullptr, 0};
    };
    if (net) {  // the smaller buffer goes first, so that the two are never held at once
      if (taken == net->ws.size()) net->ws.push_back({nullptr, 0});
      give_back(taken);
    }
    cudaError_t e = cudaMalloc((void**)p, bytes);
    if (e != cudaSuccess && net) {  // nor do buffers of an earlier prediction stand in this one's way
      cudaGetLastError();
      for (size_t i = taken + 1; i < net->ws.size(); ++i) give_back(i);
      e = cudaMalloc((void**)p, bytes);
    }
    if (e != cudaSuccess) {
      cudaGetLastError();  // not sticky; keep it out of the next launch check
      return fhmg_internal_fail(FHMG_ENOMEM, cudaGetErrorString(e));
    }
    if (net)
      net->ws[taken++] = {*p, bytes};
    else
      mem.push_back(*p);
    return FHMG_OK;
  }
  int init(fhmg_problem p, int K_) {
    void* sv;
    int s = fhmg_internal_problem_geom(p, &dim, &N, &M, &Lx, &sv, &thost);
    if (s) return s;
    st = (cudaStream_t)sv;
    K = K_ < N ? K_ : N;
    nm = dim == 1 ? K : K * K;
    if ((s = alloc(&S, (size_t)N * K)) || (s = alloc(&lam, nm)) || (s = alloc(&tdev, M + 1))) return s;
    running = true;
    sine_basis<<<nblk((long long)N * K), 256, 0, st>>>(N, K, S);
    ++g_nn_launches;
    mode_lambdas<<<(nm + 127) / 128, 128, 0, st>>>(dim, N, Lx, K, nm, lam);
    ++g_nn_launches;
    NCK(cudaGetLastError());
    NCK(cudaMemcpyAsync(tdev, thost, sizeof(double) * (M + 1), cudaMemcpyHostToDevice, st));
    return FHMG_OK;
  }
  // features of the kept modes (all: keep NULL) at every time level, row order k-major
  int features(double alpha, const int* keep, const int* kpos, float* X) {
    float *loglam, *logt;
    double* ta;
    int s;
    if ((s = alloc(&loglam, nm)) || (s = alloc(&logt, M)) || (s = alloc(&ta, M))) return s;
    feature_tables<<<(std::max(nm, M) + 127) / 128, 128, 0, st>>>(nm, lam, M, tdev, alpha, loglam, ta, logt);
    ++g_nn_launches;
    build_features_kept<<<nblk((long long)nm * M), 256, 0, st>>>(nm, lam, loglam, M, ta, logt, alpha, keep, kpos, X);
    ++g_nn_launches;
    NCK(cudaGetLastError());
    return FHMG_OK;
  }
  // FP64 coefficients (training targets): x is FP64, nl x N^dim; out FP32 nl x K^dim
  int project64(const double* x, int nl, float* out) {
    double *S64, *T;
    int s = alloc(&S64, (size_t)N * K);
    if (s || (s = alloc(&T, dim == 1 ? (size_t)nl * K : (size_t)nl * K * N))) return s;
    sine_basis64<<<nblk((long long)N * K), 256, 0, st>>>(N, K, S64);
    ++g_nn_launches;
    const long long na = dim == 1 ? (long long)nl * K : (long long)nl * K * N;
    project64_a<<<nblk(na), 256, 0, st>>>(dim, N, K, nl, x, S64, T);
    ++g_nn_launches;
    const long long nb_ = dim == 1 ? (long long)nl * K : (long long)nl * K * K;
    project64_b<<<nblk(nb_), 256, 0, st>>>(dim, N, K, nl, T, S64, 2.0 / (N + 1), out);
    ++g_nn_launches;
    NCK(cudaGetLastError());
    return FHMG_OK;
  }
  // coefficients of nl grid functions (time levels) of x (FP32, nl x N^dim) on the modes:
  // out[l][k], scaled by (2/(N+1))^dim so that x = sum_k out_k s_k exactly for a sine series
  int project(const float* x, int nl, float* out) {
    const float sc = 2.f / (N + 1);
    if (dim == 1) return gemm(st, nl, K, N, sc, x, N, 0, S, K, 0, out, K);
    float* T1;
    int s = alloc(&T1, (size_t)nl * K * N);
    if (s) return s;
    // T1[l] = S^T (K x N) x[l] (N x N)  -> K x N
    if ((s = gemm(st, K, N, N, sc, S, K, 1, x, N, 0, T1, N, nl, 0, (long long)N * N, (long long)K * N))) return s;
    // out[l] = T1[l] (K x N) S (N x K) -> K x K
    return gemm(st, K, K, N, sc, T1, N, 0, S, K, 0, out, K, nl, (long long)K * N, 0, (long long)K * K);
  }
};

}  // namespace

extern "C" {

int fhmg_wsnet_launches(long long* n) {
  if (!n) return fhmg_internal_fail(FHMG_EINVAL, "n is NULL");
  *n = g_nn_launches.load();
  return FHMG_OK;
}

int fhmg_ws_predict(fhmg_wsnet net, fhmg_problem prob, const double* f, double alpha, int K, int bf16, double* u0) {
  if (!net || !prob || !f || !u0 || K < 1) return fhmg_internal_fail(FHMG_EINVAL, "bad arguments");
  Spectral sp;
  sp.net = net;
  int s = sp.init(prob, K);
  if (s) return s;
  const int N = sp.N, M = sp.M, nm = sp.nm, dim = sp.dim;
  const long long npts = dim == 1 ? N : (long long)N * N;
  // coefficients of the source (constant in time: its last time level)
  float *f32, *c, *X, *Y, *G, *T1;
  if ((s = sp.alloc(&f32, npts)) || (s = sp.alloc(&c, nm)) || (s = sp.alloc(&X, (size_t)nm * M * kFeat)) ||
      (s = sp.alloc(&Y, (size_t)nm * M)) || (s = sp.alloc(&G, (size_t)nm * M)))
    return s;
  d2f<<<nblk(npts), 256, 0, sp.st>>>(npts, f + (long long)(M - 1) * npts, f32);
  ++g_nn_launches;
  NCK(cudaGetLastError());
  if ((s = sp.project(f32, 1, c))) return s;
  if ((s = sp.features(alpha, nullptr, nullptr, X))) return s;
  if ((s = forward_rows(net, X, nm * M, bf16, Y, sp.st, net->err))) return s;
  mode_amplitudes<<<nblk((long long)nm * M), 256, 0, sp.st>>>(nm, M, c, Y, sp.lam, G);
  ++g_nn_launches;
  NCK(cudaGetLastError());
  // synthesis u0[m] = sum_k G[m][k] s_k, in FP32, written as FP64
  if (dim == 1) {
    // u0 (M x N) = G (M x K) S^T (K x N)
    if ((s = gemm_to_f64(sp.st, M, N, sp.K, G, sp.K, sp.S, sp.K, 1, u0, N, 1, 0, 0, 0))) return s;
  } else {
    const int K2 = sp.K;
    if ((s = sp.alloc(&T1, (size_t)M * K2 * N))) return s;
    // T1[m] = G[m] (K x K) S^T (K x N);  u0[m] = S (N x K) T1[m] (K x N)
    if ((s = gemm(sp.st, K2, N, K2, 1.f, G, K2, 0, sp.S, K2, 1, T1, N, M, (long long)K2 * K2, 0, (long long)K2 * N)))
      return s;
    if ((s = gemm_to_f64(sp.st, N, N, K2, sp.S, K2, T1, N, 0, u0, N, M, 0, (long long)K2 * N, (long long)N * N)))
      return s;
  }
  int err = 0;
  NCK(cudaMemcpyAsync(&err, net->err, sizeof err, cudaMemcpyDeviceToHost, sp.st));
  NCK(cudaStreamSynchronize(sp.st));
  if (err) return fhmg_internal_fail(FHMG_ETIMEOUT, "the network kernel gave up waiting on a shared-memory stage");
  sp.running = false;
  return FHMG_OK;
}

int fhmg_ws_dataset(fhmg_problem prob, const double* u, const double* f, double alpha, int K, float rel_thr,
                    float* X_out, float* Y_out, long long* nrows) {
  if (!prob || !u || !f || !X_out || !Y_out || !nrows || K < 1) return fhmg_internal_fail(FHMG_EINVAL, "bad arguments");
  Spectral sp;
  int s = sp.init(prob, K);
  if (s) return s;
  const int N = sp.N, M = sp.M, nm = sp.nm, dim = sp.dim;
  const long long npts = dim == 1 ? N : (long long)N * N;
  float *c, *uh;
  if ((s = sp.alloc(&c, nm)) || (s = sp.alloc(&uh, (size_t)M * nm))) return s;
  if ((s = sp.project64(f + (long long)(M - 1) * npts, 1, c)) || (s = sp.project64(u, M, uh))) return s;
  // modes kept: |c_k| >= rel_thr * max |c|
  std::vector<float> ch(nm);
  NCK(cudaMemcpyAsync(ch.data(), c, sizeof(float) * nm, cudaMemcpyDeviceToHost, sp.st));
  NCK(cudaStreamSynchronize(sp.st));
  float cmax = 0.f;
  for (float v : ch) cmax = std::fabs(v) > cmax ? std::fabs(v) : cmax;
  std::vector<int> keep(nm), kpos(nm);
  int nk = 0;
  for (int k = 0; k < nm; ++k) {
    keep[k] = std::fabs(ch[k]) >= rel_thr * cmax && cmax > 0.f;
    kpos[k] = nk;
    nk += keep[k];
  }
  int *dkeep, *dkpos;
  if ((s = sp.alloc(&dkeep, nm)) || (s = sp.alloc(&dkpos, nm))) return s;
  NCK(cudaMemcpyAsync(dkeep, keep.data(), sizeof(int) * nm, cudaMemcpyHostToDevice, sp.st));
  NCK(cudaMemcpyAsync(dkpos, kpos.data(), sizeof(int) * nm, cudaMemcpyHostToDevice, sp.st));
  if ((s = sp.features(alpha, dkeep, dkpos, X_out))) return s;
  mode_targets<<<nblk((long long)nm * M), 256, 0, sp.st>>>(nm, M, c, uh, sp.lam, rel_thr, dkeep, dkpos, Y_out);
  ++g_nn_launches;
  NCK(cudaGetLastError());
  NCK(cudaStreamSynchronize(sp.st));
  *nrows = (long long)nk * M;
  return FHMG_OK;
}

int fhmg_wsnet_train(fhmg_wsnet net, const float* X, const float* Y, long long nsamples, int batch, int steps,
                     float lr, unsigned long long seed, float* last_loss, void* stream) {
  if (!net || !X || !Y || nsamples < batch || batch < 1 || steps < 0)
    return fhmg_internal_fail(FHMG_EINVAL, "bad arguments");
  cudaStream_t st = (cudaStream_t)stream;
  std::mt19937_64 rng(seed);
  std::uniform_int_distribution<long long> pick(0, nsamples - batch);
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  for (int it = 0; it < steps; ++it) {
    // contiguous mini-batches at random offsets (the samples are stored shuffled)
    const long long o = pick(rng);
    const float* xb = X + o * kFeat;
    const float* yb = Y + o;
    int s = forward32(net, st, xb, batch);
    if (s || (s = backward32(net, st, xb, yb, batch))) return s;
    ++net->step;
    const float c1 = 1.f - std::pow(b1, (float)net->step), c2 = 1.f - std::pow(b2, (float)net->step);
    adam_step<<<nblk(net->nparams), 256, 0, st>>>(net->nparams, net->P, net->G, net->Mo, net->Vo, lr, b1, b2, c1, c2,
                                                 eps);
    ++g_nn_launches;
    NCK(cudaGetLastError());
  }
  if (last_loss) {
    NCK(cudaMemcpyAsync(last_loss, net->loss, 4, cudaMemcpyDeviceToHost, st));
    NCK(cudaStreamSynchronize(st));
  }
  return FHMG_OK;
}

}  // extern "C"
