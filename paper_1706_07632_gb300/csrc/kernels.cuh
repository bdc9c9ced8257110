// CUDA kernels (sm_103a) for multigrid waveform relaxation with an H-matrix time operator.
//
// Grid functions are time-major with space contiguous: value (m, p) at m * ld + p, m = 0..M-1
// standing for t_1..t_M, p the spatial index (1D: p = n - 1; 2D: p = iy * N + ix).
//
// The H-matrix walk over leaf rows (the hot path) is in panel.cuh; this file holds the
// geometry helpers and the stencil / transfer kernels around it.
#pragma once
#include <cstdint>
#include <algorithm>
#include <cuda_runtime.h>

namespace fhmg {

// Geometry of the columns a smoothing half-sweep updates.
struct Geo {
  int dim;       // 0: compact columns, no stencil; 1 or 2: colour of a grid
  int N;         // interior points per dimension (dim > 0)
  int colour;    // 0 or 1 (dim > 0)
  long long ld;  // elements per time level of the arrays addressed
  double inv_h2; // 1/h^2 (dim > 0)
  int split;     // 2D: 1 if the grid functions are stored by colour (split_pos)
};

// Number of points of a colour (dim 1: colour 0 = odd n (1-based), colour 1 = even n;
// dim 2: colour 0 = ix + iy even (0-based, same parity as 1-based i + j), colour 1 = odd).
__host__ __device__ inline long long colour_count(int dim, int N, int colour) {
  if (dim == 0) return N;
  if (dim == 1) return colour == 0 ? (N + 1) / 2 : N / 2;
  long long first = colour == 0 ? (N + 1) / 2 : N / 2;  // points in an even row
  return (long long)((N - 1) / 2) * N + first;
}

// Spatial index of the c-th point of a colour.
__host__ __device__ inline long long colour_pos(int dim, int N, int colour, long long c, int* iy_out,
                                                int* ix_out) {
  if (dim == 1) {
    long long p = 2 * c + colour;
    *iy_out = 0;
    *ix_out = (int)p;
    return p;
  }
  long long first = colour == 0 ? (N + 1) / 2 : N / 2;
  long long q = c / N, rem = c % N;
  int iy, ix;
  if (rem < first) {
    iy = (int)(2 * q);
    ix = (int)(colour + 2 * rem);
  } else {
    iy = (int)(2 * q + 1);
    ix = (int)((1 - colour) + 2 * (rem - first));
  }
  *iy_out = iy;
  *ix_out = ix;
  return (long long)iy * N + ix;
}

// Storage by colour of the 2D FP32 grid functions (inner cycles): per time level the points of colour
// 0, then those of colour 1, each in the order of colour_pos -- within a row the points of a colour
// are neighbours, so a half-sweep reads and writes whole sectors, where rows of both colours would
// have it move the other colour's half too.  split_row: the place of the first point of a colour in
// row iy; a point (iy, ix) of the colour sits ix / 2 behind it.
__host__ __device__ inline long long split_row(int N, int colour, int iy) {
  const long long first = colour == 0 ? (N + 1) / 2 : N / 2;
  return (colour ? colour_count(2, N, 0) : 0) + (long long)(iy >> 1) * N + ((iy & 1) ? first : 0);
}
__host__ __device__ inline long long split_pos(int N, int iy, int ix) {
  return split_row(N, (iy + ix) & 1, iy) + (ix >> 1);
}

// Places (relative to the point's own) of the neighbours of a point of a colour, which depend on the
// parity of its row only: left, up and down; right = left + step.
struct NbrOffsets {
  int left[2], up[2], down[2];  // |offset| <= N^2 / 2 + N
  int step;
};
__host__ __device__ inline NbrOffsets nbr_offsets(const Geo& g) {
  NbrOffsets o;
#pragma unroll
  for (int par = 0; par < 2; ++par) {
    if (g.dim == 2 && g.split) {
      const int s = (par + g.colour) & 1;  // ix = 2 j + s
      const int f = g.colour == 0 ? (g.N + 1) / 2 : g.N / 2, fo = g.N - f;
      const int d = (int)(g.colour == 0 ? colour_count(2, g.N, 0) : -colour_count(2, g.N, 0));
      o.left[par] = d + (par ? fo - f : 0) - 1 + s;
      o.up[par] = par ? d - f : d - g.N + fo;
      o.down[par] = par ? d + g.N - f : d + fo;
    } else {
      o.left[par] = -1;
      o.up[par] = -g.N;
      o.down[par] = g.N;
    }
  }
  o.step = g.dim == 2 && g.split ? 1 : 2;
  return o;
}

// ---------------------------------------------------------------- stencil / transfer kernels
//
// Launch shape of the grid-function kernels: blockIdx.x / threadIdx.x run along a grid row (x),
// blockIdx.y is the row (y; 0 in 1D), blockIdx.z strides over the time levels, so no index is
// recovered by a division.

// Transfers between a level (fine) and the one below it, for up to NJ instances in one launch (a
// batched cycle has an instance's grids at every depth: one launch for each took a third of the launches of
// a batch of 16 and, with the gaps between them, 14 of its 74 ms: 73.7 -> 66.2 ms).  Block b works on the instance whose
// range of blocks holds it.  Within an instance 2^lx threads run along a grid row (x) and 256 / 2^lx
// along the time levels, so that short rows fill their blocks too.
template <typename T>
struct TransferJob {
  const T* F;   // restriction: right-hand side
  T* U;         // fine grid function (restriction: read; prolongation: corrected)
  T* Xc;        // restriction: FW(u)
  T* Bc;        // restriction: FW(F - A_h u)
  T* E;         // prolongation: the correction; restriction: its start, set to zero (null: left alone)
  double inv_h2;
  long long first;  // first block
  int dim, Nf, M, lx, bx, by, bz;
};
template <typename T, int NJ>
struct TransferBatch {
  TransferJob<T> job[NJ];
  int n;
};
template <typename T>
constexpr bool kPlain2D = sizeof(T) == 8;  // 2D FP32 grid functions are stored by colour: kernels of their own below

// Launch shape for n instances (restriction: a thread per coarse point, else per fine point): returns the
// number of blocks, about 16 per SM over all of them, each with an equal share of the time levels' work.
// A block takes as many time levels side by side as short rows leave threads for, unless that leaves
// SMs without a block (the FP64 pipe, 2 lanes per clock and SM, is what the work must be spread over).
template <typename T>
inline long long transfer_shape(TransferJob<T>* jobs, int n, bool restriction, int sms) {
  long long units = 0;  // blocks of one step each
  auto rows = [&](const TransferJob<T>& j) { return restriction ? (j.Nf - 1) / 2 : j.Nf; };
  auto steps = [](const TransferJob<T>& j) { return (j.M + (256 >> j.lx) - 1) / (256 >> j.lx); };
  for (int k = 0; k < n; ++k) {
    TransferJob<T>& j = jobs[k];
    const int nx = rows(j);
    j.by = j.dim == 1 ? 1 : nx;
    for (j.lx = 0;; ++j.lx) {
      j.bx = (nx + (1 << j.lx) - 1) >> j.lx;
      if (j.lx == 8 || (j.bx == 1 && (long long)j.by * steps(j) * n >= 4LL * sms)) break;
    }
    units += (long long)j.bx * j.by * steps(j);
  }
  const long long per = std::max<long long>(1, (units + 16LL * sms - 1) / (16LL * sms));
  long long blocks = 0;
  for (int k = 0; k < n; ++k) {
    TransferJob<T>& j = jobs[k];
    j.first = blocks;
    j.bz = (int)((steps(j) + per - 1) / per);
    blocks += (long long)j.bx * j.by * j.bz;
  }
  return blocks;
}

struct TransferPlace {
  int x, y, m0, dm;  // point, first time level of this thread and the step to its next one
};
template <typename T, int NJ>
__device__ __forceinline__ const TransferJob<T>& transfer_place(const TransferBatch<T, NJ>& B, TransferPlace& q) {
  int k = 0;
  if (NJ > 1)
    while (k + 1 < B.n && B.job[k + 1].first <= (long long)blockIdx.x) ++k;
  const TransferJob<T>& J = B.job[k];
  const unsigned b = (unsigned)((long long)blockIdx.x - J.first);
  const unsigned row = b / (unsigned)J.bx;
  q.x = (int)((b - row * (unsigned)J.bx) << J.lx) + (int)(threadIdx.x & ((1u << J.lx) - 1));
  const unsigned z = row / (unsigned)J.by;
  q.y = (int)(row - z * (unsigned)J.by);
  const int tm = 256 >> J.lx;
  q.m0 = (int)z * tm + (int)(threadIdx.x >> J.lx);
  q.dm = J.bz * tm;
  return J;
}

// Restriction of the defect with the time operator commuted out:
//   Xc = FW(u)  and  Bc = FW(F - A_h u), so that the coarse right-hand side is Bc - R~ Xc
// (FW acts per time level and R~ per spatial point, so FW(R~ u) = R~ FW(u)).  One thread per
// coarse point (cx, cy) per time level.  In FP64 the FP64 pipe bounds it (15 operations
// per point in 1D: 4095 points x M = 4096 take 0.29 ms, of which the pipe needs 0.22), else memory.  A
// missing neighbour reads the next point instead and counts as zero, so that no load sits behind a branch.
template <typename T, int NJ>
__global__ void __launch_bounds__(256) restrict_pre_kernel(const __grid_constant__ TransferBatch<T, NJ> B) {
  TransferPlace q;
  const TransferJob<T>& J = transfer_place(B, q);
  const int Nf = J.Nf, M = J.M;
  const int Nc = (Nf - 1) / 2;
  const int cx = q.x, cy = q.y;
  if (cx >= Nc) return;
  const T* __restrict__ U = J.U;
  const T* __restrict__ F = J.F;
  T* __restrict__ Xc = J.Xc;
  T* __restrict__ Bc = J.Bc;
  T* __restrict__ E = J.E;
  const T ih2 = (T)J.inv_h2;
  if (!kPlain2D<T> || J.dim == 1) {
    const bool l = cx > 0, r = 2 * cx + 2 < Nf - 1;  // the outer neighbours exist
    for (int m = q.m0; m < M; m += q.dm) {
      const long long pc = (long long)m * Nf + 2 * cx + 1;
      T u[5], f[3];
#pragma unroll
      for (int o = 0; o < 3; ++o) {
        u[o + 1] = U[pc + o - 1];
        f[o] = F[pc + o - 1];
      }
      u[0] = U[pc - (l ? 2 : 1)];
      u[4] = U[pc + (r ? 2 : 1)];
      if (!l) u[0] = 0;
      if (!r) u[4] = 0;
      T xs = 0, bs = 0;
#pragma unroll
      for (int o = 0; o < 3; ++o) {
        const T w = o == 1 ? (T)0.5 : (T)0.25;
        const T uc = u[o + 1], ul = u[o], ur = u[o + 2];
        xs += w * uc;
        bs += w * (f[o] - (2 * uc - ul - ur) * ih2);
      }
      const long long c = (long long)m * Nc + cx;
      Xc[c] = xs;
      Bc[c] = bs;
      if (E) E[c] = 0;
    }
  } else {
    const long long nc = (long long)Nc * Nc, nf = (long long)Nf * Nf;
    const int py = 2 * cy + 1, px = 2 * cx + 1;
    for (int m = q.m0; m < M; m += q.dm) {
      const T* u = U + (long long)m * nf;
      const T* f = F + (long long)m * nf;
      T xs = 0, bs = 0;
#pragma unroll
      for (int oy = -1; oy <= 1; ++oy)
#pragma unroll
        for (int ox = -1; ox <= 1; ++ox) {
          const int yy = py + oy, xx = px + ox;
          const T w = (T)((oy == 0 ? 2 : 1) * (ox == 0 ? 2 : 1)) * (T)0.0625;
          const long long pp = (long long)yy * Nf + xx;
          const T uc = u[pp];
          T s = 0;
          const T a0 = u[pp - (xx > 0 ? 1 : 0)], a1 = u[pp + (xx < Nf - 1 ? 1 : 0)];
          const T a2 = u[pp - (yy > 0 ? Nf : 0)], a3 = u[pp + (yy < Nf - 1 ? Nf : 0)];
          s += xx > 0 ? a0 : (T)0;
          s += xx < Nf - 1 ? a1 : (T)0;
          s += yy > 0 ? a2 : (T)0;
          s += yy < Nf - 1 ? a3 : (T)0;
          xs += w * uc;
          bs += w * (f[pp] - (4 * uc - s) * ih2);
        }
      const long long c = (long long)m * nc + (long long)cy * Nc + cx;
      Xc[c] = xs;
      Bc[c] = bs;
      if (E) E[c] = 0;
    }
  }
}

// 1D weights of fine index x (0-based) on coarse indices: odd x -> coarse (x-1)/2 (1), even x ->
// coarse x/2 - 1 and x/2 (1/2 each; missing ones are boundary zeros)
template <typename T>
__device__ __forceinline__ void lin_weights(int x, int Nc, int& c0, T& w0, int& c1, T& w1) {
  if (x & 1) {
    c0 = (x - 1) / 2; w0 = 1; c1 = c0; w1 = 0;
  } else {
    c0 = x / 2 - 1; w0 = (T)0.5; c1 = x / 2; w1 = (T)0.5;
    if (c0 < 0) { c0 = 0; w0 = 0; }
    if (c1 >= Nc) { c1 = Nc - 1; w1 = 0; }
  }
}

// u_f += P e_c, linear (1D) / bilinear (2D) interpolation in space, per time level; one thread per
// fine point (1D, 4095 points x M = 4096, FP64: 0.10 ms, of which the FP64 pipe needs 0.09).
template <typename T, int NJ>
__global__ void __launch_bounds__(256) prolong_add_kernel(const __grid_constant__ TransferBatch<T, NJ> B) {
  TransferPlace q;
  const TransferJob<T>& J = transfer_place(B, q);
  const int Nf = J.Nf, M = J.M;
  const int Nc = (Nf - 1) / 2;
  const int x = q.x, y = q.y;
  if (x >= Nf) return;
  const T* __restrict__ E = J.E;
  T* __restrict__ U = J.U;
  int ax0, ax1;
  T wx0, wx1;
  lin_weights<T>(x, Nc, ax0, wx0, ax1, wx1);
  if (!kPlain2D<T> || J.dim == 1) {
    for (int m = q.m0; m < M; m += q.dm) {
      const T* e = E + (long long)m * Nc;
      U[(long long)m * Nf + x] += wx0 * e[ax0] + wx1 * e[ax1];
    }
  } else {
    const long long nc = (long long)Nc * Nc, nf = (long long)Nf * Nf;
    int ay0, ay1;
    T wy0, wy1;
    lin_weights<T>(y, Nc, ay0, wy0, ay1, wy1);
    const long long pp = (long long)y * Nf + x;
    for (int m = q.m0; m < M; m += q.dm) {
      const T* e = E + (long long)m * nc;
      const T v = wy0 * (wx0 * e[(long long)ay0 * Nc + ax0] + wx1 * e[(long long)ay0 * Nc + ax1]) +
                  wy1 * (wx0 * e[(long long)ay1 * Nc + ax0] + wx1 * e[(long long)ay1 * Nc + ax1]);
      U[(long long)m * nf + pp] += v;
    }
  }
}

// The same on grid functions stored by colour (2D), in blocks of 64 points x 4 rows (split_block): the
// rows above and below a row are then read by the same CTA at the same time level, and L2 is read 1.4
// instead of 2.5 times (u) per value.  Restriction, one thread per coarse point ...
template <typename T>
__global__ void restrict_pre_split_kernel(int Nf, double inv_h2, int M, const T* __restrict__ U, const T* __restrict__ F,
                                          T* __restrict__ Xc, T* __restrict__ Bc) {
  const int Nc = (Nf - 1) / 2;
  const int cx = blockIdx.x * blockDim.x + threadIdx.x, cy = blockIdx.y * blockDim.y + threadIdx.y;
  if (cx >= Nc || cy >= Nc) return;
  const long long nc = (long long)Nc * Nc, nf = (long long)Nf * Nf;
  const T ih2 = (T)inv_h2;
  const int py = 2 * cy + 1;
  // place of fine point (py + oy, 2 cx + 1 + ox): row base by colour, then cx + {-1, 0, 0, 1, 1}
  long long row[5][2];
#pragma unroll
  for (int oy = -2; oy <= 2; ++oy)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int yy = py + oy;  // rows outside the grid are not read
      row[oy + 2][c] = split_row(Nf, c, yy < 0 ? 0 : yy) + cx;
    }
  auto at = [&](int oy, int ox) -> long long { return row[oy + 2][(ox + oy) & 1] + ((ox + 3) >> 1) - 1; };
  const bool left = cx > 0, right = 2 * cx + 3 < Nf, up = py > 1, down = py + 2 < Nf;
  const long long cpos = split_pos(Nc, cy, cx);
  for (int m = blockIdx.z; m < M; m += gridDim.z) {
    const T* u = U + (long long)m * nf;
    const T* f = F + (long long)m * nf;
    T xs = 0, bs = 0;
#pragma unroll
    for (int oy = -1; oy <= 1; ++oy)
#pragma unroll
      for (int ox = -1; ox <= 1; ++ox) {
        const T w = (T)((oy == 0 ? 2 : 1) * (ox == 0 ? 2 : 1)) * (T)0.0625;
        const T uc = u[at(oy, ox)];
        T s = 0;
        if (ox > -1 || left) s += u[at(oy, ox - 1)];
        if (ox < 1 || right) s += u[at(oy, ox + 1)];
        if (oy > -1 || up) s += u[at(oy - 1, ox)];
        if (oy < 1 || down) s += u[at(oy + 1, ox)];
        xs += w * uc;
        bs += w * (f[at(oy, ox)] - (4 * uc - s) * ih2);
      }
    Xc[(long long)m * nc + cpos] = xs;
    Bc[(long long)m * nc + cpos] = bs;
  }
}

// ... and prolongation, one thread per pair of fine points (y, 2 j), (y, 2 j + 1), which share their
// coarse columns j - 1 and j; kProlongM time levels are loaded before the first is written (the
// compiler cannot move a load of U above a store to it)
constexpr int kProlongM = 4;
template <typename T>
__global__ void prolong_add_split_kernel(int Nf, int M, const T* __restrict__ E, T* __restrict__ U) {
  const int Nc = (Nf - 1) / 2;
  const int j = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y * blockDim.y + threadIdx.y;
  if (2 * j >= Nf || y >= Nf) return;
  const long long nf = (long long)Nf * Nf, nc = (long long)Nc * Nc;
  int ay0, ay1, ax0, ax1;
  T wy0, wy1, wx0, wx1;
  lin_weights<T>(y, Nc, ay0, wy0, ay1, wy1);
  lin_weights<T>(2 * j, Nc, ax0, wx0, ax1, wx1);  // the even point; the odd one is over column j = ax1
  const bool two = 2 * j + 1 < Nf, rows = wy1 != (T)0;
  const long long e00 = split_pos(Nc, ay0, ax0), e01 = split_pos(Nc, ay0, ax1);
  const long long e10 = split_pos(Nc, ay1, ax0), e11 = split_pos(Nc, ay1, ax1);
  const long long u0 = split_pos(Nf, y, 2 * j), u1 = two ? split_pos(Nf, y, 2 * j + 1) : u0;
  const int z = gridDim.z;
  for (int m0 = blockIdx.z; m0 < M; m0 += z * kProlongM) {
    T a0[kProlongM], a1[kProlongM], b0[kProlongM], b1[kProlongM], v0[kProlongM], v1[kProlongM];
#pragma unroll
    for (int i = 0; i < kProlongM; ++i) {
      const int m = min(m0 + i * z, M - 1);
      const T* e = E + (long long)m * nc;
      const T* u = U + (long long)m * nf;
      a0[i] = e[e00];
      a1[i] = e[e01];
      b0[i] = rows ? e[e10] : (T)0;
      b1[i] = rows ? e[e11] : (T)0;
      v0[i] = u[u0];
      v1[i] = u[u1];
    }
#pragma unroll
    for (int i = 0; i < kProlongM; ++i) {
      const int m = m0 + i * z;
      if (m >= M) break;
      T* u = U + (long long)m * nf;
      u[u0] = v0[i] + (wy0 * (wx0 * a0[i] + wx1 * a1[i]) + wy1 * (wx0 * b0[i] + wx1 * b1[i]));
      if (two) u[u1] = v1[i] + (wy0 * a1[i] + wy1 * b1[i]);
    }
  }
}

// Copies between a 2D FP64 grid function by rows and an FP32 one by colour: SPLIT_FROM: y = (float) x;
// SPLIT_TO: x = y; SPLIT_ADD: x += y.  One thread per pair of points of a row.
enum { SPLIT_FROM = 0, SPLIT_TO = 1, SPLIT_ADD = 2 };
template <int OP, typename Conv>
__global__ void split_copy_kernel(int N, int M, double* __restrict__ x, float* __restrict__ y, Conv to_float) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x, iy = blockIdx.y;
  if (2 * j >= N) return;
  const long long n = (long long)N * N, xp = (long long)iy * N + 2 * j;
  const long long a = split_row(N, iy & 1, iy) + j, b = split_row(N, 1 - (iy & 1), iy) + j;  // even, odd column
  const bool two = 2 * j + 1 < N;
  for (int m = blockIdx.z; m < M; m += gridDim.z) {
    double* xm = x + m * n + xp;
    float* ym = y + m * n;
    if (OP == SPLIT_FROM) {
      ym[a] = to_float(xm[0]);
      if (two) ym[b] = to_float(xm[1]);
    } else if (OP == SPLIT_TO) {
      xm[0] = (double)ym[a];
      if (two) xm[1] = (double)ym[b];
    } else {
      xm[0] += (double)ym[a];
      if (two) xm[1] += (double)ym[b];
    }
  }
}

// Gathers, for the points of one colour, X = u and B = F - A_h u into compact arrays (the time
// product R~ X is then subtracted by the MATVEC walk).  colour < 0: all points, in place order.
// One thread per point of the row blockIdx.y (1D: the only row): the colour's points of row y are
// x = x0 + 2 j with compact indices c0 + j (colour_pos order), so nothing is divided.
template <typename T>
__global__ void gather_defect_kernel(int dim, int N, int colour, double inv_h2, int M, const T* __restrict__ U,
                                     const T* __restrict__ F, T* __restrict__ Xo, T* __restrict__ Bo) {
  const int y = blockIdx.y;
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const long long nf = dim == 1 ? N : (long long)N * N;
  long long ncol, c;
  int x;
  if (colour < 0) {
    if (j >= N) return;
    x = j;
    ncol = nf;
    c = (long long)y * N + x;
  } else {
    ncol = colour_count(dim, N, colour);
    const int first = colour == 0 ? (N + 1) / 2 : N / 2;  // points of the colour in an even row
    const bool even_row = dim == 1 || (y & 1) == 0;
    const int n_row = even_row ? first : N - first;
    if (j >= n_row) return;
    x = (even_row ? colour : 1 - colour) + 2 * j;
    c = dim == 1 ? j : (long long)(y / 2) * N + (even_row ? 0 : first) + j;
  }
  const long long pp = (long long)y * N + x;
  const T ih2 = (T)inv_h2;
  const T diag = dim == 1 ? (T)2 : (T)4;
  for (int m = blockIdx.z; m < M; m += gridDim.z) {
    const T* u = U + (long long)m * nf;
    const T uc = u[pp];
    T s = 0;
    if (x > 0) s += u[pp - 1];
    if (x < N - 1) s += u[pp + 1];
    if (dim == 2) {
      if (y > 0) s += u[pp - N];
      if (y < N - 1) s += u[pp + N];
    }
    if (Xo) Xo[(long long)m * ncol + c] = uc;
    Bo[(long long)m * ncol + c] = F[(long long)m * nf + pp] - (diag * uc - s) * ih2;
  }
}

// F = f + d_{m,m} g  (initial data moved to the right-hand side); blockIdx.y unused (flat points)
template <typename T>
__global__ void add_initial_kernel(long long npts, int M, const T* __restrict__ f, const T* __restrict__ dmm,
                                   const T* __restrict__ g, T* __restrict__ F) {
  for (long long pp = blockIdx.x * (long long)blockDim.x + threadIdx.x; pp < npts;
       pp += (long long)gridDim.x * blockDim.x)
    for (int m = blockIdx.z; m < M; m += gridDim.z) {
      const long long idx = (long long)m * npts + pp;
      F[idx] = f[idx] + (g ? dmm[m] * g[pp] : (T)0);
    }
}

// Launch shapes of the kernels on grid functions stored by colour: blocks of 64 points x 4 rows, time
// levels strided along z as in plane_grid
inline dim3 split_block() { return dim3(64, 4); }
inline dim3 split_grid(long long nx, long long ny, int M, int sms) {
  const long long bx = (nx + 63) / 64, by = (ny + 3) / 4;
  long long bz = ((long long)sms * 16 + bx * by - 1) / (bx * by);
  bz = bz > M ? M : bz < 1 ? 1 : bz;
  return dim3((unsigned)bx, (unsigned)by, (unsigned)(bz > 65535 ? 65535 : bz));
}

// Launch shape for a grid function with nx points per row and ny rows (1 in 1D) over M time levels:
// enough CTAs along the time levels for about 16 per SM, each CTA then strides over time.
inline dim3 plane_grid(long long nx, long long ny, int M, int sms, int threads = 256) {
  const long long bx = (nx + threads - 1) / threads;
  const long long per = bx * ny;
  long long bz = ((long long)sms * 16 + per - 1) / per;
  if (bz > M) bz = M;
  if (bz < 1) bz = 1;
  if (bz > 65535) bz = 65535;
  return dim3((unsigned)bx, (unsigned)ny, (unsigned)bz);
}

}  // namespace fhmg
