// tcgen05 variant of the panel walk for wide panels (2D grids): BF16 products with FP32
// accumulation in tensor memory, FP32 grid functions.
//
// The walk of panel.cuh transposed onto the 5th-generation tensor cores.  A CTA owns a tile of
// 128 spatial columns; thread c of the four walk warps owns column c (TMEM lane c), and four memory
// warps load and store the columns a leaf ahead and behind (see the kernel).  Every
// chunk product of a leaf row i becomes one tcgen05.mma with M = 128 (the columns), N = the chunk's
// output rows, K = its reduction index, A from shared memory (the columns' operand tile, 128 x K,
// K-major) and B = the chunk itself (N x K, K-major, streamed by TMA bulk copies in the canonical
// no-swizzle core-matrix layout of build_panel_umma):
//   DENSE(j)  acc[c, r] += sum_k x_j[c, k] D_ij[r, k]        A = ring tile of leaf j
//   UPART     acc[c, r] += sum_k z[c, k] U_i[r, k]           A = the columns' z values, staged
//   DIAG      smoother: res[c, r] = sum_k y[c, k] Dinv'[r, k], y = b - acc, x = res + dinv_rr y
//             product:  acc[c, r] += sum_k x_i[c, k] D'_ii[r, k], out = b - acc - d_rr x
//   VPART     v[c, q] = sum_k x_i[c, k] V_i[q, k], then z[c, code_q] (+)= v[c, q]
// (D', Dinv': without their diagonal, which is applied in FP32 by the threads).  One elected thread
// issues the MMAs; tcgen05.commit signals their completion on mbarriers: the slot's "empty" barrier
// (which also collects one arrival per walk warp, so a slot is refilled only when the MMA and
// every warp are done with it) and the acc / res / v barriers that the threads wait on before they
// read tensor memory with tcgen05.ld.  Threads write the A tiles (x ring, y, z) with 16-byte stores
// in the core-matrix layout, then fence.proxy.async and meet on the walk warps' mbarrier before the MMA
// that reads them is issued.  Every wait is bounded and watches the shared abort flag; every exit
// path frees the tensor memory after the MMAs in flight completed.
#pragma once
#include <cstdint>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "walk.h"

namespace fhmg {

constexpr int kUmmaCols = 128;                 // columns per tile = MMA M = TMEM lanes
constexpr int kUmmaBlock = 2 * kUmmaCols + 32;  // walk threads, memory threads, producer warp
constexpr uint32_t kUmmaTmemCols = 256;        // acc / res [0,64), v [64,128), two leaf buffers [128,256)

struct UmmaSmem {
  size_t ring, zstage, zpool, bar, ebar, cbar, xbar, desc, flag, tslot, total;
};
// x ring (W tiles of 128 x 64 BF16), for the product one staging tile that holds the columns' z values for
// the U products, z pool (pool x 128 FP32), mbarriers, slot descriptors, abort flag, TMEM address.  The
// smoother stages z, then y (for the inverse's product), in the tile that x_i takes at the end of the
// leaf (each is read by MMAs that completed before the next is written), and so leaves the L1 cache
// room: its lines are what the memory warps' loads in flight wait for (see umma_launch_t).
// Operand tiles are 128-byte aligned.
__host__ __device__ inline UmmaSmem umma_smem(int pool, int W, int slot_bytes, int ns, bool smoother) {
  auto a128 = [](size_t x) { return (x + 127) & ~(size_t)127; };
  const size_t tile = (size_t)kUmmaCols * kUmmaL * 2;
  UmmaSmem s;
  s.ring = a128((size_t)ns * slot_bytes);
  s.zstage = s.ring + (size_t)W * tile;
  s.zpool = s.zstage + (smoother ? 0 : tile);
  s.bar = a128(s.zpool + (size_t)pool * kUmmaCols * 4);
  s.ebar = s.bar + 8 * (size_t)ns;
  s.cbar = s.ebar + 8 * (size_t)ns;  // consumer warps' barrier
  s.xbar = s.cbar + 8;               // acc, res, v (MMA completion), exit, done, leaf buffers: filled[2], walked[2]
  s.desc = (s.xbar + 9 * 8 + 15) & ~(size_t)15;
  s.flag = s.desc + 16 * (size_t)ns;
  s.tslot = s.flag + 16;
  s.total = a128(s.tslot + 16);
  return s;
}

// byte offset of entry (r, k) of a K-major operand tile with K columns (core-matrix layout)
__device__ __forceinline__ uint32_t umma_off(int r, int k, int K) {
  return (uint32_t)((((r >> 3) * (K >> 3)) + (k >> 3)) * 128 + (r & 7) * 16 + (k & 7) * 2);
}

// shared-memory matrix descriptor: start address, leading (K) byte offset 128, stride (8-row
// group) byte offset, fixed bits 46-48 = 0b001, no swizzle
__device__ __forceinline__ uint64_t umma_desc(uint32_t addr, uint32_t sbo) {
  return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)(128 >> 4) << 16) | ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) |
         ((uint64_t)1 << 46);
}

// instruction descriptor of kind::f16: FP32 D, BF16 A and B, both K-major, M = 128, N
__device__ __forceinline__ uint32_t umma_idesc(int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(kUmmaCols >> 4) << 24);
}

// ---- operand layout of 64-column tiles: K-major, 128-byte swizzle ----
// A tile row holds its 64 K entries (BF16) in 128 bytes; 8-row groups form 1024-byte atoms in which
// the 16-byte chunk c of row r sits at chunk position c ^ (r % 8) (the tensor core reads the atoms
// without bank conflicts).  Tiles start on 1024-byte boundaries.
__host__ __device__ inline uint32_t sw128_off(int r, int k) {
  return (uint32_t)((r >> 3) * 1024 + (r & 7) * 128 + ((((k >> 3) ^ r) & 7) << 4) + (k & 7) * 2);
}
// shared-memory descriptor of such a tile: start address, leading byte offset unused (1), 8-row
// groups 1024 bytes apart, fixed bits 46-48 = 0b001, swizzle mode 128B (2 in bits 61-63); a K step
// of 16 entries (32 bytes) advances the start address field by 2
__device__ __forceinline__ uint64_t sw128_desc(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) |
         ((uint64_t)2 << 61);
}

// D[tmem] (+)= A B^T over K = 16 * steps, A (128 x K) and B (N x K) K-major tiles at a_addr / b_addr
__device__ __forceinline__ void umma_product(uint32_t tmem, uint32_t a_addr, uint32_t b_addr, int K, int N,
                                             bool accumulate) {
  const uint32_t idesc = umma_idesc(N);
  const uint32_t sbo = (uint32_t)(K / 8) * 128;
  for (int s = 0; s < K / 16; ++s) {
    const uint64_t ad = umma_desc(a_addr + 256u * s, sbo);
    const uint64_t bd = umma_desc(b_addr + 256u * s, sbo);
    const uint32_t acc = (accumulate || s > 0) ? 1u : 0u;
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
        : "memory");
  }
}

__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void tc_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void async_proxy_fence() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// 16 consecutive TMEM columns of this thread's lane (the warp's lane quarter), as floats
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
  // the loaded registers are read only after the wait
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    asm volatile("" : "+r"(r[j]));
    v[j] = __uint_as_float(r[j]);
  }
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  const uint32_t lo = __bfloat16_as_ushort(__float2bfloat16_rn(a));
  const uint32_t hi = __bfloat16_as_ushort(__float2bfloat16_rn(b));
  return lo | (hi << 16);
}

// row c of a K-major operand tile with K columns: 8 consecutive entries k0..k0+7 as one 16-byte store
__device__ __forceinline__ void put8(unsigned char* tile, int c, int k0, int K, const float* v) {
  uint4 q;
  q.x = pack_bf16(v[0], v[1]);
  q.y = pack_bf16(v[2], v[3]);
  q.z = pack_bf16(v[4], v[5]);
  q.w = pack_bf16(v[6], v[7]);
  *reinterpret_cast<uint4*>(tile + umma_off(c, k0, K)) = q;
}

// row c of a K-major operand tile: entries k0..k0+7 already packed as BF16 pairs
__device__ __forceinline__ void put8_packed(unsigned char* tile, int c, int k0, int K, const uint32_t* q) {
  *reinterpret_cast<uint4*>(tile + umma_off(c, k0, K)) = make_uint4(q[0], q[1], q[2], q[3]);
}

// 16 consecutive TMEM columns of this thread's lane written
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float (&v)[16]) {
  uint32_t r[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) r[j] = __float_as_uint(v[j]);
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15};" ::"r"(r[0]),
      "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
      "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%8], {%0,%1,%2,%3,%4,%5,%6,%7};" ::"r"(r[0]), "r"(r[1]), "r"(r[2]),
               "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// a load kept in program order with its like and with every other access to memory (so that a group of
// loads is in flight before the first use).  Not by the non-coherent path: a line solve may work in place
// (X aliases B), so its launch writes what it reads, each element after its only read, by the same thread
__device__ __forceinline__ float ld_ordered(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
  return v;
}

// one lane of a converged warp
__device__ __forceinline__ bool umma_elect() {
  uint32_t p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0;
}

// Columns of a 2D colour in tiles of 4 grid rows x 32 points of the colour (64 grid points), thread c
// point c % 32 of row c / 32: the rows above and below a row are then read by the same CTA, twice
// instead of three times from L2 (20 instead of 32 bytes per value)
__host__ __device__ inline long long umma_tiles(const Geo& g, long long ncols) {
  if (g.dim != 2) return (ncols + kUmmaCols - 1) / kUmmaCols;
  return (long long)((g.N + 3) / 4) * (((g.N + 1) / 2 + 31) / 32);
}

// T = float grid functions; the jobs' Dinv are the level inverses (without diagonal) in the
// build_panel_umma layout (BF16 bits), ddiag the diagonal applied in FP32.
//
// Three roles: four walk warps (the chunk products), four memory warps (thread c: column c, as in the
// walk) and a producer warp (the chunk stream).  The memory warps run ahead of the walk through two
// leaf buffers in tensor memory (64 columns each): they load a leaf's right-hand side (smoother: F +
// neighbour sum / h^2; product: x, as BF16 pairs) into one while the walk works on the other, and
// write the leaf's result (x; B - d x - sum) back once the walk has left it there.  The walk then
// never waits for DRAM, which took most of its time when its own threads loaded the next leaf
// (a line solve of 100003 x 512 columns 214 -> 176 us; with room for the L1 cache 151).  What bounds the
// memory warps is the loads they can keep in flight: a finest half-sweep of a 1023^2 x 512 grid took 2.37
// ms with loads by the walk, 2.31 with memory warps, 1.60 with grid functions stored by colour (whole
// sectors), 1.47 with rolled loops (instruction cache), 1.04 with 60 instead of 28 KB of L1, 0.99 with a
// pointer per neighbour; its bytes need 0.48 ms.  96 registers and at most 97 KB of shared memory: two CTAs per SM.
template <int MODE>
__global__ void __launch_bounds__(kUmmaBlock, 2) humma_kernel(const __grid_constant__ WalkBatch<float, uint16_t> B) {
  constexpr int L = kUmmaL, NT = kUmmaCols;
  extern __shared__ __align__(16) unsigned char sm[];
  const UmmaSmem lay = umma_smem(B.pool, B.W, B.slot_bytes, B.ns, MODE == MODE_SMOOTH);
  unsigned char* slots = sm;
  unsigned char* ring = sm + lay.ring;
  float* zpool = reinterpret_cast<float*>(sm + lay.zpool);
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + lay.bar);
  uint64_t* empty = reinterpret_cast<uint64_t*>(sm + lay.ebar);
  uint64_t* cbar = reinterpret_cast<uint64_t*>(sm + lay.cbar);
  uint64_t* accbar = reinterpret_cast<uint64_t*>(sm + lay.xbar);
  uint64_t* resbar = accbar + 1;
  uint64_t* vbar = accbar + 2;
  uint64_t* exitbar = accbar + 3;
  uint64_t* donebar = accbar + 4;
  uint64_t* filled = accbar + 5;  // [2] a leaf buffer holds a leaf's input
  uint64_t* walked = accbar + 7;  // [2] ... its result
  int4* sdesc = reinterpret_cast<int4*>(sm + lay.desc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(sm + lay.flag);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + lay.tslot);
  const size_t tile_bytes = (size_t)NT * L * 2;

  const int t = threadIdx.x;
  const int w = t >> 5;
  const int lane = t & 31;
  const int ns = B.ns;
  const int W = B.W;

  if (t == 0) {
    for (int s = 0; s < ns; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, NT / 32 + 1);  // every walk warp + the MMAs' commit
    }
    mbar_init(cbar, NT / 32);
    for (int b = 0; b < 9; ++b) mbar_init(accbar + b, b == 3 ? 2 * NT / 32 : b >= 5 ? NT / 32 : 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (w == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(kUmmaTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_before_sync();
  __syncthreads();  // the last block-wide barrier: from here on the roles run apart
  tc_after_sync();
  const uint32_t tmem = *tslot;

  if (t >= 2 * NT) {
    // ---- producer: one lane streams every chunk of every tile of this CTA, in order ----
    if (t != 2 * NT) return;
    long long k = 0;
    int slot = 0;
    uint32_t phase = 1;  // of the slot's previous release (the first round finds every slot free)
    bool ok = true, stop = false;
    for (long long g = blockIdx.x; g < B.ntiles && ok && !stop; g += gridDim.x) {
      const WalkJob<float, uint16_t>& J = B.job[job_of(B, g)];
      const int nch = __ldg(J.P.cptr + J.P.nb);
      int4 cdn = __ldg(J.P.chunks);
      for (int c = 0; c < nch; ++c, ++k) {
        const int4 cd = cdn;
        if (c + 1 < nch) cdn = __ldg(J.P.chunks + c + 1);
        if (k + 1 == B.withhold) {
          stop = true;
          break;
        }
        if (!mbar_wait_or_abort(empty + slot, phase, abort_flag)) {
          ok = false;
          break;
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        const int type = cd.x & 15;
        const void* src = (MODE == MODE_SMOOTH && type == PK_DIAG) ? (const void*)(J.Dinv + (long long)cd.y * L * L)
                                                                    : (const void*)(J.P.pkg + 16LL * (long long)cd.w);
        sdesc[slot] = cd;
        bulk_load(slots + (size_t)slot * B.slot_bytes, src, (uint32_t)cd.z, full + slot);
        if (++slot == ns) {
          slot = 0;
          phase ^= 1;
        }
      }
    }
    if (!ok && !*abort_flag) {
      *abort_flag = 1;
      atomicExch(B.err, 1);
    }
    for (int s = 0; s < ns && s < k; ++s) {
      const long long n_s = (k - 1 - s) / ns + 1;
      mbar_wait(full + s, (uint32_t)((n_s - 1) & 1));
    }
    return;
  }

  const uint32_t lane_base = (uint32_t)(32 * (w & 3)) << 16;  // this warp's TMEM lane quarter
  const uint32_t t_acc = tmem, t_v = tmem + 64;
  const uint32_t t_buf = tmem + 128 + lane_base;  // + 64 * (leaf & 1)
  auto give_up = [&](bool ok) -> bool {
    if (__all_sync(0xffffffffu, ok)) return false;
    if (lane == 0) {
      *abort_flag = 1;
      atomicExch(B.err, 1);
    }
    return true;
  };

  if (t >= NT) {
    // ---- memory warps ----
    const int c = t - NT;
    bool failed = false;
    long long n = 0;  // leaves filled so far (over all tiles); leaf n uses buffer n & 1
    double local_max = 0.0;
    // where the leaves in the two buffers go (the even one and the odd one)
    struct Dest {
      const WalkJob<float, uint16_t>* J;
      long long at;  // element offset of the leaf's first row
      int leaf;
      bool valid;
    };
    Dest d0{nullptr, 0, 0, false}, d1{nullptr, 0, 0, false};
    // the result of leaf m (in buffer m & 1) to global memory
    auto write_leaf = [&](long long m) -> bool {
      const int buf = (int)(m & 1);
      if (give_up(mbar_wait_or_abort(walked + buf, (uint32_t)((m >> 1) & 1), abort_flag, B.spin))) return false;
      tc_after_sync();
      const Dest d = buf ? d1 : d0;
      const long long ld = d.J->geo.ld;
#pragma unroll 1
      for (int r0 = 0; r0 < L; r0 += 16) {
        float a[16];
        tmem_ld16(t_buf + 64 * buf + r0, a);
        if (MODE == MODE_SMOOTH) {
          if (d.valid) {
            float* x = d.J->X + d.at + (long long)r0 * ld;
#pragma unroll
            for (int j = 0; j < 16; ++j) x[(long long)j * ld] = a[j];
          }
        } else if (d.valid) {
          const float* bs = d.J->B + d.at + (long long)r0 * ld;
          const float* xs = d.J->X + d.at + (long long)r0 * ld;
          const float* dd = d.J->ddiag + (long long)d.leaf * L + r0;
          float* o = d.J->OUT ? d.J->OUT + d.at + (long long)r0 * ld : nullptr;
          float bv[16], xv[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            bv[j] = bs[(long long)j * ld];
            xv[j] = xs[(long long)j * ld];
          }
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const float b = bv[j] - __ldg(dd + j) * xv[j];
            const float r = b - a[j];
            if (o) o[(long long)j * ld] = r;
            const double av = fabs((double)r);
            local_max = (av > local_max || av != av) ? av : local_max;
          }
        }
      }
      if (MODE == MODE_MATVEC && d.J->norm != nullptr && d.leaf == d.J->P.nb - 1) {  // the tile is done
        for (int o = 16; o > 0; o >>= 1) {
          const double other = __shfl_xor_sync(0xffffffffu, local_max, o);
          local_max = (other > local_max || other != other) ? other : local_max;
        }
        if (lane == 0) atomicMax(d.J->norm, (unsigned long long)__double_as_longlong(local_max));
        local_max = 0.0;
      }
      tc_before_sync();  // the reads of the buffer ordered before it is filled again
      return true;
    };
    for (long long g = blockIdx.x; g < B.ntiles && !failed; g += gridDim.x) {
      const WalkJob<float, uint16_t>& J = B.job[job_of(B, g)];
      const long long ld = J.geo.ld;
      const float inv_h2 = (float)J.geo.inv_h2;
      const int nb = J.P.nb;
      const bool grid = MODE == MODE_SMOOTH && J.geo.dim > 0;
      bool valid;
      long long p = 0;
      // columns past the panel's end read column 0 (any valid address) and are zeroed, so that the loads
      // carry no predicate; missing neighbours read the right-hand side with weight 0 (never X: the point
      // itself and column 0 are of the colour that this launch writes)
      const float *q0 = J.B, *q1 = J.B, *q2 = J.B, *q3 = J.B;
      float w0 = 0.f, w1 = 0.f, w2 = 0.f, w3 = 0.f;
      if (grid) {
        const int N = J.geo.N;
        int iy = 0, ix;
        if (J.geo.dim == 2) {
          const int first = (N + 1) / 2, nbx = (first + 31) / 32;
          const long long tt = g - J.tile0;
          iy = (int)(tt / nbx) * 4 + (c >> 5);
          ix = ((iy + J.geo.colour) & 1) + 2 * ((int)(tt % nbx) * 32 + (c & 31));
          valid = iy < N && ix < N;
        } else {
          const long long cg = (g - J.tile0) * NT + c;
          ix = (int)(2 * cg) + J.geo.colour;
          valid = cg < J.ncols;
        }
        if (valid) {
          p = (long long)iy * N + ix;
          if (ix > 0) w0 = inv_h2;
          if (ix < N - 1) w1 = inv_h2;
          if (J.geo.dim == 2 && iy > 0) w2 = inv_h2;
          if (J.geo.dim == 2 && iy < N - 1) w3 = inv_h2;
        }
        if (J.geo.split && valid) p = split_pos(N, iy, ix);
        const NbrOffsets off = nbr_offsets(J.geo);
        const bool odd = iy & 1;
        const int left = odd ? off.left[1] : off.left[0];
        q0 = w0 != 0.f ? J.X + p + left : J.B + p;
        q1 = w1 != 0.f ? J.X + p + left + off.step : J.B + p;
        q2 = w2 != 0.f ? J.X + p + (odd ? off.up[1] : off.up[0]) : J.B + p;
        q3 = w3 != 0.f ? J.X + p + (odd ? off.down[1] : off.down[0]) : J.B + p;
      } else {
        const long long cg = (g - J.tile0) * NT + c;
        valid = cg < J.ncols;
        p = valid ? cg : 0;
      }
      const float keep = valid ? 1.f : 0.f;
      for (int i = 0; i < nb; ++i, ++n) {
        const int buf = (int)(n & 1);
        if (n >= 2 && !write_leaf(n - 2)) {
          failed = true;
          break;
        }
        const long long at = (long long)i * L * ld;
        if (grid) {
          const float* Bl = J.B + p;
#pragma unroll 1
          for (int r0 = 0; r0 < L; r0 += 8) {
            float v[8], a0[8], a1[8], a2[8], a3[8];
            uint32_t q[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const long long o = at + (long long)(r0 + j) * ld;
              v[j] = ld_ordered(Bl + o);
              a0[j] = ld_ordered(q0 + o);
              a1[j] = ld_ordered(q1 + o);
              a2[j] = ld_ordered(q2 + o);
              a3[j] = ld_ordered(q3 + o);
            }
#pragma unroll
            for (int j = 0; j < 8; ++j)
              q[j] = __float_as_uint(keep * (v[j] + w0 * a0[j] + w1 * a1[j] + w2 * a2[j] + w3 * a3[j]));
            tmem_st8(t_buf + 64 * buf + r0, q);
          }
        } else if (MODE == MODE_SMOOTH) {
          const float* Bl = J.B + at + p;
#pragma unroll 1
          for (int r0 = 0; r0 < L; r0 += 32) {
            float v[32];
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = ld_ordered(Bl + (long long)(r0 + j) * ld);
#pragma unroll
            for (int j = 0; j < 32; j += 8) {
              uint32_t q[8];
#pragma unroll
              for (int e = 0; e < 8; ++e) q[e] = __float_as_uint(v[j + e] * keep);
              tmem_st8(t_buf + 64 * buf + r0 + j, q);
            }
          }
        } else {
          const float* Xl = J.X + at + p;
#pragma unroll 1
          for (int r0 = 0; r0 < L; r0 += 32) {
            float v[32];
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = Xl[(long long)(r0 + j) * ld];
#pragma unroll
            for (int j = 0; j < 32; j += 16) {
              uint32_t q[8];
#pragma unroll
              for (int e = 0; e < 8; ++e) q[e] = pack_bf16(v[j + 2 * e] * keep, v[j + 2 * e + 1] * keep);
              tmem_st8(t_buf + 64 * buf + (r0 + j) / 2, q);
            }
          }
        }
        const Dest d{&J, at + p, i, valid};
        if (buf)
          d1 = d;
        else
          d0 = d;
        tmem_st_wait();
        tc_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(filled + buf);
      }
    }
    if (!failed) failed = (n >= 2 && !write_leaf(n - 2)) || (n >= 1 && !write_leaf(n - 1));
  } else {
    // ---- walk warps ----
    const int c = t;
    const bool leader = umma_elect() && w == 0;  // issues the MMAs
    uint32_t cbphase = 0, accph = 0, resph = 0, vph = 0;
    int cslot = 0;
    uint32_t cphase = 0;
    bool failed = false;
    long long n = 0;  // leaves walked so far
    // all walk warps meet (bounded); tensor-memory reads and shared writes before it are ordered
    // before the MMAs issued after it
    auto walk_sync = [&]() -> bool {
      async_proxy_fence();
      tc_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(cbar);
      const bool ok = mbar_wait_or_abort(cbar, cbphase, abort_flag, B.spin);
      cbphase ^= 1;
      tc_after_sync();
      return !give_up(ok);
    };
    auto wait_on = [&](uint64_t* bar, uint32_t& ph) -> bool {
      const bool ok = mbar_wait_or_abort(bar, ph, abort_flag, B.spin);
      ph ^= 1;
      tc_after_sync();
      return !give_up(ok);
    };
    for (long long g = blockIdx.x; g < B.ntiles && !failed; g += gridDim.x) {
      const WalkJob<float, uint16_t>& J = B.job[job_of(B, g)];
      const float* ddg = J.ddiag;
      const int nb = J.P.nb;
      for (int i = 0; i < nb && !failed; ++i, ++n) {
        unsigned char* xr_i = ring + (size_t)(i % W) * tile_bytes;
        unsigned char* const ystage = xr_i;  // smoother: until x_i takes its place
        unsigned char* const zstage = MODE == MODE_SMOOTH ? xr_i : sm + lay.zstage;
        const int buf = (int)(n & 1);
        const uint32_t bphase = (uint32_t)((n >> 1) & 1);
        const uint32_t t_b = t_buf + 64 * buf;
        if (MODE == MODE_MATVEC) {
          // x_i into the ring (its slot's previous tile, x_{i-W}, was last read by leaf i-1's MMAs,
          // complete since every walk thread waited on their barriers)
          if (give_up(mbar_wait_or_abort(filled + buf, bphase, abort_flag, B.spin))) {
            failed = true;
            break;
          }
          tc_after_sync();
#pragma unroll 1
          for (int r0 = 0; r0 < L / 2; r0 += 16) {
            float v[16];
            tmem_ld16(t_b + r0, v);
            uint32_t q[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) q[j] = __float_as_uint(v[j]);
#pragma unroll
            for (int j = 0; j < 16; j += 4) put8_packed(xr_i, c, 2 * (r0 + j), L, &q[j]);
          }
        }
        bool acc_used = false;
        int nu = 0;  // UPART chunks of this leaf so far
        for (bool leaf_done = false; !leaf_done && !failed;) {
          if (give_up(mbar_wait_or_abort(full + cslot, cphase, abort_flag, B.spin))) {
            failed = true;
            break;
          }
          const int4 cd = sdesc[cslot];
          leaf_done = ((cd.x >> 12) & 1) != 0;
          const int type = cd.x & 15, cnt = (cd.x >> 4) & 0xff;
          unsigned char* buf_c = slots + (size_t)cslot * B.slot_bytes;
          const uint32_t b_addr = smem_u32(buf_c);
          if (type == PK_DENSE) {
            if (leader) {
              tc_after_sync();
              umma_product(t_acc, smem_u32(ring + (size_t)(cd.y % W) * tile_bytes), b_addr, L, L, acc_used);
              umma_commit(empty + cslot);
            }
            acc_used = true;
          } else if (type == PK_UPART) {
            const int kp = cnt;  // padded to 16; padding columns of U are zero
            if (nu > 0) {  // the previous U product of this leaf has read the staging tile
              if (leader) umma_commit(accbar);
              if (!wait_on(accbar, accph)) {
                failed = true;
                break;
              }
            }
            const int* uz = reinterpret_cast<const int*>(buf_c + (size_t)L * kp * 2);
            for (int k0 = 0; k0 < kp; k0 += 8) {
              float zv[8];
#pragma unroll
              for (int e = 0; e < 8; ++e) zv[e] = zpool[uz[k0 + e] * NT + c];
              put8(zstage, c, k0, kp, zv);
            }
            if (!walk_sync()) {
              failed = true;
              break;
            }
            if (leader) {
              umma_product(t_acc, smem_u32(zstage), b_addr, kp, L, acc_used);
              umma_commit(empty + cslot);
            }
            acc_used = true;
            ++nu;
          } else if (type == PK_DIAG) {
            if (MODE == MODE_SMOOTH) {
              if (acc_used) {
                if (leader) umma_commit(accbar);
                if (!wait_on(accbar, accph)) {
                  failed = true;
                  break;
                }
              }
              if (give_up(mbar_wait_or_abort(filled + buf, bphase, abort_flag, B.spin))) {
                failed = true;
                break;
              }
              tc_after_sync();
              // y = b - acc, kept in the leaf buffer and staged as the A operand of the inverse's product
#pragma unroll 1
              for (int r0 = 0; r0 < L; r0 += 16) {
                float y[16];
                tmem_ld16(t_b + r0, y);
                if (acc_used) {
                  float a[16];
                  tmem_ld16(t_acc + lane_base + r0, a);
#pragma unroll
                  for (int j = 0; j < 16; ++j) y[j] -= a[j];
                  tmem_st16(t_b + r0, y);
                }
                put8(ystage, c, r0, L, &y[0]);
                put8(ystage, c, r0 + 8, L, &y[8]);
              }
              tmem_st_wait();
              if (!walk_sync()) {
                failed = true;
                break;
              }
              if (leader) {
                umma_product(t_acc, smem_u32(ystage), b_addr, L, L, false);
                umma_commit(empty + cslot);
                umma_commit(resbar);
              }
              if (!wait_on(resbar, resph)) {
                failed = true;
                break;
              }
              // x = res + dinv_rr y into the ring and, for the memory warps, the leaf buffer
              const float* dd = ddg + (long long)i * L;
#pragma unroll 1
              for (int r0 = 0; r0 < L; r0 += 16) {
                float a[16], y[16];
                tmem_ld16(t_acc + lane_base + r0, a);
                tmem_ld16(t_b + r0, y);
#pragma unroll
                for (int j = 0; j < 16; ++j) y[j] = a[j] + __ldg(dd + r0 + j) * y[j];
                put8(xr_i, c, r0, L, &y[0]);
                put8(xr_i, c, r0 + 8, L, &y[8]);
                tmem_st16(t_b + r0, y);
              }
              tmem_st_wait();
              if (!walk_sync()) {  // x_i complete in the ring before the V products read it
                failed = true;
                break;
              }
              if (lane == 0) mbar_arrive(walked + buf);
            } else {
              if (!walk_sync()) {  // x_i staged by every thread
                failed = true;
                break;
              }
              if (leader) {
                umma_product(t_acc, smem_u32(xr_i), b_addr, L, L, acc_used);
                umma_commit(empty + cslot);
                umma_commit(accbar);
              }
              if (!wait_on(accbar, accph)) {
                failed = true;
                break;
              }
#pragma unroll 1
              for (int r0 = 0; r0 < L; r0 += 16) {
                float a[16];
                tmem_ld16(t_acc + lane_base + r0, a);
                tmem_st16(t_b + r0, a);
              }
              tmem_st_wait();
              if (!walk_sync()) {  // every thread has read acc before the next leaf's MMAs
                failed = true;
                break;
              }
              if (lane == 0) mbar_arrive(walked + buf);
            }
          } else {  // PK_VPART: z entries from x_i
            const int np = (cnt + 15) / 16 * 16;
            if (leader) {
              umma_product(t_v, smem_u32(xr_i), b_addr, L, np, false);
              umma_commit(empty + cslot);
              umma_commit(vbar);
            }
            if (!wait_on(vbar, vph)) {
              failed = true;
              break;
            }
            const int* codes = reinterpret_cast<const int*>(buf_c + (size_t)np * L * 2);
            for (int q0 = 0; q0 < cnt; q0 += 16) {
              float a[16];
              tmem_ld16(t_v + lane_base + q0, a);
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                if (q0 + j < cnt) {
                  const int code = codes[q0 + j];
                  float* z = zpool + (code >> 1) * NT + c;
                  *z = (code & 1) ? a[j] : *z + a[j];
                }
              }
            }
            if (!leaf_done && !walk_sync()) {  // v is read before the next V product overwrites it
              failed = true;
              break;
            }
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(empty + cslot);  // this warp is done with the slot
          if (++cslot == ns) {
            cslot = 0;
            cphase ^= 1;
          }
        }
      }
    }
    if (leader) umma_commit(donebar);
  }
  // exit (normal or after a wait gave up): the MMAs issued so far complete, every walk and memory warp
  // is done with tensor memory (a barrier used once, so its phase is 0 whatever happened before), then
  // the allocating warp frees it.  Every wait is bounded, so every warp arrives.
  tc_before_sync();
  __syncwarp();
  if (lane == 0) mbar_arrive(exitbar);
  if (w == 0) {
    mbar_wait(exitbar, 0);
    mbar_wait(donebar, 0);
    tc_after_sync();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kUmmaTmemCols));
  }
}

}  // namespace fhmg
