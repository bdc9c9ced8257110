// FP64-accurate finest-grid defect  r = F - A_h u - (R~ (x) I) u  on the tcgen05 tensor cores, by
// error-free splitting of both factors of the time product into small-integer digits (the scheme of
// Ozaki, Ogita, Oishi & Rump, "Error-free transformations of matrix multiplication by using fast
// routines of matrix multiplication and its applications", Numer. Algorithms 59, 2012, with BF16
// digits and FP32 accumulation).
//
// Splitting.  Every row m of the dense time matrix R~ (lower triangular, M <= 512) has an exponent
// E_m with max_k |R~_mk| < 2^E_m; every grid point c has an exponent F_c with max_k |u_kc| < 2^F_c.
// Rounded to 49 bits, the scaled entries are sums of G = 7 balanced base-2^7 digits,
//     R~_mk = 2^E_m sum_a d_a(m,k) 2^{-7(a+1)},   u_kc = 2^F_c sum_b e_b(k,c) 2^{-7(b+1)},
// |d_0|, |e_0| <= 129, every other digit in [-64, 64].  Digits are small integers, exact in BF16, and
// a digit product (<= 2^14.1) is exact in the FP32 accumulator.  The products of digit pairs with
// equal a + b = g share the unit 2^{-7(g+2)}, so the group sums
//     A_g(m,c) = sum_{a+b=g} sum_k d_a(m,k) e_b(k,c)
// are integers; with K <= 512 their magnitude stays below (g+3) 2^21 <= 2^24 for g <= 5, so the
// tensor core's FP32 accumulation of these integers is exact (g = 6 may exceed 2^24 by a fraction,
// which costs at most a unit 2^-56 of the scale per accumulation step).  Then
//     sum_k R~_mk u_kc = 2^{E_m + F_c - 14} sum_g 2^{-7g} A_g(m,c) + O((m+1) 2^{E_m + F_c - 46}),
// the truncation coming from the 49-bit rounding of both factors and from the dropped groups
// g >= 7.  The group sums are combined in double-float arithmetic and joined to FP64 with integer
// operations (the FP64 pipe runs at 1/64 of the FP32 rate on GB300); a pre-pass at full occupancy
// forms B = F - A_h u (the stencil in 64-bit fixed point, sp_stencil) and the exponents F_c, and the
// kernel's epilogue writes r = B - R~ u.
//
// Kernel.  A CTA owns tiles of 64 grid points (64 MMA columns per digit, up to four digits in one MMA) and
// walks the output blocks I of 128 time rows (MMA M = 128; TMEM lane = time row).  For every K-block
// J <= 2I+1 of 64 time levels the eight split warps turn u's block J of the tile into the G digit tiles (B
// operands, 64 x 64, K-major, 128-byte swizzle, double-buffered), an MMA warp multiplies them with the
// digit tiles of R~'s block (I, J) (A operands, 128 x 64, produced by build_split, all-zero digit tiles
// left out) into the G group accumulators (G x 64 TMEM columns), and after the last J the eight epilogue
// warps read the groups back (tcgen05.ld), release tensor memory and form r while the next block's
// digits and MMAs run.  A producer warp streams the R~ digit tiles through an mbarrier ring with
// cp.async.bulk.  511^2 x 512, pre-pass included: 6.47 ms with eight warps that split and drained in turn,
// 64-column MMAs and an FP64 pre-pass, 2.49 ms now (1.77 of it this kernel, 1.34 of that MMAs and drains).  Every wait is bounded and watches the shared abort flag; every
// exit frees the tensor memory after the issued MMAs completed.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "panel.cuh"
#include "umma.cuh"
#include "walk.h"

namespace fhmg {

constexpr int kSpG = 7;                         // digits per factor = group accumulators
constexpr int kSpCols = 64;                     // grid points per tile (MMA N: 64 per digit, up to four digits)
constexpr int kSpRows = kSplitRows;             // time rows per output block (MMA M)
constexpr int kSpK = 64;                        // time levels per K-block
constexpr int kSpSplit = 256;                   // 8 warps that split u into digit tiles
constexpr int kSpEpi = 256;                     // 8 epilogue warps
constexpr int kSpBlock = kSpSplit + kSpEpi + 64;  // + producer warp + MMA warp
constexpr uint32_t kSpTmemCols = 512;
constexpr int kSpAtile = kSpRows * kSpK * 2;    // bytes of one R~ digit tile
constexpr int kSpBtile = kSpCols * kSpK * 2;    // bytes of one u digit tile
constexpr int kSpPieceLd = kSpRows + 1;         // float pairs per point of the epilogue's piece (odd: no bank conflicts)

constexpr int kSpMaxPairs = (kSplitMaxM / kSpRows) * (kSplitMaxM / kSpRows + 1);  // (I, J) blocks at the largest M

struct SplitSmem {
  size_t ring, xbuf, piece, bar, pairs, total;
};
__host__ __device__ inline SplitSmem split_smem(int ns) {
  SplitSmem s;
  s.ring = 0;
  s.xbuf = (size_t)ns * kSpAtile;
  s.piece = s.xbuf + 2 * (size_t)kSpG * kSpBtile;  // epilogue: [32 points][kSpPieceLd] float pairs
  s.bar = s.piece + (size_t)32 * kSpPieceLd * 8;
  // full[ns], empty[ns], xready[2], xfree[2], accdone, accfree, cbar, exitbar, donebar, then the
  // abort flag, the lowest group written and the TMEM address; then the pair table
  s.pairs = s.bar + 8 * ((size_t)2 * ns + 9) + 16;
  s.total = s.pairs + 8 * (size_t)kSpMaxPairs;
  return s;
}

// ---- integer views of FP64 values (no FP64 arithmetic) ----

// FP64 value of float f times 2^k, exactly, by integer operations (a conversion runs on the 1/64-rate
// FP64 pipe); f subnormal and results below the FP64 normal range: 0, above it: Inf
__device__ __forceinline__ double sp_f2d_scaled(float f, int k) {
  const uint32_t b = __float_as_uint(f), m = b & 0x7FFFFFFFu;
  const int e = (int)(m >> 23) + 896 + k;
  uint32_t hi = (m >> 3) + ((uint32_t)(896 + k) << 20), lo = b << 29;
  if (m < 0x00800000u || (unsigned)(e - 1) >= 2046u) {
    hi = m < 0x00800000u || e <= 0 ? 0u : 0x7FF00000u;
    lo = 0u;
  }
  return __hiloint2double((int)(hi | (b & 0x80000000u)), (int)lo);
}

// two FP32 values in one register pair: sums and products of both with one instruction
typedef unsigned long long sp_f2;
__device__ __forceinline__ sp_f2 sp_pack2(uint32_t a, uint32_t b) { return (sp_f2)a | ((sp_f2)b << 32); }
__device__ __forceinline__ sp_f2 sp_add2(sp_f2 a, sp_f2 b) {
  sp_f2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ sp_f2 sp_sub2(sp_f2 a, sp_f2 b) {
  sp_f2 d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ sp_f2 sp_fma2(sp_f2 a, sp_f2 b, sp_f2 c) {
  sp_f2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
// h += a s, its rounding error added to l (both halves), for s = 2^{-7 g}, a an integer of at most 24
// bits and h a multiple of 2^{-7 (g - 1)}, the groups' sums before g.  Fast2Sum (Dekker) without its
// condition |h| >= |a s|: with u = ulp(a s) <= 2^{-7 g}, h is a multiple of u, so where |h| < |a s| the
// sum is a multiple of u below 2^25 u, its error is 0 or u, t - h = a s + error fits 24 bits and both
// subtractions are exact.
__device__ __forceinline__ void sp_accum2(sp_f2& h, sp_f2& l, sp_f2 a, sp_f2 s) {
  const sp_f2 t = sp_fma2(a, s, h), nb = sp_sub2(h, t);  // nb: less what t gained of a s
  l = sp_add2(l, sp_fma2(a, s, nb));
  h = t;
}

// The balanced base-2^7 digits of an integer |X| <= 2^49, X = sum_b d_b 2^{7(G-1-b)}, d_1..d_6 in
// [-64, 63] and |d_0| <= 129, are the 7-bit fields of Y = X + kSpBias less 64 (d_0: the bits above
// them, unbiased): the bias carries into the next field exactly where a digit would leave its
// range, so no digit waits for the one below it.
constexpr long long kSpBias = (1LL << 6) | (1LL << 13) | (1LL << 20) | (1LL << 27) | (1LL << 34) | (1LL << 41);

// X + kSpBias for X = round(mt 2^{e - fe - 4}) (half away from zero) of the FP64 value with these
// bits, fe the largest biased exponent of its column (e <= fe: the shift is at least 4); subnormals
// as 0
__device__ __forceinline__ long long sp_biased(unsigned long long bits, int fe) {
  const int e = (int)(bits >> 52) & 0x7FF;
  const unsigned long long mt = (bits & 0xFFFFFFFFFFFFFULL) | (1ULL << 52);
  const int s1 = e == 0 ? 63 : min(fe + 3 - e, 63);  // shift less one; mt >> 63 is 0, its rounding too
  const unsigned long long r = ((mt >> s1) + 1) >> 1;
  const long long sg = (long long)bits >> 63;
  return ((long long)r ^ sg) - sg + kSpBias;
}

// The BF16 pairs (y0's digit in the low half) of the digits of two biased integers.  A field v in
// 0..127 is the BF16 128 + v with the bits 0x4300 | v, and 128 + v - 192 = v - 64 is exact in BF16:
// three integer instructions and one packed subtraction per pair of digits.  d_0 goes through FP32
// (1.5 2^23 + d_0, whose last bits are d_0): it may need 8 bits.
__device__ __forceinline__ void sp_digit_pairs(long long y0, long long y1, uint32_t (&pk)[kSpG]) {
  const uint32_t l0 = (uint32_t)y0, l1 = (uint32_t)y1;
  const uint32_t m0 = (uint32_t)(y0 >> 21), m1 = (uint32_t)(y1 >> 21);  // fields 3, 4, 5 at bits 0, 7, 14
  const __nv_bfloat162 c = __halves2bfloat162(__ushort_as_bfloat16(0x4340), __ushort_as_bfloat16(0x4340));  // 192
#pragma unroll
  for (int b = 1; b < kSpG; ++b) {
    const int f = kSpG - 1 - b;  // field
    const uint32_t w0 = f < 3 ? l0 >> (7 * f) : m0 >> (7 * (f - 3));
    const uint32_t w1 = f < 3 ? l1 >> (7 * f) : m1 >> (7 * (f - 3));
    uint32_t q = (__byte_perm(w0, w1, 0x5410) & 0x007F007Fu) | 0x43004300u;
    const __nv_bfloat162 d = __hsub2(*reinterpret_cast<__nv_bfloat162*>(&q), c);
    pk[b] = *reinterpret_cast<const uint32_t*>(&d);
  }
  const uint32_t f0 = __float_as_uint(__int_as_float(0x4B400000 + (int)(y0 >> 42)) - 12582912.0f);
  const uint32_t f1 = __float_as_uint(__int_as_float(0x4B400000 + (int)(y1 >> 42)) - 12582912.0f);
  pk[0] = __byte_perm(f0, f1, 0x7632);
}

// S = NX c - x0 - x1 (- x2 - x3), the undivided stencil of FP64 values, in 64-bit fixed point relative to
// the largest of them: each value's significand, `up` bits up, shifted right by its distance from the largest
// exponent, complemented for a negative value.  That stands for the integer and a half, on either side of
// zero: the halves cancel in S (NX against NX of them), so S changes its sign with the values and vanishes
// for equal ones, and a value is off by half a unit at most.  The unit is 2^-up of the largest value's last
// place: S is within NX 2^-59 of that value's power of two (the FP64 subtractions: a few 2^-53), then widened to
// FP64 by one conversion.  |S| < 2^63 units.  Zeros and negligible values shift out.  Outside the middle of
// the exponent range, and for Inf and NaN, the FP64 subtractions themselves.
template <int NX>
__device__ __forceinline__ double sp_stencil(unsigned long long c, const unsigned long long (&x)[NX]) {
  constexpr int up = NX == 4 ? 7 : 8;
  auto ex = [](unsigned long long b) { return (uint32_t)(b >> 32) & 0x7FF00000u; };
  uint32_t q = ex(c);
#pragma unroll
  for (int i = 0; i < NX; ++i) q = max(q, ex(x[i]));
  if (q - (64u << 20) >= (1976u << 20)) {
    auto d = [](unsigned long long b) { return __longlong_as_double((long long)b); };
    const double t = fma((double)NX, d(c), -d(x[0])) - d(x[1]);
    return NX == 4 ? t - (d(x[NX - 2]) + d(x[NX - 1])) : t;
  }
  auto fixed = [&](unsigned long long b, int left) -> long long {
    unsigned long long m = ((b & 0xFFFFFFFFFFFFFULL) | (1ULL << 52)) << left;
    asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"((q - ex(b)) >> 20));  // shifts past 63 give 0
    return (long long)m ^ ((long long)b >> 63);
  };
  long long D = fixed(c, NX == 4 ? up + 2 : up + 1) & ~(NX - 1LL);  // NX times the point's integer
#pragma unroll
  for (int i = 0; i < NX; ++i) D -= fixed(x[i], up);
  const double s = (double)D;  // times 2^{q - 1075 - up}: exponent field added
  const int hi = __double2hiint(s);
  return __hiloint2double(hi == 0 ? 0 : hi + (int)(q - ((1075u + up) << 20)), __double2loint(s));
}

constexpr int kPrepThreads = 256, kPrepM = 32;  // threads along a grid row; time levels per block

// Pre-pass: fe[p] = the largest biased exponent of u at p (zeroed by the launcher), and B = F - A_h u
// written to B -- the defect kernel then subtracts R~ u in place.  The stencil needs FP64 accuracy (at
// N = 4095 it cancels 2^24-fold), but FP64 runs at 1/64 of the FP32 rate: it is formed in integers
// (sp_stencil) and costs a conversion and a multiply-add of that pipe instead of five operations.  A
// thread takes RY points of a column of the grid (their rows are loaded once) and kPrepM time levels.
// Bound by HBM (24 bytes per value) and the issue of ~90 instructions per value; 511^2 x 512: 1.17 ms
// with one thread per grid point and two thirds of the levels in FP64, 0.70 ms now (0.84 with four rows).
template <int DIM, int RY>
__global__ void __launch_bounds__(kPrepThreads) split_prep_kernel(const double* __restrict__ U,
                                                                  const double* __restrict__ F, double* __restrict__ B,
                                                                  int* __restrict__ fe, long long ld, int M, int N,
                                                                  double ih) {
  const int x = blockIdx.x * kPrepThreads + threadIdx.x, y0 = blockIdx.y * RY;
  if (x >= N) return;
  const unsigned long long kl = x > 0 ? ~0ULL : 0ULL, kr = x < N - 1 ? ~0ULL : 0ULL;
  const int ol = x > 0 ? -1 : 0, orr = x < N - 1 ? 1 : 0;
  const int ny = DIM == 2 ? min(RY, N - y0) : 1;
  uint32_t mx[RY];
#pragma unroll
  for (int r = 0; r < RY; ++r) mx[r] = 0;
  const int m1 = min(M, (int)(blockIdx.z + 1) * kPrepM);
  for (int m = blockIdx.z * kPrepM; m < m1; ++m) {
    const long long o = (long long)m * ld + (long long)y0 * N + x;
    const unsigned long long* u = reinterpret_cast<const unsigned long long*>(U) + o;
    unsigned long long c[RY + 2];  // the column: rows y0 - 1 .. y0 + RY
    unsigned long long xl[RY], xr[RY];
    double f[RY];
#pragma unroll
    for (int r = 0; r < RY; ++r) {
      const bool in = r < ny;
      const long long q = (long long)r * N;
      c[r + 1] = in ? __ldg(u + q) : 0ULL;
      xl[r] = in ? __ldg(u + q + ol) & kl : 0ULL;
      xr[r] = in ? __ldg(u + q + orr) & kr : 0ULL;
      f[r] = in ? __ldg(F + o + q) : 0.0;
    }
    if (DIM == 2) {
      c[0] = y0 > 0 ? __ldg(u - N) : 0ULL;
      if (ny == RY) c[RY + 1] = y0 + RY < N ? __ldg(u + (long long)RY * N) : 0ULL;
    }
#pragma unroll
    for (int r = 0; r < RY; ++r) {
      if (r >= ny) break;
      mx[r] = max(mx[r], (uint32_t)(c[r + 1] >> 32) & 0x7FF00000u);
      double S;
      if (DIM == 2) {
        const unsigned long long nb[4] = {xl[r], xr[r], c[r], c[r + 2]};  // rows past the grid hold zeros
        S = sp_stencil<4>(c[r + 1], nb);
      } else {
        const unsigned long long nb[2] = {xl[r], xr[r]};
        S = sp_stencil<2>(c[r + 1], nb);
      }
      B[o + (long long)r * N] = fma(-ih, S, f[r]);
    }
  }
#pragma unroll
  for (int r = 0; r < RY; ++r)
    if (r < ny) atomicMax(fe + (long long)(y0 + r) * N + x, (int)(mx[r] >> 20));
}

// Order of R~'s digits within a block: digit a takes part in 7 - a products, so long and short ones
// alternate (0, 6, 1, 5, ...) and any two successive ring slots are held for about the same time.
__host__ __device__ constexpr int sp_digit_at(int i) { return i & 1 ? kSpG - 1 - i / 2 : i / 2; }

__global__ void __launch_bounds__(kSpBlock, 1) split_defect_kernel(const __grid_constant__ SplitArgs A) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  // the swizzled operand tiles need 1024-byte aligned addresses (the launcher adds 1 KB)
  unsigned char* sm = sm_raw + ((1024u - (smem_u32(sm_raw) & 1023u)) & 1023u);
  const SplitSmem lay = split_smem(A.ns);
  const int ns = A.ns;
  unsigned char* ring = sm + lay.ring;
  unsigned char* xbuf = sm + lay.xbuf;
  float2* const piece = reinterpret_cast<float2*>(sm + lay.piece);
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + lay.bar);
  uint64_t* empty = full + ns;
  uint64_t* xready = empty + ns;  // [2]
  uint64_t* xfree = xready + 2;   // [2]
  uint64_t* accdone = xfree + 2;
  uint64_t* accfree = accdone + 1;
  uint64_t* cbar = accdone + 2;
  uint64_t* exitbar = accdone + 3;
  uint64_t* donebar = accdone + 4;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(accdone + 5);
  volatile int* gfirst_s = abort_flag + 1;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(accdone + 5) + 2;
  int2* pairs = reinterpret_cast<int2*>(sm + lay.pairs);  // digit mask, first tile

  const int t = threadIdx.x;
  const int w = t >> 5;
  const int lane = t & 31;
  const int nI = A.M / kSpRows;
  const int npairs = nI * (nI + 1);

  for (int i = t; i < npairs; i += kSpBlock) {
    const int4 pd = __ldg(A.pairs + i);
    pairs[i] = make_int2(pd.x, pd.y);
  }
  if (t == 0) {
    for (int s = 0; s < ns; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, 1);  // the MMAs' commit
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(xready + b, kSpSplit / 32);
      mbar_init(xfree + b, 1);
    }
    mbar_init(accdone, 2);  // the MMAs' commit + the MMA thread's arrive after publishing the lowest group
    mbar_init(accfree, kSpEpi / 32);
    mbar_init(cbar, kSpEpi / 32);
    mbar_init(exitbar, (kSpSplit + kSpEpi) / 32 + 1);
    mbar_init(donebar, 1);
    *abort_flag = 0;
    *gfirst_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (w == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(kSpTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_before_sync();
  __syncthreads();  // the last block-wide barrier: from here on the roles run apart
  tc_after_sync();
  const uint32_t tmem = *tslot;

  auto raise = [&]() {
    if (!*abort_flag) {
      *abort_flag = 1;
      atomicExch(A.err, 1);
    }
  };

  if (w == (kSpSplit + kSpEpi) / 32) {
    // ---- producer: R~ digit tiles of every pair of every tile of this CTA, in the MMA thread's order
    // (a slot is only ever read by MMAs and written by bulk copies, both of the async proxy) ----
    if (lane != 0) return;
    long long k = 0;
    int slot = 0;
    uint32_t phase = 1;  // of the slot's previous release (the first round finds every slot free)
    bool ok = true, stop = false;
    for (long long g = blockIdx.x; g < A.ntiles && ok && !stop; g += gridDim.x)
      for (int q = 0; q < npairs && ok && !stop; ++q) {
        const int2 pd = pairs[q];
        for (int ia = 0; ia < kSpG; ++ia) {
          const int a = sp_digit_at(ia);
          if (!((pd.x >> a) & 1)) continue;
          if (k + 1 == A.withhold) {
            stop = true;
            break;
          }
          if (!mbar_wait_or_abort(empty + slot, phase, abort_flag)) {
            ok = false;
            break;
          }
          bulk_load(ring + (size_t)slot * kSpAtile, A.At + (size_t)(pd.y + __popc(pd.x & ((1 << a) - 1))) * kSpAtile,
                    kSpAtile, full + slot);
          ++k;
          if (++slot == ns) {
            slot = 0;
            phase ^= 1;
          }
        }
      }
    if (!ok) raise();
    for (int s = 0; s < ns && s < k; ++s) {
      const long long n_s = (k - 1 - s) / ns + 1;
      mbar_wait(full + s, (uint32_t)((n_s - 1) & 1));
    }
    return;
  }

  if (w == (kSpSplit + kSpEpi) / 32 + 1) {
    // ---- MMA warp: every lane runs the loop, so that the descriptors stay in uniform registers; one
    // elected lane issues ----
    {
      const bool leader = umma_elect();
      const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
      // descriptors: K-major, 128-byte swizzle; a K step of 16 adds 2 to the address field
      const uint64_t dbase = sw128_desc(0);
      const uint32_t ring16 = smem_u32(ring) >> 4, xbuf16 = smem_u32(xbuf) >> 4;
      int slot = 0;
      uint32_t fphase = 0, accphase = 1, xphase = 0;  // accfree: the first block finds tensor memory free
      int b = 0;
      bool failed = false;
      // ng u digits from digit b0 on times the R~ digit in the slot, into the groups from g0 on
      auto mma = [&](uint32_t bbuf16, int g0, int b0, int ng, bool fresh) {
        const uint64_t ad = dbase | (uint64_t)(ring16 + (uint32_t)slot * (kSpAtile >> 4));
        const uint64_t bd = dbase | (uint64_t)(bbuf16 + (uint32_t)b0 * (kSpBtile >> 4));
        const uint32_t idesc = umma_idesc(ng * kSpCols), d = tm + 64u * g0;
#pragma unroll
        for (int st = 0; st < kSpK / 16; ++st)
          asm volatile(
              "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
              " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
              "l"(ad + 2ULL * st), "l"(bd + 2ULL * st), "r"(idesc), "r"(st > 0 || !fresh ? 1u : 0u)
              : "memory");
      };
      auto slot_full = [&]() -> bool {
        if (!__all_sync(0xffffffffu, mbar_wait_or_abort(full + slot, fphase, abort_flag, A.spin))) return false;
        tc_after_sync();
        return true;
      };
      auto slot_done = [&]() {
        if (leader) umma_commit(empty + slot);
        if (++slot == ns) {
          slot = 0;
          fphase ^= 1;
        }
      };
      for (long long g = blockIdx.x; g < A.ntiles && !failed; g += gridDim.x)
        for (int I = 0; I < nI && !failed; ++I) {
          if (!__all_sync(0xffffffffu, mbar_wait_or_abort(accfree, accphase, abort_flag, A.spin))) {
            failed = true;
            break;
          }
          accphase ^= 1;
          int gfirst = kSpG;  // lowest group this block has written
          for (int J = 0; J <= 2 * I + 1 && !failed; ++J) {
            const int mask = pairs[I * (I + 1) + J].x;
            const uint32_t bbuf16 = xbuf16 + (uint32_t)b * (kSpG * kSpBtile >> 4);
            if (!__all_sync(0xffffffffu, mbar_wait_or_abort(xready + b, xphase, abort_flag, A.spin))) {
              failed = true;
              break;
            }
            tc_after_sync();
            // R~ digit a meets the u digits 0..6-a in the groups a..6: their tiles are consecutive in
            // shared memory and the groups in tensor memory, so one MMA covers up to four of them
            // (N = 256).  A 128 x 64 x 16 MMA is bound by its operand reads (48 cycles for 32 of tensor
            // work) and by its issue (95 cycles seen); ten wide ones replace 28 per K step: the defect
            // of a 511^2 x 512 grid, pre-pass included, 6.47 -> 5.41 ms.
            if (gfirst == 0) {
              // every group is written already: all MMAs accumulate, shapes known at compile time
#pragma unroll
              for (int ia = 0; ia < kSpG; ++ia) {
                const int a = sp_digit_at(ia);
                if (!((mask >> a) & 1)) continue;
                if (!slot_full()) {
                  failed = true;
                  break;
                }
                if (leader) {
                  mma(bbuf16, a, 0, a < 3 ? 4 : kSpG - a, false);
                  if (a < 3) mma(bbuf16, a + 4, 4, 3 - a, false);
                }
                slot_done();
              }
            } else {
              // the groups written so far are a suffix gfirst..6, which is accumulated into; the
              // groups a..gfirst-1 are written afresh
#pragma unroll 1
              for (int ia = 0; ia < kSpG; ++ia) {
                const int a = sp_digit_at(ia);
                if (!((mask >> a) & 1)) continue;
                if (!slot_full()) {
                  failed = true;
                  break;
                }
                for (int g0 = a; g0 < kSpG;) {
                  const bool fresh = g0 < gfirst;
                  const int ng = min(fresh ? gfirst - g0 : kSpG - g0, 4);
                  if (leader) mma(bbuf16, g0, g0 - a, ng, fresh);
                  g0 += ng;
                }
                gfirst = min(gfirst, a);
                slot_done();
              }
            }
            if (failed) break;
            if (leader) umma_commit(xfree + b);
            b ^= 1;
            xphase ^= b ^ 1;
          }
          if (failed) break;
          if (leader) {
            *gfirst_s = gfirst;
            umma_commit(accdone);
            mbar_arrive(accdone);  // release: the lowest group is visible to the epilogue after its wait
          }
        }
      if (leader) {
        if (failed) raise();
        umma_commit(donebar);  // completes when every MMA issued above has completed
      }
    }
    __syncwarp();
    tc_before_sync();
    if (lane == 0) mbar_arrive(exitbar);
    return;
  }

  // ---- split and epilogue warps ----
  bool failed = false;
  auto give_up = [&](bool ok) -> bool {
    if (__all_sync(0xffffffffu, ok)) return false;
    if (lane == 0) raise();
    return true;
  };
  const long long ld = A.ld;

  if (w < kSpSplit / 32) {
    // ---- split: thread t owns point n = t & 63 of the tile and 16 time levels (t >> 6) * 16 .. of a
    // K-block; the next block's values are loaded into registers once this one's digits are published
    const int sn = t & 63, sk = (t >> 6) * 16;
    const unsigned long long* Ub = reinterpret_cast<const unsigned long long*>(A.U);
    unsigned long long v[16];
    int fe = 0;
    auto load16 = [&](long long g, int J) {
      const long long p = g * kSpCols + sn;
      const bool ok = p < ld;
      const unsigned long long* src = Ub + (long long)(J * kSpK + sk) * ld + (ok ? p : 0);
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] = ok ? __ldg(src + (long long)j * ld) : 0ULL;
      if (J == 0) fe = ok ? __ldg(A.fe + p) : 0;
    };
    // L2 prefetch of 128 time rows from row m0 on of tile g of u (two lines per thread)
    auto prefetch_u = [&](long long g, int m0) {
      const unsigned long long* row = Ub + (long long)(m0 + (t >> 1)) * ld;
      const long long p = g * kSpCols + (t & 1) * 32;
      asm volatile("prefetch.global.L2 [%0];" ::"l"(row + min(p, ld - 1)));
      asm volatile("prefetch.global.L2 [%0];" ::"l"(row + min(p + 16, ld - 1)));
    };
    long long q = 0;
    load16(blockIdx.x, 0);
    for (long long g = blockIdx.x; g < A.ntiles && !failed; g += gridDim.x)
      for (int I = 0; I < nI && !failed; ++I)
        for (int J = 0; J <= 2 * I + 1; ++J, ++q) {
          const int b = (int)(q & 1);
          if (q >= 2 && give_up(mbar_wait_or_abort(xfree + b, (uint32_t)(((q >> 1) - 1) & 1), abort_flag, A.spin))) {
            failed = true;
            break;
          }
          unsigned char* xb = xbuf + (size_t)b * kSpG * kSpBtile;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            uint32_t pk[4][kSpG];
#pragma unroll
            for (int j = 0; j < 4; ++j)
              sp_digit_pairs(sp_biased(v[8 * h + 2 * j], fe), sp_biased(v[8 * h + 2 * j + 1], fe), pk[j]);
#pragma unroll
            for (int a = 0; a < kSpG; ++a)
              *reinterpret_cast<uint4*>(xb + (size_t)a * kSpBtile + sw128_off(sn, sk + 8 * h)) =
                  make_uint4(pk[0][a], pk[1][a], pk[2][a], pk[3][a]);
          }
          async_proxy_fence();
          __syncwarp();
          if (lane == 0) mbar_arrive(xready + b);
          // the next block's loads only now: the proxy fence waits for this thread's outstanding
          // memory operations.  K-blocks 2 I + 2, 2 I + 3 (the next tile's 0, 1) are new to this CTA
          // when block I is done: their lines are fetched into L2 meanwhile
          if (J == 0) {
            if (I + 1 < nI)
              prefetch_u(g, 2 * (I + 1) * kSpK);
            else if (g + gridDim.x < A.ntiles)
              prefetch_u(g + gridDim.x, 0);
          }
          const int Jn = J < 2 * I + 1 ? J + 1 : 0;
          const long long gn = Jn == 0 && I + 1 == nI ? g + gridDim.x : g;
          if (gn < A.ntiles) load16(gn, Jn);
        }
  } else {
    // ---- epilogue: r = B - R~ u for a block of 128 time rows x 64 points, B = F - A_h u from the
    // pre-pass (in OUT).  Drain: thread (lane quarter wq: 32 time rows; ch: column half of each 32
    // points) folds the seven groups into double-float sums, points 0..31 straight into the piece,
    // points 32..63 kept in registers, and releases tensor memory, so that the next block's MMAs
    // run during the rest.  Write-back, 32 points at a time: transposed through the piece, thread
    // per grid point, so that every global access runs along a row.
    const int e = t - kSpSplit, ew = e >> 5;
    const int wq = ew & 3, ch = ew >> 2;
    const uint32_t lane_base = (uint32_t)(32 * wq) << 16;
    uint32_t cbphase = 0;
    auto meet = [&]() -> bool {  // all epilogue warps (bounded)
      __syncwarp();
      if (lane == 0) mbar_arrive(cbar);
      const bool ok = mbar_wait_or_abort(cbar, cbphase, abort_flag, A.spin);
      cbphase ^= 1;
      return !give_up(ok);
    };
    unsigned long long nmax = 0;
    float2* const mine = piece + (size_t)(ch * 16) * kSpPieceLd + wq * 32 + lane;
    // the double-float sums of this thread's time row at points pbase + 8 c8 + 0..7
    auto fold8 = [&](uint32_t col, int gfirst, sp_f2 (&h)[4], sp_f2 (&l)[4]) {
      uint32_t r[kSpG][8];
#pragma unroll
      for (int gg = 0; gg < kSpG; ++gg)
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
            : "=r"(r[gg][0]), "=r"(r[gg][1]), "=r"(r[gg][2]), "=r"(r[gg][3]), "=r"(r[gg][4]), "=r"(r[gg][5]),
              "=r"(r[gg][6]), "=r"(r[gg][7])
            : "r"(tmem + lane_base + 64u * gg + col));
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      // the loaded registers are read only after the wait
#pragma unroll
      for (int gg = 0; gg < kSpG; ++gg) {
        asm volatile("" : "+r"(r[gg][0]), "+r"(r[gg][1]), "+r"(r[gg][2]), "+r"(r[gg][3]), "+r"(r[gg][4]),
                     "+r"(r[gg][5]), "+r"(r[gg][6]), "+r"(r[gg][7]));
        if (gg < gfirst) {  // a group no MMA wrote (none of R~'s digits a <= gg in the block)
#pragma unroll
          for (int j = 0; j < 8; ++j) r[gg][j] = 0;
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        h[j] = sp_pack2(r[0][2 * j], r[0][2 * j + 1]);
        l[j] = 0;
#pragma unroll
        for (int gg = 1; gg < kSpG; ++gg) {
          const uint32_t sc = __float_as_uint(1.f / (float)(1ULL << (7 * gg)));
          sp_accum2(h[j], l[j], sp_pack2(r[gg][2 * j], r[gg][2 * j + 1]), sp_pack2(sc, sc));
        }
      }
    };
    auto put8 = [&](int c8, const sp_f2 (&h)[4], const sp_f2 (&l)[4]) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        mine[(size_t)(c8 * 8 + 2 * j) * kSpPieceLd] =
            make_float2(__uint_as_float((uint32_t)h[j]), __uint_as_float((uint32_t)l[j]));
        mine[(size_t)(c8 * 8 + 2 * j + 1) * kSpPieceLd] =
            make_float2(__uint_as_float((uint32_t)(h[j] >> 32)), __uint_as_float((uint32_t)(l[j] >> 32)));
      }
    };
    // write-back of the piece: thread = point p, time rows m0 .. m0 + 15
    auto write16 = [&](long long p, int fe, int m0) {
      const float2* const pc = piece + (size_t)lane * kSpPieceLd + ew * 16;
      const bool ok = p < ld;
      double* const out = A.OUT + (long long)m0 * ld + (ok ? p : 0);
      double bv[16];
#pragma unroll
      for (int rr = 0; rr < 16; ++rr) bv[rr] = __ldcg(out + (long long)rr * ld);
#pragma unroll
      for (int rr = 0; rr < 16; ++rr) {
        const float2 P = pc[rr];
        const int k = __ldg(A.rexp + m0 + rr) + fe - 1036;  // (R~ u)_{m,c} = 2^{E_m + F_c - 14} P, F_c = fe - 1022
        double r = (bv[rr] - sp_f2d_scaled(P.x, k)) - sp_f2d_scaled(P.y, k);
        if (fe == 2047) r = __longlong_as_double(0x7FF8000000000000LL);  // an Inf or NaN in u at the point
        if (ok) {
          out[(long long)rr * ld] = r;
          const unsigned long long ab = (unsigned long long)__double_as_longlong(r) & 0x7FFFFFFFFFFFFFFFULL;
          nmax = ab > nmax ? ab : nmax;
        }
      }
    };
    long long nblk = 0;
    for (long long g = blockIdx.x; g < A.ntiles && !failed; g += gridDim.x) {
      const long long p = g * kSpCols + lane;
      const int fe0 = p < ld ? __ldg(A.fe + p) : 0, fe1 = p + 32 < ld ? __ldg(A.fe + p + 32) : 0;
      for (int I = 0; I < nI; ++I, ++nblk) {
        {  // L2 prefetch of the rows of B that this block's write-back reads, two lines per thread
          const double* row = A.OUT + (long long)(I * kSpRows + (e >> 1)) * ld;
          const long long pb = g * kSpCols + (e & 1) * 32;
          asm volatile("prefetch.global.L2 [%0];" ::"l"(row + min(pb, ld - 1)));
          asm volatile("prefetch.global.L2 [%0];" ::"l"(row + min(pb + 16, ld - 1)));
        }
        if (give_up(mbar_wait_or_abort(accdone, (uint32_t)(nblk & 1), abort_flag, A.spin))) {
          failed = true;
          break;
        }
        tc_after_sync();
        const int gfirst = *gfirst_s;
        sp_f2 h[2][4], l[2][4];
#pragma unroll
        for (int c8 = 0; c8 < 2; ++c8) {
          fold8(ch * 16 + c8 * 8, gfirst, h[0], l[0]);
          put8(c8, h[0], l[0]);
        }
#pragma unroll
        for (int c8 = 0; c8 < 2; ++c8) fold8(32 + ch * 16 + c8 * 8, gfirst, h[c8], l[c8]);
        tc_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(accfree);  // this warp is done with the block's accumulators
        const int m0 = I * kSpRows + ew * 16;
        if (!meet()) {  // points 0..31 are in the piece
          failed = true;
          break;
        }
        write16(p, fe0, m0);
        if (!meet()) {  // every thread is done with them
          failed = true;
          break;
        }
#pragma unroll
        for (int c8 = 0; c8 < 2; ++c8) put8(c8, h[c8], l[c8]);
        if (!meet()) {
          failed = true;
          break;
        }
        write16(p + 32, fe1, m0);
        if (!meet()) {  // every thread is done with the piece
          failed = true;
          break;
        }
      }
    }
    if (A.norm != nullptr && !failed) {
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long other = __shfl_xor_sync(0xffffffffu, nmax, o);
        nmax = other > nmax ? other : nmax;
      }
      if (lane == 0) atomicMax(A.norm, nmax);
    }
  }
  // exit: every split and epilogue warp and the MMA warp arrive (bounded waits everywhere, so all do), the
  // MMA thread's last commit signals that every issued MMA completed, then warp 0 frees TMEM
  tc_before_sync();
  __syncwarp();
  if (lane == 0) mbar_arrive(exitbar);
  if (w == 0) {
    mbar_wait(exitbar, 0);
    mbar_wait(donebar, 0);
    tc_after_sync();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kSpTmemCols));
  }
}

}  // namespace fhmg
