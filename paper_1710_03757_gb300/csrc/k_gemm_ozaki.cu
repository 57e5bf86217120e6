// K5 at FP64 accuracy on the tensor cores: the plaquette GEMM M = X Yt^T by
// error-free splitting (Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59,
// 2012), with FP16 digits multiplied exactly by tcgen05.mma.
//
// Digits: with e the exponent of a row's largest magnitude (every |x| < 2^e,
// k_ozaki_expo) and P = (b-1) + b(s-1) = 55, the integer F = round(x 2^{P-e})
// (|F| <= 2^P) is recoded into signed digits from the bottom,
// a_i = ((F + 2^{b-1}) mod 2^b) - 2^{b-1}, F <- (F - a_i) / 2^b, the top digit
// taking the rest, so x = 2^e sum_i a_i 2^{-(b-1)-b i} + r with
// |r| <= 2^{e-P-1}, |a_i| <= 2^{b-1} (b <= 8 bits: exact in FP16).  Adding
// 2^{b-1} at every digit's place turns all the carries into one addition: the
// fields of G = F + sum_i 2^{b-1} 2^{b i} are the digits plus 2^{b-1}, and a
// field under the exponent bits of 1024 is the FP16 number 1024 + field.  Only
// integer and FP16 operations per element: FP64 issues at 1/64 of the FP32
// rate on this GPU.
//
// Product: x y = 2^{e_x + e_y} sum_{i,j} A_i B_j.  All products of one group
// g = i + j carry the same weight, and their sum over K is an integer multiple
// of it bounded by m K 2^{2b-2} for m pairs; with b = 8 for K <= 256 and b = 7
// for K <= 1024 the groups of up to four pairs stay at or below 2^24, so their
// FP32 accumulation is exact, and the larger later groups round below 2^-53 of
// the leading one.  Groups g <= s-1 are kept (s(s+1)/2 digit products; s = 7
// for b = 8, s = 8 for b = 7, i.e. 55 bits of each operand): the dropped groups
// and residuals are below 2^-43 K-relative of |row max| |column max|, the order
// of an FP64 dot product's own error.
//
// k_gemm_ozaki: one CTA per SM over 128 x 64 output tiles.  Tensor memory holds
// one 128 x 64 FP32 accumulator per group, side by side.
//   warps 0-11   read 16 rows each of X (8 warps) and Yt (4) for one k-step of
//                16, form the digits and write them to shared memory, so no
//                digit plane exists in global memory;
//   warp 20      issues the k-step's products: slice i of A times the slices
//                0 .. s-1-i of B, whose rows lie below one another, is one MMA of
//                N = 64 (s - i) columns (two above 256) that adds to the
//                groups i .. s-1: 10 (12 at s = 8) MMAs and as many reads of
//                an A slice where one per digit product took 28 (36);
//   warps 12-19  read the groups of a finished tile, add them up in 64-bit
//                integers, round once to FP64 by integer operations and write M
//                matricized for the next level, while the first k-steps of the
//                next tile are split.
// Bound by the splitting (the ALU pipe): a tile's tensor products take some 15
// thousand of the ~50 thousand clocks; a tile of A is split anew for each of the
// column tiles, which costs less than digit planes in global memory did (14
// bytes written per element, and 28 x 24 KB of them read for a K slice of 64
// that is 96 KB in FP64): 512 products of n = K = 256, the whole call, 3.15 ->
// 0.99 ms; 32 of n = K = 576 2.02 -> 0.82, 2048 of n = K = 64 1.09 -> 0.37.
// Every mbarrier wait is bounded; on expiry the roles leave their loops, the
// kernel records an error word, waits (bounded) for its products in flight and
// frees its tensor memory.
#include <cuda_fp16.h>

#include <algorithm>
#include <cstdint>

#include "common.cuh"
#include "kernels_tc.h"
#include "tc_ptx.cuh"

namespace mctrg {

using namespace tcptx;

namespace {
constexpr int kOzTileM = 128;    // output rows per tile (tensor-memory lanes)
constexpr int kOzTileN = 64;     // output columns per tile and per accumulator
constexpr int kOzSplitWarps = 12, kOzEpiWarps = 8;
constexpr int kOzThreads = 32 * (kOzSplitWarps + kOzEpiWarps + 1);
constexpr int kOzStages = 3;     // k-steps of A in flight; B in two buffers of four k-steps
constexpr uint32_t kOzAHalf = kOzTileM * 128u, kOzABytes = 2 * kOzAHalf;

__host__ __device__ constexpr uint32_t oz_b_bytes(int slices) { return (uint32_t)slices * kOzTileN * 128u; }
constexpr size_t oz_smem(int slices) { return kOzStages * kOzABytes + 2 * oz_b_bytes(slices) + 1024; }

// Byte offset of the 16-byte piece (8 K values, half kh of the k-step) of slice
// s, row rho of A: two tiles of 128 rows x 128 bytes, four slices side by side,
// in the 128-byte swizzle; and of slice s, row j of B: rows 64 s + j of 128
// bytes, four k-steps (slots) side by side.
__device__ __forceinline__ uint32_t oz_a_piece(int s, int rho, int kh) {
  return (uint32_t)((s >> 2) * kOzAHalf + rho * 128 + (((((s & 3) << 1) | kh) ^ (rho & 7)) << 4));
}
__device__ __forceinline__ uint32_t oz_b_piece(int s, int j, int slot, int kh) {
  return (uint32_t)((s * kOzTileN + j) * 128 + ((((slot << 1) | kh) ^ (j & 7)) << 4));
}
}  // namespace

bool gemm_ozaki_supported(int n, int K) { return n >= 1 && K >= 64 && K % 64 == 0 && K <= 1024; }

// Row exponents, one warp per row: e with max = f 2^e, f in [0.5, 1).
__global__ void __launch_bounds__(256) k_ozaki_expo(const double* X, const double* Y, int64_t rows, int K, int* expo) {
  const int lane = threadIdx.x & 31;
  int64_t row = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (row >= 2 * rows) return;
  const double* x = row < rows ? X + row * K : Y + (row - rows) * K;
  // the bit patterns of non-negative doubles order like their values
  long long mb = 0;
  for (int k = lane; k < K; k += 64) {               // K is a multiple of 64
    mb = max(mb, __double_as_longlong(x[k]) & 0x7FFFFFFFFFFFFFFFll);
    mb = max(mb, __double_as_longlong(x[k + 32]) & 0x7FFFFFFFFFFFFFFFll);
  }
  for (int o = 16; o > 0; o >>= 1) mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, o));
  int e = (int)(mb >> 52) - 1022;
  if ((mb >> 52) == 0) {
    e = 0;
    if (mb != 0) frexp(__longlong_as_double(mb), &e);   // subnormal largest value
  }
  if (lane == 0) expo[row] = e;
}

namespace {
constexpr int kOzP = 55;                             // fraction bits kept

// G = F + sum_i 2^{b-1} 2^{b i}, F = round(x 2^{P-e}) with halves away from
// zero.  x = q 2^{E-52} with q the 53-bit significand, so |F| = q 2^{sh},
// sh = max(be, 1) - 1075 + P - e <= 2 for a row whose e is that of a normal
// number.  With T = q 2^3 >> (2 - sh), |F| = (T + 1) >> 1, and the sign comes in
// as the complement: F = (1 + T) >> 1 or (1 + ~T) >> 1.
template <int BITS, int S>
__device__ __forceinline__ unsigned long long oz_fixed(double x, int e) {
  unsigned long long bias = 0;
#pragma unroll
  for (int i = 0; i < S; ++i) bias |= (1ull << (BITS - 1)) << (BITS * i);
  const int hi = __double2hiint(x), be = (hi & 0x7fffffff) >> 20;
  const unsigned mh = ((unsigned)hi & 0xFFFFFu);
  unsigned long long t;
  if (e >= -900) {
    // (subnormal elements are shifted out, with or without the leading bit)
    const unsigned long long q = ((unsigned long long)(mh | 0x100000u) << 32) | (unsigned)__double2loint(x);
    t = (q << 3) >> min(1077 - kOzP + e - be, 63);
  } else {
    const unsigned long long q = ((unsigned long long)(mh | (be ? 0x100000u : 0u)) << 32) | (unsigned)__double2loint(x);
    const int back = 1077 - kOzP + e - max(be, 1);
    // rows of subnormal numbers: q is as short as the shift is long
    t = back >= 0 ? (q << 3) >> min(back, 63) : (q << 3) << -back;
  }
  const unsigned sg = (unsigned)(hi >> 31);
  return ((((unsigned long long)((unsigned)(t >> 32) ^ sg) << 32) | ((unsigned)t ^ sg)) + (2 * bias + 1)) >> 1;
}

// The digits of two consecutive K values, given by their G, as pairs of FP16, top slice first.
template <int BITS, int S>
__device__ __forceinline__ void oz_digits(unsigned long long y0, unsigned long long y1, uint32_t (&out)[S]) {
  uint32_t d[S];
  if constexpr (BITS == 8) {
    // the top field is 9 bits wide (a value that rounds up to 2^e)
    const uint32_t h0 = (uint32_t)(y0 >> 32), h1 = (uint32_t)(y1 >> 32), l0 = (uint32_t)y0, l1 = (uint32_t)y1;
    d[0] = __byte_perm(h0, h1, 0x7632) | 0x64006400u;
    const uint32_t b = __byte_perm(h0, h1, 0x5410), c = __byte_perm(l0, l1, 0x7632), f = __byte_perm(l0, l1, 0x5410);
    d[1] = __byte_perm(b, 0x64646464u, 0x4341);
    d[2] = __byte_perm(b, 0x64646464u, 0x4240);
    d[3] = __byte_perm(c, 0x64646464u, 0x4341);
    d[4] = __byte_perm(c, 0x64646464u, 0x4240);
    d[5] = __byte_perm(f, 0x64646464u, 0x4341);
    d[6] = __byte_perm(f, 0x64646464u, 0x4240);
  } else {
#pragma unroll
    for (int i = 0; i < S; ++i) {
      const int sh = BITS * (S - 1 - i);
      const uint32_t m = i == 0 ? 0xffu : (1u << BITS) - 1;
      const uint32_t f0 = (uint32_t)(y0 >> sh) & m, f1 = (uint32_t)(y1 >> sh) & m;
      d[i] = (f1 << 16) | f0 | 0x64006400u;
    }
  }
  const uint16_t o16 = (uint16_t)(0x6400 + (1 << (BITS - 1)));   // 1024 + 2^{b-1}
  const __half2 off = __halves2half2(__ushort_as_half(o16), __ushort_as_half(o16));
#pragma unroll
  for (int i = 0; i < S; ++i) {
    const __half2 v = __hsub2(*reinterpret_cast<const __half2*>(&d[i]), off);
    out[i] = *reinterpret_cast<const uint32_t*>(&v);
  }
}

__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}

// (hi 2^sh + lo) 2^p rounded once to FP64 (to nearest, ties to even) by integer
// operations (two conversions and two products on the FP64 pipe take 64 clocks
// of it per warp, as long as a tile's tensor products); sh <= 28, |hi| + |lo| < 2^62.
__device__ __forceinline__ double oz_round(long long hi, long long lo, int sh, int p) {
  if ((hi | lo) == 0) return 0.0;
  // hi 2^sh + lo = t 2^sh + r, 0 <= r < 2^sh; its magnitude likewise
  const unsigned mask = (1u << sh) - 1;
  long long t = hi + (lo >> sh);
  unsigned r = (unsigned)lo & mask;
  const bool neg = t < 0;
  if (neg) {
    t = -t - (r != 0);
    r = (0u - r) & mask;
  }
  if (t == 0 && r == 0) return 0.0;
  // significand of 64 bits: t from the top, then r, then whether anything fell off
  const unsigned long long rr = (unsigned long long)r << (64 - sh);
  int lz = __clzll(t);
  unsigned long long m;
  unsigned lost = 0;
  if (t != 0) {                                      // 1 <= lz <= 63
    m = ((unsigned long long)t << lz) | (rr >> (64 - lz));
    lost = (rr << lz) != 0;
  } else {
    const int z = __clzll((long long)rr);
    m = rr << z;
    lz = 64 + z;
  }
  int ex = 1023 + 63 - lz + sh + p;                  // biased exponent of the leading bit
  if (ex < 1) {                                      // subnormal: the significand moves down
    const int d = min(1 - ex, 63);
    lost |= (m << (64 - d)) != 0;
    m >>= d;
    ex = 1;
  }
  if (ex > 2046) return __longlong_as_double(neg ? 0xfff0000000000000ll : 0x7ff0000000000000ll);
  const unsigned tail = ((unsigned)m & 0x7ffu) | lost;
  const unsigned long long mant = m >> 11;
  const unsigned up = tail > 0x400u || (tail == 0x400u && ((unsigned)mant & 1u));
  const unsigned long long bits = ((unsigned long long)(ex - 1) << 52) + mant + up;
  return __longlong_as_double((long long)(bits | (neg ? 0x8000000000000000ull : 0ull)));
}

__device__ __forceinline__ void tmem_ld_16x8(uint32_t taddr, uint32_t (&v)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"(taddr));
}
struct OzRing {
  uint64_t *full, *empty_a, *empty_b;
  volatile int* fail;
};

// A warp's part of the splitting: 16 rows of X (from row0 of the tile) or Yt.
// Lane 8 q + kp has the K values 2 kp and 2 kp + 1 of the rows 2 q + (0, 1, 8, 9):
// eight lanes read a row's 128 bytes, and the four rows that a warp stores at
// a time lie in different banks.  The loads of a k-step are issued before the
// digits of the one before it, also across tiles.
template <int BITS, int S, bool IS_B>
__device__ __forceinline__ void oz_split(const GemmOzArgs& a, int64_t tiles, const OzRing& ring, uint8_t* buf, int row0) {
  const int n = a.n, K = a.K, steps = K / 16;
  const int nts = (n + kOzTileN - 1) / kOzTileN, per = (n + kOzTileM - 1) / kOzTileM * nts;
  const int lane = threadIdx.x & 31, kp = lane & 7, q = lane >> 3, kh = kp >> 2;
  row0 += 2 * q;
  const double* src = IS_B ? a.Y : a.X;
  const int* expo = IS_B ? a.expY : a.expX;
  double2 v[4], next[4];
  const double* x = nullptr;                         // this lane's first row of the tile that is being read
  int e[4], en[4], left = 0;                         // exponents (and the next tile's); rows from x to the end
  auto open_tile = [&](int64_t t) {
    const int64_t it = t / per;
    const int w = (int)(t - it * per);
    const int r = (IS_B ? (w % nts) * kOzTileN : (w / nts) * kOzTileM) + row0;
    left = n - r;
    const int64_t g = it * n + r;
    x = src + g * K + 2 * kp;
#pragma unroll
    for (int p = 0; p < 4; ++p) en[p] = (p & 1) + 8 * (p >> 1) < left ? expo[g + (p & 1) + 8 * (p >> 1)] : 0;
  };
  auto load = [&]() {                                // the next k-step's values, which x points at
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const int row = (p & 1) + 8 * (p >> 1);
      const double* y = x + row * K;
      if (row >= left) next[p] = make_double2(0.0, 0.0);
      else if (a.aligned) next[p] = __ldg((const double2*)y);
      else next[p] = make_double2(__ldg(y), __ldg(y + 1));
    }
    x += 16;
  };
  int st = 0, ast = 0, aph = 1;                      // k-step, stage of A and the parity of its last release
  open_tile(blockIdx.x);
  load();
  for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
#pragma unroll
    for (int p = 0; p < 4; ++p) e[p] = en[p];
#pragma unroll 1
    for (int k = 0; k < steps; ++k) {
#pragma unroll
      for (int p = 0; p < 4; ++p) v[p] = next[p];
      if (k + 1 == steps && tile + gridDim.x < tiles) open_tile(tile + gridDim.x);
      if (k + 1 < steps || tile + gridDim.x < tiles) load();
      bool ok = st < kOzStages || mbar_wait(&ring.empty_a[ast], aph);
      const int grp = st >> 2, slot = st & 3;
      if (IS_B && slot == 0 && grp >= 2) ok = ok && mbar_wait(&ring.empty_b[grp & 1], ((grp >> 1) - 1) & 1);
      if (!__all_sync(0xffffffffu, ok && !*ring.fail)) {   // the warp leaves together
        *ring.fail = 1;
        return;
      }
      uint8_t* dst = buf + (IS_B ? (grp & 1) * oz_b_bytes(S) : ast * kOzABytes) + (kp & 3) * 4;
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        // row0 = 2 q mod 8, so the swizzled piece is found once for rows 8 apart
        const int rho = row0 + (p & 1);
        uint32_t d[S];
        oz_digits<BITS, S>(oz_fixed<BITS, S>(v[p].x, e[p]), oz_fixed<BITS, S>(v[p].y, e[p]), d);
#pragma unroll
        for (int s = 0; s < S; ++s) {
          const uint32_t piece = IS_B ? oz_b_piece(0, rho, slot, kh) : oz_a_piece(s & 3, rho, kh);
          const uint32_t rest = (p >> 1) * 1024u + (IS_B ? (uint32_t)s * kOzTileN * 128u : (uint32_t)(s >> 2) * kOzAHalf);
          *(uint32_t*)(dst + piece + rest) = d[s];
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&ring.full[ast]);
      if (++ast == kOzStages) { ast = 0; aph ^= 1; }
      ++st;
    }
  }
}
}  // namespace

// ---------------------------------------------------------------------------
template <int BITS, int S>
__global__ void __launch_bounds__(kOzThreads, 1) k_gemm_ozaki(GemmOzArgs a, int64_t tiles) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* As = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* Bs = As + kOzStages * kOzABytes;
  __shared__ __align__(8) uint64_t full_bar[kOzStages], empty_a[kOzStages], empty_b[2], acc_full, acc_empty, done_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_fail;
  __shared__ short s_exp[kOzEpiWarps][64];           // exponents of a warp's 32 rows and 32 columns
  const int n = a.n, K = a.K, steps = K / 16;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int mts = (n + kOzTileM - 1) / kOzTileM, nts = (n + kOzTileN - 1) / kOzTileN, per = mts * nts;

  if (threadIdx.x == 0) {
    s_fail = 0;
    for (int s = 0; s < kOzStages; ++s) { mbar_init(&full_bar[s], kOzSplitWarps); mbar_init(&empty_a[s], 1); }
    mbar_init(&empty_b[0], 1);
    mbar_init(&empty_b[1], 1);
    mbar_init(&acc_full, 1);
    mbar_init(&acc_empty, kOzEpiWarps);
    mbar_init(&done_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(&tmem_slot)), "r"(512u));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  if (warp < kOzSplitWarps) {
    OzRing ring{full_bar, empty_a, empty_b, &s_fail};
    if (warp < 8) oz_split<BITS, S, false>(a, tiles, ring, As, warp * 16);
    else oz_split<BITS, S, true>(a, tiles, ring, Bs, (warp - 8) * 16);
  } else if (warp < kOzSplitWarps + kOzEpiWarps) {
    // warp w reads the tensor-memory lanes 32 (w mod 4) .. and half of the columns
    const int quad = warp & 3, half = (warp - kOzSplitWarps) >> 2;
    const int w0 = 2 * (BITS - 1);                    // weight exponent of group 0
    const int D = a.D;
    uint32_t ph = 0;
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x, ph ^= 1) {
      const int64_t it = tile / per;
      const int w = (int)(tile - it * per);
      const int rw = (w / nts) * kOzTileM + quad * 32, cw = (w % nts) * kOzTileN + half * 32;
      const int r0 = rw + (lane >> 2), c0 = cw + 2 * (lane & 3);
      short* sx = s_exp[warp - kOzSplitWarps];
      __syncwarp();
      sx[lane] = rw + lane < n ? (short)(a.expX[it * n + rw + lane] - w0 - BITS * (S - 1)) : (short)0;
      sx[32 + lane] = cw + lane < n ? (short)a.expY[it * n + cw + lane] : (short)0;
      __syncwarp();
      int par = a.fixed_parity;
      if (par < 0) par = tensor_parity(a.L, a.level_new, (a.c0 + it) % a.Nnew);
      double* Mo = a.M + it * n * n;
      const bool wide = a.wide && par == 0;
      if (!__all_sync(0xffffffffu, mbar_wait(&acc_full, ph) && !s_fail)) { s_fail = 1; break; }
      tc_fence_after();
#pragma unroll 1
      for (int q = 0; q < 8; ++q) {                   // 16 rows x 8 columns each
        const int rh = q & 1, c8 = q >> 1;
        __syncwarp();
        uint32_t v[S][4];
#pragma unroll
        for (int g = 0; g < S; ++g)
          tmem_ld_16x8(tmem + ((uint32_t)(quad * 32 + rh * 16) << 16) + (uint32_t)(g * kOzTileN + half * 32 + c8 * 8), v[g]);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (q == 7) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acc_empty);
        }
        const int cc = c0 + c8 * 8;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int r = r0 + rh * 16 + h * 8;
          if (r >= n) continue;
          const int er = sx[rh * 16 + h * 8 + (lane >> 2)];
          double o[2];
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            // the groups are integers (exact below 2^24; the later ones at most
            // 2^27), packed into two 64-bit words, each below 2^53
            auto val = [&](int g) { return __float2int_rn(__uint_as_float(v[g][2 * h + j])); };
            long long hi = val(3), lo = val(S - 1);
#pragma unroll
            for (int g = 0; g < 3; ++g) hi = mad_wide(val(g), 1 << (BITS * (3 - g)), hi);
#pragma unroll
            for (int g = 4; g < S - 1; ++g) lo = mad_wide(val(g), 1 << (BITS * (S - 1 - g)), lo);
            o[j] = oz_round(hi, lo, BITS * (S - 4), er + sx[32 + c8 * 8 + 2 * (lane & 3) + j]);
          }
          if (wide) {
            if (cc < n) *(double2*)(Mo + (int64_t)r * n + cc) = make_double2(o[0], o[1]);
          } else {
            const int al = r / D, be = r - al * D;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              if (cc + j >= n) continue;
              const int de = (cc + j) / D, ga = cc + j - de * D;
              if (par == 0) Mo[(int64_t)r * n + cc + j] = o[j];                       // (l,u),(r,d)
              else Mo[(int64_t)(be * D + de) * n + (ga * D + al)] = o[j];             // (u,r),(d,l)
            }
          }
        }
      }
    }
  } else {
    if (lane == 0) {
      // MMA issuer: accumulator g at tensor-memory columns 64 g
      int st = 0, ast = 0;
      uint32_t fph = 0, tph = 1;
      bool ok = true;
      for (int64_t tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x, tph ^= 1) {
        if (tile != blockIdx.x && !mbar_wait(&acc_empty, tph)) { ok = false; break; }
        tc_fence_after();
        for (int k = 0; k < steps; ++k, ++st) {
          if (!mbar_wait(&full_bar[ast], fph) || s_fail) { ok = false; break; }
          tc_fence_after();
          const int buf = (st >> 2) & 1, slot = st & 3;
          const uint64_t a0 = umma_desc(smem_u32(As + ast * kOzABytes));
          const uint64_t b0 = umma_desc(smem_u32(Bs + buf * oz_b_bytes(S))) + (uint64_t)(slot * 2);
#pragma unroll
          for (int i = 0; i < S; ++i) {
            constexpr int kMax = 256 / kOzTileN;     // slices of B in one instruction
            const uint64_t ad = a0 + (uint64_t)((((uint32_t)(i >> 2) * kOzAHalf) + (i & 3) * 32) >> 4);
            const int first = S - i < kMax ? S - i : kMax, rest = S - i - first;
            // slice 0 of A reaches every group: it starts the sums
            const uint32_t acc = (k == 0 && i == 0) ? 0u : 1u;
            umma<1>(tmem + (uint32_t)(i * kOzTileN), ad, b0, umma_idesc_f16(kOzTileM, kOzTileN * first), acc);
            if (rest > 0)
              umma<1>(tmem + (uint32_t)((i + kMax) * kOzTileN), ad, b0 + (uint64_t)((kMax * kOzTileN * 128) >> 4),
                      umma_idesc_f16(kOzTileM, kOzTileN * rest), acc);
          }
          umma_commit(&empty_a[ast]);
          if (slot == 3) umma_commit(&empty_b[buf]);
          if (++ast == kOzStages) { ast = 0; fph ^= 1; }
        }
        if (ok) umma_commit(&acc_full);
      }
      if (!ok) s_fail = 1;
      umma_commit(&done_bar);
      if (!mbar_wait(&done_bar, 0)) s_fail = 1;
    }
    __syncwarp();
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && s_fail) atomicOr(a.err, 1u);
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u));
  }
}

// ---------------------------------------------------------------------------
template <int BITS, int S>
static cudaError_t launch_ozaki(const GemmOzArgs& a, int64_t tiles, cudaStream_t st) {
  static std::atomic<uint64_t> attr{0};
  cudaError_t e = raise_smem_limit(k_gemm_ozaki<BITS, S>, (int)oz_smem(S), attr);
  if (e != cudaSuccess) return e;
  k_gemm_ozaki<BITS, S><<<(unsigned)std::min<int64_t>(tiles, 152), kOzThreads, oz_smem(S), st>>>(a, tiles);
  return cudaGetLastError();
}

cudaError_t launch_gemm_ozaki(const GemmOzArgs& args, cudaStream_t st) {
  GemmOzArgs a = args;
  if (a.n_items <= 0) return cudaSuccess;
  if (!gemm_ozaki_supported(a.n, a.K) || a.n_items > (1 << 30)) return cudaErrorInvalidValue;
  const int64_t rows = a.n_items * a.n;
  k_ozaki_expo<<<(unsigned)((2 * rows + 7) / 8), 256, 0, st>>>(a.X, a.Y, rows, a.K, a.expX);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  a.expY = a.expX + rows;
  // 16-byte accesses where the caller's arrays lie on such boundaries
  a.aligned = (((uintptr_t)a.X | (uintptr_t)a.Y) & 15) == 0;
  a.wide = ((uintptr_t)a.M & 15) == 0 && a.n % 2 == 0;
  const int64_t tiles = a.n_items * ((a.n + kOzTileM - 1) / kOzTileM) * ((a.n + kOzTileN - 1) / kOzTileN);
  return a.K <= 256 ? launch_ozaki<8, 7>(a, tiles, st) : launch_ozaki<7, 8>(a, tiles, st);
}

}  // namespace mctrg
