// K2, two-stage route: the SVD of a level matrix (Sec. II, Eq. exactSVD) with
// most of its reduction on the tensor cores.  GB300 issues FP64 at 2 lanes
// per clock per SM; the one-stage bidiagonalization spends (8/3) n^3 flops
// there.  This route splits the reduction in two (the successive band
// reduction of Bischof, Lang and Sun, 2000):
//
//  1. dense -> upper band with b = 8 superdiagonals, in panels of b columns.
//     Panel k: Householder QR of the column panel (FP64, k_band_qr), the
//     product W = V^T A of its reflectors with the trailing matrix
//     (k_band_gemm_w), the row panel updated and reduced by an LQ
//     factorization (k_band_lq), the product X = A U^T with the LQ reflectors
//     (k_band_gemm_x), and the two-sided trailing update
//     A <- A - [V | Y] [Z ; U], Z = T^T W, Y = (X - V Z U^T) T_U (k_band_update).
//     The three products carry the (8/3) n^3 flops.  They run as exact
//     integer products on the tensor cores: the trailing matrix is held in
//     62-bit fixed point (int64 relative to 2^e > 2 |A|_F; orthogonal updates
//     keep every entry below |A|_F), the FP64 operands (V, U, Y, Z) in 62-bit
//     fixed point relative to their own row or column exponent, each operand
//     split into eight signed 8-bit digits stored as FP16 (exact), and the
//     digit products with i + j <= 7 (W and X: 8) accumulated by tcgen05.mma in
//     tensor memory, one FP32 accumulator per digit group g = i + j (Ozaki, Ogita,
//     Oishi and Rump 2012; sums of up to 256 products of 8-bit digits are
//     integers below 2^24 for the leading groups, so FP32 holds them
//     exactly; longer sums are read out and added in integers every 256).  The update is applied in integer arithmetic, so apart from
//     the panel factorizations stage 1 issues no FP64 instruction per
//     trailing element.
//  2. band -> bidiagonal by bulge chasing (k_band_chase, eight warps a CTA whose
//     sweeps follow one another, one to four matrices in each warp's lanes,
//     the band in shared memory): per sweep i a right reflector clears row i
//     beyond the superdiagonal, and alternating left and right reflectors of
//     length <= b chase the bulge it creates down the band (LAPACK's dgbbrd
//     does this with Givens rotations; Householder reflectors here).
//     O(n^2 b) FP64 flops.
//  Then the bisection of the bidiagonalization route gives the singular
//  values, its inverse iteration the kept right vectors of the bidiagonal,
//  and k_band_backtr applies the chase's and the panels' right reflectors to
//  them, v = P1 P2 v_B.
//
// Every mbarrier wait is bounded; on expiry a kernel records an error word
// and skips its output, and frees its tensor memory.
#include <cuda_fp16.h>

#include <cstdint>

#include "common.cuh"
#include "kernels_band.h"
#include "tc_ptx.cuh"

namespace mctrg {

using namespace tcptx;

namespace {
constexpr int B = kBandW;        // band width / panel width
constexpr int kSl = 8;           // digit slices per operand (8 bits each)
constexpr int kFixBits = 62;     // fixed-point fraction bits of the trailing matrix (|A|_F below 2^61)
constexpr int kFloatP = 62;      // fixed-point bits of an FP64 operand below 2^e
constexpr int kZeroExp = -1100;  // exponent of an all-zero row or column
constexpr int kWin = 24;         // chase window: offsets c - r in [-7, 15] (+1 pad)
constexpr int kTileM = 128;      // rows of an MMA tile (tensor-memory lanes)
constexpr uint32_t kTileBytes = 128u * 128u;   // 128 rows x 128 bytes (4 slices x 16 K)

// Doubles of one matrix's panel scratch.
__host__ __device__ __forceinline__ size_t work_stride(int n) { return (size_t)26 * n + 128; }

// Per-matrix panel scratch, in doubles.
struct Work {
  double* V;    // [n][8]  reflectors of the column panel, rows relative to k
  double* T;    // [64]    their T factor (upper triangular)
  double* Z;    // [8][n]  W = V^T A, then Z = T^T W (columns relative to k+b)
  double* ZU;   // [64]    Z U^T
  double* Y;    // [n][8]  rows relative to k+b
  int* el;      // [n]     row exponents of [V | Y]
  int* er;      // [n]     column exponents of [Z 2^-ez ; U]
  int* ez;      // [1]     exponent of Z: every |z| < 2^ez
};
__device__ __forceinline__ Work work_of(double* base, int n) {
  Work w;
  w.V = base;
  w.T = w.V + (size_t)n * 8;
  w.Z = w.T + 64;
  w.ZU = w.Z + (size_t)8 * n;
  w.Y = w.ZU + 64;
  w.el = (int*)(w.Y + (size_t)n * 8);
  w.er = (int*)(w.Y + (size_t)n * 9);
  w.ez = w.er + n;
  return w;
}

// 2^p as a double, from exponent bits (beyond the normal range a product of
// two powers, which underflows or overflows as the scaling would).
__device__ __forceinline__ double p2(int p) {
  if (p >= -1022 && p <= 1023) return __hiloint2double((1023 + p) << 20, 0);
  p = max(-2044, min(2046, p));
  const int h = p / 2;
  return __hiloint2double((1023 + h) << 20, 0) * __hiloint2double((1023 + (p - h)) << 20, 0);
}

// round(x 2^sh) as an integer from the bits of x (no FP64 instruction); the
// caller keeps the result below 2^62.
__device__ __forceinline__ long long fix_of(double x, int sh_total) {
  const long long b = __double_as_longlong(x);
  const int be = (int)((b >> 52) & 0x7ff);
  const long long q = (b & 0xFFFFFFFFFFFFFll) | (be ? (1ll << 52) : 0ll);
  const int sh = (be ? be - 1075 : -1074) + sh_total;
  long long F;
  if (sh >= 0) F = q << sh;
  else if (sh > -62) F = (q + (1ll << (-sh - 1))) >> (-sh);
  else F = 0;
  return b < 0 ? -F : F;
}

// Exponent e with |x| < 2^e for the largest magnitude x (kZeroExp for 0).
__device__ __forceinline__ int exp_above(double amax) {
  const int be = (__double2hiint(amax) >> 20) & 0x7ff;
  if (amax == 0.0) return kZeroExp;
  return be ? be - 1022 : -1022;
}

// The eight balanced 8-bit digits of two integers (|x| < 2^63 - 2^62), as FP16
// (exact), packed per slice: out[s] holds digit s (0 the top one) of x0 in the
// low half and of x1 in the high half.  Adding 0x80 to every byte turns the
// balanced digits into the plain bytes of one 64-bit sum; a byte b placed
// under the exponent of 1024 reads as 1024 + b, so one permute and one packed
// subtraction make two digits.
__device__ __forceinline__ void digits2(long long x0, long long x1, uint32_t (&out)[kSl]) {
  const unsigned long long y0 = (unsigned long long)x0 + 0x8080808080808080ull;
  const unsigned long long y1 = (unsigned long long)x1 + 0x8080808080808080ull;
  const __half2 off = __halves2half2(__ushort_as_half(0x6480), __ushort_as_half(0x6480));   // 1024 + 128
#pragma unroll
  for (int h = 0; h < 2; ++h) {                  // the 32-bit halves, high first
    const uint32_t w0 = (uint32_t)(h ? y0 : y0 >> 32), w1 = (uint32_t)(h ? y1 : y1 >> 32);
    const uint32_t top = __byte_perm(w0, w1, 0x7632), low = __byte_perm(w0, w1, 0x5410);
    const uint32_t d[4] = {__byte_perm(top, 0x64646464u, 0x4341), __byte_perm(top, 0x64646464u, 0x4240),
                           __byte_perm(low, 0x64646464u, 0x4341), __byte_perm(low, 0x64646464u, 0x4240)};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const __half2 v = __hsub2(*reinterpret_cast<const __half2*>(&d[i]), off);
      out[h * 4 + i] = *reinterpret_cast<const uint32_t*>(&v);
    }
  }
}
// The digits of eight consecutive K values, one 16-byte piece per slice.
__device__ __forceinline__ void digits8(const long long (&x)[8], uint4 (&out)[kSl]) {
  uint32_t d[4][kSl];
#pragma unroll
  for (int p = 0; p < 4; ++p) digits2(x[2 * p], x[2 * p + 1], d[p]);
#pragma unroll
  for (int s = 0; s < kSl; ++s) out[s] = make_uint4(d[0][s], d[1][s], d[2][s], d[3][s]);
}

// Operand A of a k-step (128 rows x 16 K values): two 16 KB tiles of 128 rows x
// 128 bytes, four slices side by side in the 128-byte swizzle.  Byte offset of
// the 16-byte piece of slice s, row rho, half kh of the K values.
__device__ __forceinline__ uint32_t a_piece(int s, int rho, int kh) {
  return (uint32_t)((s >> 2) * kTileBytes + rho * 128 + (((((s & 3) << 1) | kh) ^ (rho & 7)) << 4));
}
// Operand B: 128 rows (slice s, column j: row 16 s + j) x 128 bytes, four
// k-steps (or four column tiles) side by side in slots of 32 bytes.
__device__ __forceinline__ uint32_t b_piece(int s, int j, int slot, int kh) {
  return (uint32_t)((s * 16 + j) * 128 + ((((slot << 1) | kh) ^ (j & 7)) << 4));
}

// The digit products of a k-step in the groups 0 .. G-1 as eight MMAs (36
// products for G = 8, 43 for G = 9): slice i of A times the slices 0 ..
// min(7, G-1-i) of B side by side (16 columns each) adds to the accumulators of
// the digit groups i .. G-1, 16 columns each.  One MMA per product read the A
// slice from shared memory 36 times, eight of them read it 8 times.
template <int G>
__device__ __forceinline__ void issue_products(uint32_t tmem, const uint8_t* A, const uint8_t* Bt, int slot, bool first) {
  const uint64_t a0 = umma_desc(smem_u32(A)), b0 = umma_desc(smem_u32(Bt)) + (uint64_t)(slot * 2);
#pragma unroll
  for (int i = 0; i < kSl; ++i) {
    const uint64_t ad = a0 + (uint64_t)((((uint32_t)(i >> 2) * kTileBytes) + (i & 3) * 32) >> 4);
    const int cols = G - i < kSl ? G - i : kSl;      // slices of B
    if (G > kSl && i == 1 && first) {
      // slice 0 of A has set the groups 0 .. 7: the product of slices 1 and 7 starts group 8
      umma<1>(tmem + (uint32_t)(kSl * 16), ad, b0 + (uint64_t)((7 * 16 * 128) >> 4), umma_idesc_f16(kTileM, 16), 0u);
      umma<1>(tmem + 16u, ad, b0, umma_idesc_f16(kTileM, 16 * 7), 1u);
    } else {
      umma<1>(tmem + (uint32_t)(i * 16), ad, b0, umma_idesc_f16(kTileM, 16 * cols), (first && i == 0) ? 0u : 1u);
    }
  }
}

// Tensor-memory loads without the wait: 32 lanes x 8 or 4 columns (lane = row),
// and 16 rows x 8 columns as four registers (rows lane / 4 and lane / 4 + 8,
// columns 2 (lane % 4) and the next).
static __device__ __forceinline__ void tmem_ld_x8(uint32_t taddr, uint32_t (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(taddr));
}
static __device__ __forceinline__ void tmem_ld_x4(uint32_t taddr, uint32_t (&v)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"(taddr));
}
static __device__ __forceinline__ void tmem_ld_16x8(uint32_t taddr, uint32_t (&v)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"(taddr));
}
static __device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(cols));
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tmem_free(uint32_t tmem, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols));
}

// round(v 2^p) for an integer v (p of either sign).
__device__ __forceinline__ long long shift_round(long long v, int p) {
  if (p >= 0) return p < 63 ? v << p : 0;
  if (p <= -63) return 0;
  return (v + (1ll << (-p - 1))) >> (-p);
}

// Warp sum (every lane receives it).
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Householder reflector (dlarfg) of a vector with first entry alpha and
// squared norm sq of the rest: H = I - tau v v^T, v_0 = 1, v_i = x_i scl,
// H x = beta e_1.  |alpha - beta| = |alpha| + |x| (no cancellation).
__device__ __forceinline__ void reflector(double alpha, double sq, double& beta, double& tau, double& scl) {
  if (sq == 0.0) { beta = alpha; tau = 0.0; scl = 0.0; return; }
  const double t = fma(alpha, alpha, sq), rn = inv_sqrt(t), nrm = t * rn;
  beta = -copysign(nrm, alpha);
  const double d = alpha - beta;
  tau = fabs(d) * rn;
  scl = inv(d);
}

// Scalars shared by the phases of a panel factorization.
struct PanelShared {
  double p[B], c[B], cs[B], tau[B], scl, G[B * B], T[B * B];
};

// Householder factorization of eight vectors x_0 .. x_7 of length m in shared
// memory (x_i at X + i ld): reflector j annihilates x_j beyond entry j and is
// applied to the later ones.  Per reflector one dot phase (a warp takes one
// dot over the whole vectors: x_j . x_i over the entries beyond j, j's square
// among them, with x_j not yet scaled), the scalars in one warp, one update
// phase (three barriers a reflector; six, a dot phase for the norm alone and
// the T recurrence in one thread before: QR 6.2 -> 4.6 ms and LQ 10.0 -> 6.8 for
// 1920 matrices of n = 256).  out(i, j, x) receives the final entry j <= i of x_i; on return X holds
// the reflectors (unit entry at j, zeros before it).  Bound by the FP64 pipe
// (a warp-wide FP64 instruction holds it 16 cycles), so the layout counts
// those: whole-vector dots share one five-step reduction, and the reflector's
// root and reciprocal are formed once.
template <class Out>
__device__ __forceinline__ void panel_factor(double* X, int ld, int m, PanelShared& sh, Out out) {
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, nt = blockDim.x;
  for (int j = 0; j < B; ++j) {
    const double* xj = X + (size_t)j * ld;
    if (warp < B - j) {
      const double* xi = xj + (size_t)warp * ld;
      double p = 0.0;
      for (int r = j + 1 + lane; r < m; r += 32) p = fma(xj[r], xi[r], p);
      p = warp_sum(p);
      if (lane == 0) sh.p[j + warp] = p;
    }
    __syncthreads();
    if (warp == 0) {
      double beta, tau, scl;
      reflector(xj[j], sh.p[j], beta, tau, scl);
      if (lane > j && lane < B) {
        const double xl = X[(size_t)lane * ld + j];
        const double c = tau * fma(scl, sh.p[lane], xl);
        sh.cs[lane] = c * scl;
        out(lane, j, xl - c);                        // final: no later reflector touches entry j
      }
      if (lane == 0) { sh.tau[j] = tau; sh.scl = scl; out(j, j, beta); }
      __syncwarp();
      if (lane >= j && lane < B) X[(size_t)lane * ld + j] = lane == j ? 1.0 : 0.0;
    }
    __syncthreads();
    const double scl = sh.scl;
    double cs[B];
#pragma unroll
    for (int i = 1; i < B; ++i) cs[i] = i > j ? sh.cs[i] : 0.0;
    for (int r = j + 1 + t; r < m; r += nt) {
      const double x = xj[r];
#pragma unroll
      for (int i = 1; i < B; ++i)
        if (i > j) X[(size_t)i * ld + r] = fma(-cs[i], x, X[(size_t)i * ld + r]);
      X[(size_t)j * ld + r] = x * scl;
    }
    __syncthreads();
  }
}

// Up to four dots a . x_c, c = c0 .. c0 + nd - 1, over m entries by one warp,
// reduced together; out[0 .. nd-1].
__device__ __forceinline__ void warp_dots4(const double* a, const double* X, int ld, int c0, int nd, int m, double* out) {
  const int lane = threadIdx.x & 31;
  const double* x = X + (size_t)c0 * ld;
  double p0 = 0.0, p1 = 0.0, p2 = 0.0, p3 = 0.0;
  for (int r = lane; r < m; r += 32) {
    const double ar = a[r];
    p0 = fma(ar, x[r], p0);
    if (nd > 1) p1 = fma(ar, x[ld + r], p1);
    if (nd > 2) p2 = fma(ar, x[2 * ld + r], p2);
    if (nd > 3) p3 = fma(ar, x[3 * ld + r], p3);
  }
  const double v = reduce4(p0, p1, p2, p3, lane);
  if ((lane & 7) == 0 && (lane >> 3) < nd) out[lane >> 3] = v;
}

// T of Q = H_0 ... H_{b-1} = I - Y T Y^T (forward, columnwise, as LAPACK's
// dlarft) for the reflectors X of panel_factor: the 28 products y_a . y_c in
// groups of up to four that share y_a, then the recurrence by one warp, lane i
// holding row i of T.
__device__ __forceinline__ void panel_t(const double* X, int ld, int m, PanelShared& sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  // the groups (a, first c): 0:1 0:5 1:2 1:6 2:3 2:7 3:4 4:5 5:6 6:7
  for (int g = warp; g < 10; g += nw) {
    const int a = g < 6 ? g >> 1 : g - 3, c0 = a + 1 + (g < 6 ? (g & 1) * 4 : 0);
    warp_dots4(X + (size_t)a * ld, X, ld, c0, min(4, B - c0), m, sh.G + a * B + c0);
  }
  __syncthreads();
  if (warp == 0) {
    double row[B];
#pragma unroll
    for (int j = 0; j < B; ++j) {
      double s = 0.0;
#pragma unroll
      for (int l = 0; l < j; ++l) s = fma(row[l], sh.G[l * B + j], s);   // row[l] = 0 for l < i
      row[j] = lane == j ? sh.tau[j] : (lane < j ? -sh.tau[j] * s : 0.0);
      if (lane < B) sh.T[lane * B + j] = row[j];
    }
  }
  __syncthreads();
}

// Exponent e with |x| < 2^e (kZeroExp for 0), from the bits of x: no FP64 instruction.
__device__ __forceinline__ int exp_of(double x) {
  const int hi = __double2hiint(x) & 0x7fffffff, be = hi >> 20;
  return be ? be - 1022 : ((hi | __double2loint(x)) ? -1022 : kZeroExp);
}
}  // namespace

bool band_supported(int n) { return n >= 64 && n <= kBandMaxN && n % B == 0; }

// sum over the sweeps i of ceil((n - 2 - i) / b)
int band_nref(int n) {
  const int m = n - 2, q = m / B, r = m % B;
  return B * q * (q + 1) / 2 + r * (q + 1);
}

size_t band_work_doubles(int n) { return work_stride(n); }

size_t band_panel_doubles(int n) { return (size_t)n * (B + 1) + band_work_doubles(n) + 1; }
size_t band_refl_doubles(int n) { return (size_t)band_nref(n) * B; }

void band_carve(void* panels, void* refl, int n, int64_t S, BandArgs& a) {
  double* p = (double*)panels;
  a.band = p; p += (size_t)S * n * (B + 1);
  a.work = p; p += (size_t)S * band_work_doubles(n);
  a.eA = (int*)p;
  a.refl = (double*)refl;
  a.n = n;
}

// ---------------------------------------------------------------------------
// Fixed-point copy of each matrix: e with |M|_F < 2^(e-1), Wk = round(M 2^(62-e)).
__global__ void __launch_bounds__(256) k_band_init(BandArgs a) {
  __shared__ double red[8];
  const int s = blockIdx.x, n = a.n;
  const double* M = a.M + (size_t)s * n * n;
  long long* A = (long long*)a.Wk + (size_t)s * n * n;
  double ss = 0.0;
  for (int i = threadIdx.x; i < n * n; i += blockDim.x) ss = fma(M[i], M[i], ss);
  ss = warp_sum(ss);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  ss = 0.0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) ss += red[w];
  const int e = ss > 0.0 ? exp_above(sqrt(ss)) + 1 : 0;
  if (threadIdx.x == 0) a.eA[s] = e;
  for (int i = threadIdx.x; i < n * n; i += blockDim.x) A[i] = fix_of(M[i], kFixBits - e);
}

// ---------------------------------------------------------------------------
// Panel k, QR of the column panel A[k:n][k:k+b] (m = n - k rows, the panel in
// shared memory column by column).  Writes R into the band, V (unit lower
// trapezoidal) and T into the scratch.
__global__ void __launch_bounds__(256) k_band_qr(BandArgs a, int k) {
  extern __shared__ double P[];                      // [b][m]
  __shared__ PanelShared sh;
  const int s = blockIdx.x, n = a.n, m = n - k, t = threadIdx.x;
  const long long* A = (const long long*)a.Wk + (size_t)s * n * n;
  const double unit = p2(a.eA[s] - kFixBits);
  Work w = work_of(a.work + (size_t)s * work_stride(n), n);
  for (int r = t; r < m; r += blockDim.x) {
#pragma unroll
    for (int j = 0; j < B; ++j) P[j * m + r] = (double)A[(size_t)(k + r) * n + k + j] * unit;
  }
  __syncthreads();
  double* band = a.band + ((size_t)s * n + k) * (B + 1);
  panel_factor(P, m, m, sh, [&](int c, int j, double x) { band[j * (B + 1) + (c - j)] = x; });
  for (int r = t; r < m; r += blockDim.x) {
#pragma unroll
    for (int j = 0; j < B; ++j) w.V[(size_t)r * 8 + j] = P[j * m + r];
  }
  panel_t(P, m, m, sh);
  if (t < 64) w.T[t] = sh.T[t];
}

// ---------------------------------------------------------------------------
// Tensor-core products W = V^T A and X = A U^T: one CTA of 256 threads per
// (matrix, 128 columns or rows of the trailing matrix, the MMA's M side); N is
// the reflectors' side (8 columns, padded to 16, for each of 8 slices) and K
// runs in stages of 16.  The threads split a stage of A into digit slices in
// one of two shared-memory buffers while the MMAs of the other run, thread 0
// issues the eight MMAs and commits them to the buffer's mbarrier; the
// reflectors are split four stages at a time.
//
// What bounds them: reading the trailing matrix (8 bytes an element; W at 2.8
// TB/s of DRAM) and splitting it (about 14 instructions an element), and X's
// FP64 epilogue; two CTAs an SM.  Third panel of 304 matrices of n = 256: W 141
// -> 54 us, X 129 -> 85 us, against one buffer, stages of 32 and one MMA per
// digit product.
namespace {
constexpr uint32_t kStageBytes = 2 * kTileBytes;   // one k-step of A
constexpr uint32_t kBBytes = 128 * 128;            // B: 128 rows x 4 k-steps
// Digit groups of W and X.  A and the reflectors are in fixed point relative to
// 2^eA > 2 |A|_F and to 1, so where |A|_F is well above the entries (a flat
// spectrum: |A|_F = 10 s_1 at n = 256) the products need bits beyond the eight
// groups that hold 64 of the whole: with eight, what was left out was the
// largest error of the reduction (its singular values' rms error at n = 256,
// flat, 2.3e-16 s_1; at n = 576 3.1e-16).
constexpr int kProdGroups = 9;

// Shared state of a product kernel.
struct ProdShared {
  uint64_t bar[2];
  uint32_t tmem_slot;
  int fail;
};
__device__ __forceinline__ uint8_t* align1k(uint8_t* p) { return (uint8_t*)(((uintptr_t)p + 1023) & ~(uintptr_t)1023); }

__device__ __forceinline__ uint32_t prod_begin(ProdShared& ps, uint8_t* Bs, uint32_t bbytes) {
  if (threadIdx.x == 0) {
    ps.fail = 0;
    mbar_init(&ps.bar[0], 1);
    mbar_init(&ps.bar[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // the rows 8 .. 15 of each slice of B stay zero
  for (int i = threadIdx.x; i < (int)(bbytes / 16); i += blockDim.x) ((uint4*)Bs)[i] = make_uint4(0, 0, 0, 0);
  if (threadIdx.x < 32) tmem_alloc(&ps.tmem_slot, 256);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  return ps.tmem_slot;
}

// Stages s0 .. s1-1 of the product (at most 16, so that the sums over K stay
// exact): split(st, dst) writes stage st of A (and fetches the next one's
// data), refl(r, j) is the FP64 value of reflector j at K index r.  Returns
// false when a wait expired.
template <class Split, class Refl>
__device__ __forceinline__ bool prod_stages(ProdShared& ps, uint32_t tmem, uint8_t* As, uint8_t* Bs, int klen, int s0,
                                            int s1, Split split, Refl refl) {
  const int t = threadIdx.x;
  int committed = s0;
  for (int st = s0; st < s1; ++st) {
    const int buf = st & 1;
    // the MMAs of stage st - 2 (and all before them) are done with this buffer
    if (st >= 2 && !mbar_wait(&ps.bar[buf], ((st >> 1) - 1) & 1)) atomicOr(&ps.fail, 1);
    split(st, As + (size_t)buf * kStageBytes);
    uint8_t* Bb = Bs + (size_t)((st >> 2) & 1) * kBBytes;
    if ((st & 3) == 0) {                             // the reflectors of the next four stages
      const int j = t & 7, kk = 2 * (t >> 3), r = st * 16 + kk;
      uint32_t d[kSl];
      digits2(r < klen ? fix_of(refl(r, j), kFloatP - 1) : 0ll,
              r + 1 < klen ? fix_of(refl(r + 1, j), kFloatP - 1) : 0ll, d);
#pragma unroll
      for (int s = 0; s < kSl; ++s)
        *(uint32_t*)(Bb + b_piece(s, j, kk >> 4, (kk >> 3) & 1) + (kk & 7) * 2) = d[s];
    }
    fence_async_smem();
    __syncthreads();
    if (ps.fail) break;
    if (t == 0) {
      tc_fence_after();
      issue_products<kProdGroups>(tmem, As + (size_t)buf * kStageBytes, Bb, st & 3, st == s0);
      umma_commit(&ps.bar[buf]);
    }
    ++committed;
  }
  const int last = committed - 1;
  if (last >= s0 && !mbar_wait(&ps.bar[last & 1], (last >> 1) & 1)) atomicOr(&ps.fail, 1);
  tc_fence_after();
  __syncthreads();
  return ps.fail == 0;
}

__device__ __forceinline__ void prod_end(ProdShared& ps, uint32_t tmem, bool ok, uint32_t* err) {
  if (!ok && threadIdx.x == 0) {
    atomicOr(err, 1u);
    // give products still in flight another bounded wait before their memory is freed
    for (uint32_t i = 0; i < kSpinLimit; ++i) __nanosleep(20);
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x < 32) tmem_free(tmem, 256);
}

// Columns 0 .. NJ-1 from `col` of this thread's row: the group sums g, added to
// hi 2^40 + lo (groups 0 .. 3 and 4 .. 8).
template <int NJ>
__device__ __forceinline__ void prod_read(uint32_t taddr, long long (&hi)[NJ], long long (&lo)[NJ]) {
  uint32_t v[kProdGroups][NJ];
#pragma unroll
  for (int g = 0; g < kProdGroups; ++g) {
    if constexpr (NJ == 8) tmem_ld_x8(taddr + (uint32_t)(g * 16), v[g]);
    else tmem_ld_x4(taddr + (uint32_t)(g * 16), v[g]);
  }
  tmem_wait_ld();
#pragma unroll
  for (int j = 0; j < NJ; ++j) {
    long long h = __float2int_rn(__uint_as_float(v[0][j])), l = __float2int_rn(__uint_as_float(v[4][j]));
#pragma unroll
    for (int g = 1; g < 4; ++g) h = (h << 8) + __float2int_rn(__uint_as_float(v[g][j]));
#pragma unroll
    for (int g = 5; g < kProdGroups; ++g) l = (l << 8) + __float2int_rn(__uint_as_float(v[g][j]));
    hi[j] += h;
    lo[j] += l;
  }
}

// The whole product over K = klen: the accumulators hold the sums of at most
// 256 products (exact in FP32 for the leading groups) and are read out and
// added in integers after every 16 stages.  read() adds them up.
template <class Split, class Refl, class Read>
__device__ __forceinline__ bool prod_all(ProdShared& ps, uint32_t tmem, uint8_t* As, uint8_t* Bs, int klen, Split split,
                                         Refl refl, Read read) {
  const int nst = (klen + 15) >> 4;
  for (int s0 = 0; s0 < nst; s0 += 16) {
    if (!prod_stages(ps, tmem, As, Bs, klen, s0, min(s0 + 16, nst), split, refl)) return false;
    read();
    if (s0 + 16 < nst) {                             // before the next stages overwrite the accumulators
      tc_fence_before();
      __syncthreads();
      tc_fence_after();
    }
  }
  return true;
}
constexpr size_t kProdSmem = 2 * kStageBytes + 2 * kBBytes + 1024;
}  // namespace

// W^T = A^T V over the rows k..n-1 (K) for the trailing columns k+b.. of one
// 128-column tile; a thread splits 8 rows of its column per stage (the warps
// read whole rows of the tile).
__global__ void __launch_bounds__(256, 2) k_band_gemm_w(BandArgs a, int k) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ ProdShared ps;
  uint8_t* As = align1k(smem_raw);
  uint8_t* Bs = As + 2 * kStageBytes;
  const int s = blockIdx.x, n = a.n, t = threadIdx.x, warp = t >> 5;
  const int rho = t & 127, kh = t >> 7;             // MMA row (column of A), and which 8 of a stage's 16 rows
  const int c = k + B + blockIdx.y * kTileM + rho;
  const int m = n - k;
  const long long* A = (const long long*)a.Wk + (size_t)s * n * n;
  Work w = work_of(a.work + (size_t)s * work_stride(n), n);
  const uint32_t tmem = prod_begin(ps, Bs, 2 * kBBytes);
  long long x[8];
  auto load = [&](int st) {
    const int rb = st * 16 + kh * 8;                 // relative to k; m is a multiple of 8
    const long long* p = A + (size_t)(k + rb) * n + c;
    const bool in = c < n && rb < m;
#pragma unroll
    for (int e = 0; e < 8; ++e) x[e] = in ? p[(size_t)e * n] : 0ll;
  };
  load(0);
  // row c of W^T: value = (hi 2^40 + lo) 2^(eA - 75); the two warp groups take four columns each
  const int jh = kh * 4;
  long long hi[4] = {}, lo[4] = {};
  const bool ok = prod_all(
      ps, tmem, As, Bs, m,
      [&](int st, uint8_t* dst) {
        uint4 d[kSl];
        digits8(x, d);
#pragma unroll
        for (int sl = 0; sl < kSl; ++sl) *(uint4*)(dst + a_piece(sl, rho, kh)) = d[sl];
        load(st + 1);                                // past the end: zeros
      },
      [&](int r, int j) { return w.V[(size_t)r * 8 + j]; },
      [&]() { prod_read<4>(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)jh, hi, lo); });
  if (ok) {
    if (c < n) {
      const double sc = p2(a.eA[s] - kFixBits - 13);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        w.Z[(size_t)(jh + j) * n + (c - k - B)] = fma((double)hi[j], 1099511627776.0 * sc, (double)lo[j] * sc);
    }
  }
  prod_end(ps, tmem, ok, a.err);
}

// ---------------------------------------------------------------------------
// Panel k, row panel: Z = T^T W, RP = A[k:k+b][k+b:] - V[0:b] Z, LQ of RP, T_U,
// Z U^T, the column exponents of [Z ; U].  U and T_U go into the working matrix
// (rows k..k+b-1), L into the band.
__global__ void __launch_bounds__(256, 4) k_band_lq(BandArgs a, int k) {
  extern __shared__ double R[];                      // [b][mp] the row panel, then Z
  __shared__ PanelShared sh;
  __shared__ double Ts[64], Vt[64], zu[64];
  __shared__ int s_ez;
  const int s = blockIdx.x, n = a.n, t = threadIdx.x, warp = t >> 5;
  const int mp = n - k - B;                          // columns k+b .. n-1
  double* Zs = R + (size_t)B * mp;
  long long* A = (long long*)a.Wk + (size_t)s * n * n;
  double* Ad = (double*)A;
  const int eA = a.eA[s];
  const double unit = p2(eA - kFixBits);
  Work w = work_of(a.work + (size_t)s * work_stride(n), n);
  if (t < 64) { Ts[t] = w.T[t]; Vt[t] = w.V[t]; }    // T and the top b x b block of V
  if (t == 0) s_ez = kZeroExp;
  __syncthreads();
  int ez = kZeroExp;
  for (int q = t; q < mp; q += blockDim.x) {
    const int c = k + B + q;
    asm volatile("" ::: "memory");                   // T and V stay in shared memory: in registers they would spill
    double wv[B], z[B];
#pragma unroll
    for (int i = 0; i < B; ++i) wv[i] = w.Z[(size_t)i * n + q];
#pragma unroll
    for (int j = 0; j < B; ++j) {
      double acc = 0.0;
#pragma unroll
      for (int i = 0; i <= j; ++i) acc = fma(Ts[i * B + j], wv[i], acc);
      z[j] = acc;
    }
    // the top b x b block of V is unit lower triangular
#pragma unroll
    for (int i = 0; i < B; ++i) {
      double acc = fma((double)A[(size_t)(k + i) * n + c], unit, -z[i]);
#pragma unroll
      for (int j = 0; j < i; ++j) acc = fma(-Vt[i * B + j], z[j], acc);
      R[i * mp + q] = acc;
      Zs[i * mp + q] = z[i];
      w.Z[(size_t)i * n + q] = z[i];
      ez = max(ez, exp_of(z[i]));
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ez = max(ez, __shfl_xor_sync(0xffffffffu, ez, o));
  if ((t & 31) == 0) atomicMax(&s_ez, ez);
  __syncthreads();
  ez = s_ez == kZeroExp ? eA : s_ez;
  if (t == 0) *w.ez = ez;
  double* band = a.band + ((size_t)s * n + k) * (B + 1) + B;
  panel_factor(R, mp, mp, sh, [&](int i, int j, double x) { band[i * (B + 1) + (j - i)] = x; });
  // Z U^T: warp i takes z_i against u_0..3 and u_4..7
  for (int g = warp; g < 2 * B; g += blockDim.x >> 5)
    warp_dots4(Zs + (size_t)(g >> 1) * mp, R, mp, (g & 1) * 4, 4, mp, zu + (g >> 1) * B + (g & 1) * 4);
  panel_t(R, mp, mp, sh);                            // T_U (its barriers cover zu)
  if (t < 64) {
    w.ZU[t] = zu[t];
    Ad[(size_t)(k + t / B) * n + k + (t % B)] = sh.T[t];
  }
  // U rows into the working matrix; the exponent of the update's right operand
  // column [Z 2^-ez ; U]
  for (int q = t; q < mp; q += blockDim.x) {
    int e = kZeroExp;
#pragma unroll
    for (int j = 0; j < B; ++j) {
      const double u = R[j * mp + q], z = Zs[j * mp + q];
      Ad[(size_t)(k + j) * n + k + B + q] = u;
      const int xz = exp_of(z);
      e = max(e, max(exp_of(u), xz == kZeroExp ? kZeroExp : xz - ez));
    }
    w.er[q] = e;
  }
}

// ---------------------------------------------------------------------------
// X = A U^T over the trailing rows (one 128-row tile, the MMA's rows) and
// columns k+b.. (K); then per row Y = (X - V Z U^T) T_U and the row exponent
// of [V | Y].  Eight lanes read the 128 bytes of a row's 16 columns (two each),
// so a warp's load covers whole sectors of four rows; the rows of one load are
// two apart, which keeps their pieces in different banks.
__global__ void __launch_bounds__(256, 2) k_band_gemm_x(BandArgs a, int k) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ ProdShared ps;
  __shared__ double ZUs[64], TUs[64];
  uint8_t* As = align1k(smem_raw);
  uint8_t* Bs = As + 2 * kStageBytes;
  const int s = blockIdx.x, n = a.n, t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int r0 = k + B + blockIdx.y * kTileM;
  const int mp = n - k - B;                          // K = columns k+b .. n-1
  const long long* A = (const long long*)a.Wk + (size_t)s * n * n;
  const double* Ad = (const double*)A;
  Work w = work_of(a.work + (size_t)s * work_stride(n), n);
  if (t < 64) { ZUs[t] = w.ZU[t]; TUs[t] = Ad[(size_t)(k + t / B) * n + k + (t % B)]; }
  const uint32_t tmem = prod_begin(ps, Bs, 2 * kBBytes);
  const int l8 = lane & 7;
  // row (within the tile) of load q
  auto row_of = [&](int q) { return warp * 16 + (q >> 1) * 8 + (q & 1) + 2 * (lane >> 3); };
  longlong2 x[4];
  auto load = [&](int st) {
    const int cb = st * 16 + 2 * l8;                 // relative to k + b
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = r0 + row_of(q);
      x[q] = (r < n && cb < mp) ? *(const longlong2*)(A + (size_t)r * n + k + B + cb) : make_longlong2(0, 0);
    }
  };
  load(0);
  long long hi[8] = {}, lo[8] = {};                  // (warps 0 .. 3)
  const bool ok = prod_all(
      ps, tmem, As, Bs, mp,
      [&](int st, uint8_t* dst) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          uint32_t d[kSl];
          digits2(x[q].x, x[q].y, d);
#pragma unroll
          for (int sl = 0; sl < kSl; ++sl) *(uint32_t*)(dst + a_piece(sl, row_of(q), l8 >> 2) + (l8 & 3) * 4) = d[sl];
        }
        load(st + 1);
      },
      [&](int r, int j) { return Ad[(size_t)(k + j) * n + k + B + r]; },
      [&]() { if (warp < 4) prod_read<8>(tmem + ((uint32_t)(warp * 32) << 16), hi, lo); });
  if (ok && warp < 4) {
    const int r = r0 + t;
    if (r < n) {
      const int eA = a.eA[s];
      const double sc = p2(eA - kFixBits - 13);
      double vr[B], xv[B], y[B];
#pragma unroll
      for (int i = 0; i < B; ++i) vr[i] = w.V[(size_t)(r - k) * 8 + i];
#pragma unroll
      for (int j = 0; j < B; ++j) {
        double acc = fma((double)hi[j], 1099511627776.0 * sc, (double)lo[j] * sc);
#pragma unroll
        for (int i = 0; i < B; ++i) acc = fma(-vr[i], ZUs[i * B + j], acc);
        xv[j] = acc;
      }
      // exponent of the update's left operand row [V 2^ez | Y] (both parts of
      // the order of the trailing matrix; the right operand carries Z 2^-ez)
      const int ez = *w.ez;
      int e = kZeroExp;
#pragma unroll
      for (int j = 0; j < B; ++j) {
        double acc = 0.0;
#pragma unroll
        for (int i = 0; i <= j; ++i) acc = fma(xv[i], TUs[i * B + j], acc);
        y[j] = acc;
        const int ev = exp_of(vr[j]);
        e = max(e, max(exp_of(acc), ev == kZeroExp ? kZeroExp : ev + ez));
      }
      const int ro = r - k - B;
#pragma unroll
      for (int j = 0; j < B; ++j) w.Y[(size_t)ro * 8 + j] = y[j];
      w.el[ro] = e;
    }
  }
  prod_end(ps, tmem, ok, a.err);
}

// ---------------------------------------------------------------------------
// Trailing update A[k+b:][k+b:] -= [V | Y] [Z ; U] for one 128-row tile and up
// to 256 columns (grid z), the 16-column tiles in turn: K = 2b = 16 (one k-step), applied in fixed point.
// The operands are [V 2^ez | Y] and [Z 2^-ez ; U] (the same product): V and U
// are of order 1, Y and Z of that of the trailing matrix, 2^ez (below |A|_F by the
// bits that 2^eA in its place cost: at n = 256 and a flat spectrum five).  The row operand shares one exponent
// over the tile's rows, the column operand one over each block of 64 columns
// (the largest of the per-row / per-column exponents: digits keep 62 bits of
// the largest entry), so every element of a tile takes the same shifts.
//
// Both operands are split once, before the loop over the column tiles; its two
// accumulators (128 columns of tensor memory each) let the MMAs of the next
// tile run while the warps apply this one, with no block barrier: a full
// mbarrier per accumulator is completed by the MMAs, an empty one by the eight
// warps.  A warp takes 16 rows; the 16 x 8 form of the tensor-memory load gives
// four lanes the eight columns of a row, so the reads and writes of the
// trailing matrix cover whole sectors (one row per lane, the first form of
// this kernel, touched 32 lines with every instruction and wrote half sectors:
// 186 us for the third panel of 304 matrices of n = 256, 87 us so).  What bounds
// it: the 16 bytes an element read and written (2.7 TB/s of DRAM at that size).
struct UpdShared {
  uint64_t full[2], empty[2];
  uint32_t tmem_slot;
  int fail, el, er[4];
};
__global__ void __launch_bounds__(256, 2) k_band_update(BandArgs a, int k) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ UpdShared us;
  uint8_t* As = align1k(smem_raw);
  uint8_t* Bs = As + kStageBytes;                    // blocks of 64 columns: 128 rows x 128 bytes
  const int s = blockIdx.x, n = a.n, t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int r0 = k + B + blockIdx.y * kTileM;       // first row of the tile
  const int z0 = blockIdx.z * 256;                   // first trailing column of this CTA's (at most 256)
  const int mp = min(256, n - k - B - z0);
  long long* A = (long long*)a.Wk + (size_t)s * n * n;
  const double* Ad = (const double*)A;
  Work w = work_of(a.work + (size_t)s * work_stride(n), n);
  const int eA = a.eA[s], ez = *w.ez;
  if (t == 0) {
    us.fail = 0;
    us.el = kZeroExp;
    for (int q = 0; q < 4; ++q) us.er[q] = kZeroExp;
    for (int q = 0; q < 2; ++q) { mbar_init(&us.full[q], 1); mbar_init(&us.empty[q], 8); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(&us.tmem_slot, 256);
  __syncthreads();
  {
    // the largest row exponent of the tile and the column exponents of the blocks
    int e = (t < 128 && r0 + t < n) ? w.el[r0 + t - k - B] : kZeroExp, f = t < mp ? w.er[z0 + t] : kZeroExp;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
      f = max(f, __shfl_xor_sync(0xffffffffu, f, o));
    }
    if (lane == 0) {
      if (t < 128) atomicMax(&us.el, e);
      atomicMax(&us.er[t >> 6], f);
    }
  }
  __syncthreads();
  const int el = us.el;
  {
    // A operand: row rho = [V[r] 2^ez | Y[r]]
    const int rho = t & 127, part = t >> 7, r = r0 + rho;
    long long x[8];
    const bool in = r < n && el != kZeroExp;
#pragma unroll
    for (int e = 0; e < 8; ++e)
      x[e] = !in ? 0ll
                 : part == 0 ? fix_of(w.V[(size_t)(r - k) * 8 + e], kFloatP - el + ez)
                             : fix_of(w.Y[(size_t)(r - k - B) * 8 + e], kFloatP - el);
    uint4 d[kSl];
    digits8(x, d);
#pragma unroll
    for (int sl = 0; sl < kSl; ++sl) *(uint4*)(As + a_piece(sl, rho, part)) = d[sl];
  }
  for (int p = t; p < 2 * ((mp + 15) & ~15); p += 256) {
    // B operand: column c = [Z[:, c] 2^-ez ; U[:, c]]
    const int half = (mp + 15) & ~15, part = p >= half, c = p - part * half;
    const int er = us.er[c >> 6];
    const bool in = c < mp && er != kZeroExp;
    long long x[8];
#pragma unroll
    for (int e = 0; e < 8; ++e)
      x[e] = !in ? 0ll
                 : part == 0 ? fix_of(w.Z[(size_t)e * n + z0 + c], kFloatP - er - ez)
                             : fix_of(Ad[(size_t)(k + e) * n + k + B + z0 + c], kFloatP - er);
    uint4 d[kSl];
    digits8(x, d);
    uint8_t* Bb = Bs + (size_t)(c >> 6) * kBBytes;
#pragma unroll
    for (int sl = 0; sl < kSl; ++sl) *(uint4*)(Bb + b_piece(sl, c & 15, (c >> 4) & 3, part)) = d[sl];
  }
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = us.tmem_slot;
  const int ntile = (mp + 15) >> 4;
  // MMAs of tile ct into accumulator ct & 1 (thread 0)
  auto issue = [&](int ct) {
    issue_products<kSl>(tmem + (uint32_t)((ct & 1) * 128), As, Bs + (size_t)(ct >> 2) * kBBytes, ct & 3, true);
    umma_commit(&us.full[ct & 1]);
  };
  // this thread's rows (two) and column pair within a tile
  const int rw = (warp & 3) * 32 + (warp >> 2) * 16 + (lane >> 2), cl = 2 * (lane & 3);
  const uint32_t tlane = (uint32_t)((warp & 3) * 32 + (warp >> 2) * 16) << 16;
  const int ra = r0 + rw, rb = ra + 8;
  long long* pa = A + (size_t)ra * n + k + B + z0 + cl;
  long long* pb = pa + (size_t)8 * n;
  const bool oka = ra < n && el != kZeroExp, okb = rb < n && el != kZeroExp;
  longlong2 nx[4];                                   // the next tile's elements: (row a, row b) x (columns, columns + 8)
  auto load = [&](int ct) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int c = ct * 16 + 8 * h;                 // mp is a multiple of 8
      nx[2 * h] = (oka && c < mp) ? *(const longlong2*)(pa + c) : make_longlong2(0, 0);
      nx[2 * h + 1] = (okb && c < mp) ? *(const longlong2*)(pb + c) : make_longlong2(0, 0);
    }
  };
  if (t == 0) issue(0);
  __syncwarp();
  load(0);
  for (int ct = 0; ct < ntile; ++ct) {
    bool ok = true;
    if (t == 0 && ct + 1 < ntile) {
      // the warps have read tile ct - 1 out of the accumulator that tile ct + 1 takes
      if (ct >= 1) ok = mbar_wait(&us.empty[(ct + 1) & 1], ((ct - 1) >> 1) & 1);
      tc_fence_after();
      if (ok) issue(ct + 1);
    }
    __syncwarp();
    longlong2 q[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) q[i] = nx[i];
    if (ct + 1 < ntile) load(ct + 1);
    ok = mbar_wait(&us.full[ct & 1], (ct >> 1) & 1) && ok;
    if (__any_sync(0xffffffffu, !ok)) {              // expired: the other warps' waits expire too
      if (lane == 0) atomicOr(&us.fail, 1);
      break;
    }
    tc_fence_after();
    const int er = us.er[ct >> 2];
    // value of an element: (hi 2^32 + lo) 2^(el + er - 68), in fixed-point units 2^(eA - kFixBits)
    const int sh = el + er - eA - 68 + kFixBits;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      // group sums are integers of at most 8 x 16 x 2^14 = 2^21 in magnitude,
      // read back exactly by adding 1.5 2^23 (an FP32 add; the bias 0x4B400000
      // of each is taken out of the pair sums) and paired in 32 bits
      uint32_t v[kSl][4];
#pragma unroll
      for (int g = 0; g < kSl; ++g)
        tmem_ld_16x8(tmem + tlane + (uint32_t)((ct & 1) * 128 + g * 16 + h * 8), v[g]);
      tmem_wait_ld();
      if (h == 1) {                                  // the last read of this accumulator
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&us.empty[ct & 1]);
      }
      constexpr uint32_t kBias = 0x4B400000u * 257u;
      auto pair = [&](int g, int e) {
        const uint32_t b0 = __float_as_uint(__uint_as_float(v[g][e]) + 12582912.0f);
        const uint32_t b1 = __float_as_uint(__uint_as_float(v[g + 1][e]) + 12582912.0f);
        return (int)(b0 * 256u + b1 - kBias);
      };
      long long del[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const long long hi = (long long)pair(0, e) * 65536 + pair(2, e);
        const long long lo = (long long)pair(4, e) * 65536 + pair(6, e);
        if (sh < 0 && sh > -32) del[e] = (hi << (32 + sh)) + ((lo + (1ll << (-sh - 1))) >> (-sh));
        else if (sh <= -32) del[e] = shift_round(hi + (lo >> 32), 32 + sh);   // what is left of lo is far below a unit
        else del[e] = shift_round(hi, 32 + sh) + shift_round(lo, sh);
      }
      q[2 * h].x -= del[0]; q[2 * h].y -= del[1];
      q[2 * h + 1].x -= del[2]; q[2 * h + 1].y -= del[3];
      const int c = ct * 16 + 8 * h;
      if (c < mp && er != kZeroExp) {
        if (oka) *(longlong2*)(pa + c) = q[2 * h];
        if (okb) *(longlong2*)(pb + c) = q[2 * h + 1];
      }
    }
  }
  __syncthreads();
  if (us.fail && t == 0) {
    atomicOr(a.err, 1u);
    // give products still in flight another bounded wait before their memory is freed
    for (uint32_t i = 0; i < kSpinLimit; ++i) __nanosleep(20);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_free(tmem, 256);
}

// ---------------------------------------------------------------------------
// Stage 2: bulge chasing, several matrices per warp (LPM lanes each: every FP64
// instruction serves all of them, the reflector's formation included); each
// band and its bulges in shared memory, entry (r, c) at W[r * kWin + (c - r + 7)]
// (c - r in -7..15).  Per step a right reflector of length L <= b clears a row
// beyond its superdiagonal over rows row .. row+15 (one or two rows per lane),
// then a left reflector clears the bulge below the diagonal over columns c0 ..
// c0+15.
//
// Bound by the FP64 pipe: forming a reflector costs about as many warp
// instructions (18: the norm's reduction, a reciprocal square root, a
// reciprocal) as applying it with 16 lanes per matrix (17), so eight lanes per
// matrix, four matrices per warp, take 26 instead of 35 instructions per
// matrix and step.  Both forms do the same arithmetic in the same order.
__device__ __forceinline__ void chase_reflector(double x, int l, int L, int hb, double& v, double& tau, double& beta) {
  double p = (l >= 1 && l < L) ? x * x : 0.0;
  p += __shfl_xor_sync(0xffffffffu, p, 1);
  p += __shfl_xor_sync(0xffffffffu, p, 2);
  p += __shfl_xor_sync(0xffffffffu, p, 4);
  const double sq = __shfl_sync(0xffffffffu, p, hb), alpha = __shfl_sync(0xffffffffu, x, hb);
  if (sq == 0.0) { v = l == 0 ? 1.0 : 0.0; tau = 0.0; beta = alpha; return; }
  // |beta| = sqrt(alpha^2 + sq); d = alpha - beta (no cancellation);
  // tau = (beta - alpha) / beta = |d| / |beta|, v = x / d
  const double t = fma(alpha, alpha, sq), rn = inv_sqrt(t), nrm = t * rn;
  beta = -copysign(nrm, alpha);
  const double d = alpha - beta;
  tau = fabs(d) * rn;
  v = l == 0 ? 1.0 : (l < L ? x * inv(d) : 0.0);
}

// Steps of sweep i of the chase on an n x n band (right reflectors it stores).
// (step t has c0 = i + 1 + 8t and runs while c0 < n - 1)
__host__ __device__ __forceinline__ int sweep_steps(int i, int n) {
  const int m = n - 2 - i;
  return m > 0 ? (m + B - 1) / B : 0;
}

// Sweeps run pipelined: warp w of kChaseWarps takes sweeps w, w + kChaseWarps,
// ...; step t of sweep i starts once sweep i-1 has finished step t+3 (or all
// of its steps), which keeps the regions of concurrent steps apart (a step of
// sweep i touches rows [c0-8, c0+8) and columns [c0, c0+16) with
// c0 = i + 1 + 8t).  Progress words in shared memory, a ring of kRing slots
// holding i * 256 + steps done; waits are bounded (error word on expiry).
constexpr int kChaseWarps = 8, kRing = 16, kLag = 3;

// mats: matrices per CTA (at most 32 / LPM; fewer where shared memory holds fewer).
template <int LPM>
__global__ void __launch_bounds__(kChaseWarps * 32) k_band_chase(BandArgs a, int nref, int mats) {
  constexpr int RPL = 16 / LPM;                       // rows (or columns) of a 16-block per lane
  extern __shared__ double Bw[];
  __shared__ int prog[kRing];
  __shared__ int s_fail;
  const int n = a.n, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int l = lane & (LPM - 1), q4 = lane / LPM, hb = lane & ~(LPM - 1);
  const int s = mats * blockIdx.x + q4;
  const bool live = q4 < mats && s < a.S;             // lanes of absent matrices touch nothing
  const int nn = live ? n : 0;
  double* W = Bw + (size_t)(live ? q4 : 0) * n * kWin;
  for (int i = threadIdx.x; i < mats * n * kWin; i += blockDim.x) Bw[i] = 0.0;
  if (threadIdx.x < kRing) prog[threadIdx.x] = -1;
  if (threadIdx.x == 0) s_fail = 0;
  __syncthreads();
  for (int hh = 0; hh < mats; ++hh) {
    const int sm = mats * blockIdx.x + hh;
    if (sm >= a.S) break;
    const double* band = a.band + (size_t)sm * n * (B + 1);
    double* Wm = Bw + (size_t)hh * n * kWin;
    for (int i = threadIdx.x; i < n * (B + 1); i += blockDim.x) {
      const int r = i / (B + 1), o = i % (B + 1);
      if (r + o < n) Wm[r * kWin + o + 7] = band[i];
    }
  }
  __syncthreads();
#define AT(r, c) W[(r) * kWin + ((c) - (r) + 7)]
  double* refl = a.refl + (size_t)(live ? s : 0) * nref * B;
  volatile int* vprog = prog;
  // reflector index of this warp's first sweep
  int base = 0;
  for (int i = 0; i < warp && i + 1 < n; ++i) base += sweep_steps(i, n);
  bool fail = false;
  for (int i = warp; i + 1 < n && !fail; i += kChaseWarps) {
    const int T = sweep_steps(i, n), Tp = i > 0 ? sweep_steps(i - 1, n) : 0;
    if (lane == 0) vprog[i % kRing] = i * 256;
    int c0 = i + 1, c1 = min(i + B, n - 1), row = i;
    for (int t = 0; t < T; ++t) {
      if (i > 0) {                                    // wait for sweep i-1 to be kLag steps ahead
        const int need = min(t + kLag, Tp);
        if (lane == 0) {
          uint32_t it = 0;
          for (;; ++it) {
            const int v = vprog[(i - 1) % kRing];
            if ((v >> 8) > i - 1 || ((v >> 8) == i - 1 && (v & 255) >= need)) break;
            if (it > tcptx::kSpinLimit || *(volatile int*)&s_fail) { atomicOr(&s_fail, 1); break; }
            __nanosleep(20);
          }
          __threadfence_block();
        }
        __syncwarp();
        if (*(volatile int*)&s_fail) { fail = true; break; }
      }
      const int L = c1 - c0 + 1, Ll = live ? L : 0;
      const int idx = base + t;
      double v, tau, beta, vv[B], x[RPL][B];
      // right reflector: clear row `row` at columns c0+1 .. c1; rows row .. row+15
      chase_reflector(l < Ll ? AT(row, c0 + l) : 0.0, l, L, hb, v, tau, beta);
      if (live && l < B) refl[(size_t)idx * B + l] = l == 0 ? tau : v;
#pragma unroll
      for (int q = 0; q < B; ++q) vv[q] = __shfl_sync(0xffffffffu, v, hb + q);
#pragma unroll
      for (int h = 0; h < RPL; ++h) {
        const int r = row + l + LPM * h;
        double acc = 0.0;
#pragma unroll
        for (int q = 0; q < B; ++q) {
          const int cc = c0 + q;
          x[h][q] = (r < nn && cc <= c1 && cc - r >= -7) ? AT(r, cc) : 0.0;
          acc = fma(x[h][q], vv[q], acc);
        }
        acc *= -tau;
#pragma unroll
        for (int q = 0; q < B; ++q) {
          const int cc = c0 + q;
          const double y = fma(acc, vv[q], x[h][q]);
          if (r < nn && cc <= c1 && cc - r >= -7) AT(r, cc) = y;
        }
      }
      __syncwarp();
      if (l < Ll) AT(row, c0 + l) = l == 0 ? beta : 0.0;
      __syncwarp();
      // left reflector: clear column c0 at rows c0+1 .. c1; columns c0 .. c0+15
      chase_reflector(l < Ll ? AT(c0 + l, c0) : 0.0, l, L, hb, v, tau, beta);
#pragma unroll
      for (int q = 0; q < B; ++q) vv[q] = __shfl_sync(0xffffffffu, v, hb + q);
#pragma unroll
      for (int h = 0; h < RPL; ++h) {
        const int cc = c0 + l + LPM * h;
        double acc = 0.0;
#pragma unroll
        for (int q = 0; q < B; ++q) {
          x[h][q] = (cc < nn && q < L) ? AT(c0 + q, cc) : 0.0;
          acc = fma(x[h][q], vv[q], acc);
        }
        acc *= -tau;
#pragma unroll
        for (int q = 0; q < B; ++q) {
          const double y = fma(acc, vv[q], x[h][q]);
          if (cc < nn && q < L) AT(c0 + q, cc) = y;
        }
      }
      __syncwarp();
      if (l < Ll) AT(c0 + l, c0) = l == 0 ? beta : 0.0;
      __syncwarp();
      if (lane == 0) {                                // publish: step t of sweep i done
        __threadfence_block();
        vprog[i % kRing] = i * 256 + t + 1;
      }
      row = c0;
      c0 += B;
      c1 = min(c1 + B, n - 1);
    }
    for (int q = i; q < i + kChaseWarps && q + 1 < n; ++q) base += sweep_steps(q, n);
  }
  __syncthreads();
  if (s_fail) {
    if (threadIdx.x == 0) atomicOr(a.err, 1u);
    return;
  }
  if (live && warp == 0) {
    double* bd = a.bd + (size_t)s * 3 * n;
    for (int r = l; r < n; r += LPM) {
      bd[r] = AT(r, r);
      bd[n + r] = r + 1 < n ? AT(r, r + 1) : 0.0;
      bd[2 * n + r] = 0.0;
    }
  }
#undef AT
}

// ---------------------------------------------------------------------------
// v = P1 P2 v_B for a group of up to GV kept vectors of one matrix, one CTA of 128
// threads; the vectors in shared memory (row stride n + 1: the vectors in
// different banks).  GV is 16, or 4 where groups of 16 are fewer than the SMs (the
// same sums either way; 16 matrices of n = 576, 24 vectors: 5.0 -> 2.6 ms).  P2: the chase's sweeps in reverse order; the right
// reflectors of one sweep act on disjoint column blocks c0 = i + 1 + 8q, so
// they commute and are applied at once, one (reflector, vector) pair per
// thread.  P1: the panels' compact reflectors in reverse order,
// v <- v - U^T T_U U v: U staged in shared memory, thread (a, j) forms
// (U v_a)_j, then (T_U U v_a)_j, then the threads (a, part) update
// v_a.
constexpr int kBtThreads = 128;
template <int GV>
__global__ void __launch_bounds__(kBtThreads) k_band_backtr(BandArgs a, BandVecArgs va, int nref) {
  extern __shared__ double Vs[];                     // [GV][n+1], then U [8][n]
  __shared__ double tv[GV][B + 1], tp[GV][B + 1], s_scale[GV];
  const int s = blockIdx.x, n = a.n, t = threadIdx.x;
  const int ld = n + 1;
  double* Us = Vs + (size_t)GV * ld;
  const int g0 = GV * blockIdx.y;                     // first kept vector of this group
  const int nk = min(va.nk[s] - g0, GV);
  if (nk <= 0) return;
  double* vrow = va.vrows + ((size_t)s * va.kstride + g0) * n;
  for (int e = t; e < nk * n; e += kBtThreads) Vs[(e / n) * ld + e % n] = vrow[e];
  __syncthreads();
  const double* refl = a.refl + (size_t)s * nref * B;
  int base = nref;                                    // reflector index of sweep i's first step
  for (int i = n - 2; i >= 0 && nk > 0; --i) {
    const int T = sweep_steps(i, n);
    base -= T;
    for (int p = t; p < nk * T; p += kBtThreads) {
      const int q = p / nk, av = p - q * nk;
      const double* rv = refl + (size_t)(base + q) * B;
      const double tau = rv[0];
      if (tau == 0.0) continue;
      const int c0 = i + 1 + B * q, L = min(B, n - c0);
      double* x = Vs + (size_t)av * ld + c0;
      double vv[B];
      vv[0] = 1.0;
#pragma unroll
      for (int l = 1; l < B; ++l) vv[l] = l < L ? rv[l] : 0.0;
      double acc = x[0];
#pragma unroll
      for (int l = 1; l < B; ++l)
        if (l < L) acc = fma(vv[l], x[l], acc);
      acc *= tau;
#pragma unroll
      for (int l = 0; l < B; ++l)
        if (l < L) x[l] = fma(-acc, vv[l], x[l]);
    }
    __syncthreads();
  }
  const double* Ad = (const double*)(a.Wk + (size_t)s * n * n);
  const int av = t & (GV - 1), hj = t / GV;           // vector, and j (or the part of the columns)
  for (int k = n - 2 * B; k >= 0 && nk > 0; k -= B) {
    const int cb = k + B, mp = n - cb;
    for (int e = t; e < B * mp; e += kBtThreads) {
      const int j = e / mp, c = e - j * mp;
      Us[j * n + c] = Ad[(size_t)(k + j) * n + cb + c];
    }
    __syncthreads();
    if (av < nk && hj < B) {                          // (U v_a)_j
      const double* x = Vs + (size_t)av * ld + cb;
      const double* u = Us + (size_t)hj * n;
      double acc = 0.0;
      for (int c = 0; c < mp; ++c) acc = fma(u[c], x[c], acc);
      tv[av][hj] = acc;
    }
    __syncthreads();
    if (av < nk && hj < B) {                          // (T_U U v_a)_i, T_U upper triangular
      double acc = 0.0;
      for (int j = hj; j < B; ++j) acc = fma(Ad[(size_t)(k + hj) * n + k + j], tv[av][j], acc);
      tp[av][hj] = acc;
    }
    __syncthreads();
    if (av < nk) {
      double* x = Vs + (size_t)av * ld + cb;
      double tq[B];
#pragma unroll
      for (int j = 0; j < B; ++j) tq[j] = tp[av][j];
      for (int c = hj; c < mp; c += kBtThreads / GV) {
        double y = x[c];
#pragma unroll
        for (int j = 0; j < B; ++j) y = fma(-Us[j * n + c], tq[j], y);
        x[c] = y;
      }
    }
    __syncthreads();
  }
  // the two stages' n^2 / 16 reflectors have moved the vectors' lengths by some sqrt(n) roundings: unit again
  const double* sg = va.sig + (size_t)s * va.n_pad;
  const int* kept = va.kept + (size_t)s * va.kstride + g0;
  for (int q = t >> 5; q < nk; q += kBtThreads / 32) {
    const double* x = Vs + (size_t)q * ld;
    double p = 0.0;
    for (int c = t & 31; c < n; c += 32) p = fma(x[c], x[c], p);
    p = warp_sum(p);
    if ((t & 31) == 0) s_scale[q] = p > 0.0 ? (va.unit_rows ? 1.0 : sg[kept[q]]) * inv_sqrt(p) : 0.0;
  }
  __syncthreads();
  for (int e = t; e < nk * n; e += kBtThreads) vrow[e] = s_scale[e / n] * Vs[(e / n) * ld + e % n];
}

// ---------------------------------------------------------------------------
namespace {
constexpr size_t kUpdSmem = kStageBytes + 4 * kBBytes + 1024;
}  // namespace

cudaError_t launch_band_reduce(const BandArgs& a, bool chase, cudaStream_t st) {
  if (a.S <= 0) return cudaSuccess;
  if (!band_supported(a.n)) return cudaErrorInvalidValue;
  static std::atomic<uint64_t> at_w{0}, at_x{0}, at_u{0}, at_q{0}, at_l{0};
  cudaError_t e = raise_smem_limit(k_band_gemm_w, (int)kProdSmem, at_w);
  if (e == cudaSuccess) e = raise_smem_limit(k_band_gemm_x, (int)kProdSmem, at_x);
  if (e == cudaSuccess) e = raise_smem_limit(k_band_update, (int)kUpdSmem, at_u);
  if (e == cudaSuccess) e = raise_smem_limit(k_band_qr, (int)(B * kBandMaxN * sizeof(double)), at_q);
  if (e == cudaSuccess) e = raise_smem_limit(k_band_lq, (int)(2 * B * kBandMaxN * sizeof(double)), at_l);
  if (e != cudaSuccess) return e;
  const int n = a.n, S = a.S;
  k_band_init<<<S, 256, 0, st>>>(a);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  for (int k = 0; k < n; k += B) {
    k_band_qr<<<S, 256, (size_t)B * (n - k) * sizeof(double), st>>>(a, k);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (k + B >= n) break;
    const int mp = n - k - B;
    const int tiles = (mp + kTileM - 1) / kTileM;
    k_band_gemm_w<<<dim3(S, tiles), 256, kProdSmem, st>>>(a, k);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_band_lq<<<S, 256, (size_t)2 * B * mp * sizeof(double), st>>>(a, k);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_band_gemm_x<<<dim3(S, tiles), 256, kProdSmem, st>>>(a, k);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_band_update<<<dim3(S, tiles, (mp + 255) / 256), 256, kUpdSmem, st>>>(a, k);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return chase ? launch_band_chase(a, st) : cudaSuccess;
}

template <int LPM>
static cudaError_t launch_chase(const BandArgs& a, int mats, cudaStream_t st) {
  static std::atomic<uint64_t> at{0};
  cudaError_t e = raise_smem_limit(k_band_chase<LPM>, 227 * 1024, at);
  if (e != cudaSuccess) return e;
  k_band_chase<LPM><<<(a.S + mats - 1) / mats, kChaseWarps * 32, (size_t)mats * a.n * kWin * sizeof(double), st>>>(
      a, band_nref(a.n), mats);
  return cudaGetLastError();
}

cudaError_t launch_band_chase(const BandArgs& a, cudaStream_t st) {
  if (a.S <= 0) return cudaSuccess;
  if (!band_supported(a.n)) return cudaErrorInvalidValue;
  // four matrices per CTA (of n <= 288: 4 x 48 KB) once two per SM do not hold
  // the batch: 1920 of n = 256 23.8 -> 19.6 ms; below that two, whose shorter
  // step is the shorter chain (304: 3.6 ms in 152 CTAs, 4.9 in 76)
  constexpr size_t kCap = 226 * 1024;
  const size_t per = (size_t)a.n * kWin * sizeof(double);
  if (a.S > 2 * 152 && 4 * per <= kCap) return launch_chase<8>(a, 4, st);
  return launch_chase<16>(a, 2 * per <= kCap ? 2 : 1, st);
}

template <int GV>
static cudaError_t launch_backtr(const BandVecArgs& va, cudaStream_t st) {
  const BandArgs& a = *va.band;
  static std::atomic<uint64_t> at{0};
  auto bytes = [](int n) { return (size_t)((GV + B) * n + GV) * sizeof(double); };
  cudaError_t e = raise_smem_limit(k_band_backtr<GV>, (int)bytes(kBandMaxN), at);
  if (e != cudaSuccess) return e;
  const dim3 grid((unsigned)a.S, (unsigned)((std::max(1, va.kmax) + GV - 1) / GV));
  k_band_backtr<GV><<<grid, kBtThreads, bytes(a.n), st>>>(a, va, band_nref(a.n));
  return cudaGetLastError();
}

cudaError_t launch_band_backtr(const BandVecArgs& va, cudaStream_t st) {
  const int64_t S = va.band->S;
  if (S <= 0) return cudaSuccess;
  return S * ((std::max(1, va.kmax) + 15) / 16) < 152 ? launch_backtr<4>(va, st) : launch_backtr<16>(va, st);
}

}  // namespace mctrg
