// K2 for levels whose matrices have rank at most K < n by construction: the
// plaquette matrix is M = X Yt^T with inner dimension K = d^2 (d the parents'
// leg dimension), and the first level that every trajectory splits on its own
// has d^2 < n = D^2 (n = 64 or 144 with K = 16, n = 576 with K = 256).  Its SVD
// (Sec. II, Eq. exactSVD) is that of the K x K core of the two QR factors
// (Businger and Golub's QR-then-SVD for products), M = Qx (Rx Ry^T) Qy^T: the
// other n - K singular values are zero.  Householder QR is backward stable
// normwise, so the core's values carry an error of a few eps |X| |Yt|, the
// class of the product M's own rounding.
//
// The one-sided Jacobi that these levels took before works on all of M: 18.6 ms
// for 4096 matrices of n = 64, 23.3 ms for 768 of n = 144 (both K = 16), 424 ms
// for 32 of n = 576 (K = 256; one matrix per CTA).  Now, for the same levels:
// the QR of both factors 1.0, 0.42 and 11 ms, the cores' SVD 1.7 ms and 0.45 ms
// (K = 16, Jacobi) and 13 ms (K = 256, two-stage reduction and bisection), the
// expansion 0.4, 0.24 and 1.7 ms; and the n x n product goes, since only the
// core is needed.  Whole runs when this came: L = 16, chi = 8, 256 trajectories
// 50.6 -> 35.6 ms; chi = 12, 48 trajectories 60.3 -> 36.7; chi = 24, 8
// trajectories 556 -> 149.
#include <algorithm>

#include "common.cuh"
#include "kernels_lr.h"

namespace mctrg {

namespace {
constexpr size_t kQrSmemCap = 200 * 1024;

// Doubles of the per-step vectors: column, w, per-warp partial dots, scalars.
__host__ __device__ __forceinline__ size_t qr_aux_doubles(int n, int K, int nw) {
  return (size_t)n + K + (size_t)nw * K + nw + 4;
}

// Rows i > k of one step: a = A[i] - v_i w, column k+1 handed to the next step
// with its dots over the rows below it (w is linear in the column, so the
// next step needs no pass of its own).  G lanes hold a row's columns
// k+1+l+G q; a warp takes 32 / G rows at once, R times.  Returns this lane's
// share of the new column's square below row k+1.
template <int QL, int G, int R>
__device__ __forceinline__ double qr_pass(double* A, int n, int K, int k, double* vcol, const double* wv,
                                          double* wpart, int warp, int nw, int lane) {
  constexpr int RG = 32 / G;
  const int gl = lane & (G - 1), sub = lane / G;
  const int c0 = k + 1 + gl;
  double w[QL], acc[QL];
#pragma unroll
  for (int q = 0; q < QL; ++q) {
    w[q] = c0 + G * q < K ? wv[c0 + G * q] : 0.0;
    acc[q] = 0.0;
  }
  double nsq = 0.0;
  const int step = nw * RG * R;
  // the warp's loop bound is the same for every lane: rows past the end are masked
  for (int ib = k + 1 + warp * RG * R; ib < n; ib += step) {
    double a[R][QL];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int i = ib + r * RG + sub;
      const bool ok = i < n;
      const double vi = ok ? vcol[i] : 0.0;
#pragma unroll
      for (int q = 0; q < QL; ++q)
        a[r][q] = ok ? fma(-vi, w[q], A[(size_t)i * K + min(c0 + G * q, K - 1)]) : 0.0;
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int i = ib + r * RG + sub;
      const bool ok = i < n;
      const double x = __shfl_sync(0xffffffffu, a[r][0], sub * G);
      const double xm = ok && i > k + 1 ? x : 0.0;
#pragma unroll
      for (int q = 0; q < QL; ++q) {
        if (ok && c0 + G * q < K) A[(size_t)i * K + c0 + G * q] = a[r][q];
        acc[q] = fma(xm, a[r][q], acc[q]);
      }
      if (ok && gl == 0) vcol[i] = x;
      if (gl == 0) nsq = fma(xm, xm, nsq);
    }
  }
  // the row groups of a warp share its partial dots
#pragma unroll
  for (int o = 16; o >= G; o >>= 1) {
#pragma unroll
    for (int q = 0; q < QL; ++q) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
    nsq += __shfl_xor_sync(0xffffffffu, nsq, o);
  }
  if (sub == 0) {
#pragma unroll
    for (int q = 0; q < QL; ++q)
      if (c0 + G * q < K) wpart[warp * K + c0 + G * q] = acc[q];
  }
  return nsq;
}

template <int QL, int NQ, int G>
__device__ __forceinline__ double qr_dispatch(int ql, double* A, int n, int K, int k, double* vcol, const double* wv,
                                              double* wpart, int warp, int nw, int lane) {
  constexpr int R = QL <= 2 ? 4 : 2;
  if constexpr (QL == NQ) return qr_pass<QL, G, R>(A, n, K, k, vcol, wv, wpart, warp, nw, lane);
  else {
    if (ql <= QL) return qr_pass<QL, G, R>(A, n, K, k, vcol, wv, wpart, warp, nw, lane);
    return qr_dispatch<QL + 1, NQ, G>(ql, A, n, K, k, vcol, wv, wpart, warp, nw, lane);
  }
}
}  // namespace

// One CTA per (item, side).  The matrix lives in shared memory when it fits
// (K = 16: 8 KB at n = 64, several CTAs an SM), else in place in the level's
// X / Yt buffer (K = 256: 1.2 MB at n = 576, L2).  Bound by the FP64 pipe:
// 2 n K^2 - 2 K^3 / 3 FMAs; the reflector's square root and divisions run in
// one thread (a warp-wide FP64 instruction holds the pipe 16 cycles).
template <int NQ, int G>
__global__ void __launch_bounds__(256) k_lowrank_qr(LowRankQrArgs a, int use_smem) {
  extern __shared__ double sm[];
  const int n = a.n, K = a.K, tid = threadIdx.x, T = blockDim.x, nw = T >> 5;
  const int lane = tid & 31, warp = tid >> 5;
  const int64_t it = blockIdx.x, slot = (int64_t)blockIdx.y * a.S + it;
  double* Xg = (blockIdx.y == 0 ? a.X : a.Yt) + it * n * K;
  double* Vt = a.Vt + slot * K * n;
  double* taus = a.taus + slot * K;
  double* A = use_smem ? sm : Xg;
  double* vcol = use_smem ? sm + (size_t)n * K : sm;
  double* wv = vcol + n;
  double* wpart = wv + K;
  double* red = wpart + (size_t)nw * K;              // [nw] partial squares, then beta, tau, scale
  if (use_smem)
    for (int e = tid; e < n * K; e += T) A[e] = Xg[e];
  for (int e = tid; e < nw * K; e += T) wpart[e] = 0.0;
  __syncthreads();
  {
    // column 0 and its dots with the others: rows spread over the warps, every lane the columns l, l+32, ...
    double sq = 0.0;
    for (int i = tid; i < n; i += T) {
      const double x = A[(size_t)i * K];
      vcol[i] = x;
      if (i > 0) sq = fma(x, x, sq);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if (lane == 0) red[warp] = sq;
    for (int c = 1 + lane; c < K; c += 32) {
      double acc = 0.0;
      for (int i = 1 + warp; i < n; i += nw) acc = fma(A[(size_t)i * K], A[(size_t)i * K + c], acc);
      wpart[warp * K + c] = acc;
    }
  }
  __syncthreads();
  for (int k = 0; k < K; ++k) {
    if (tid == 0) {
      double xn2 = 0.0;
      for (int w = 0; w < nw; ++w) xn2 += red[w];
      const double alpha = vcol[k];
      double beta = alpha, tau = 0.0, scl = 0.0;
      if (xn2 > 0.0) {
        beta = -copysign(sqrt(fma(alpha, alpha, xn2)), alpha);
        tau = (beta - alpha) / beta;
        scl = 1.0 / (alpha - beta);
      }
      red[nw] = beta; red[nw + 1] = tau; red[nw + 2] = scl;
      taus[k] = tau;
    }
    __syncthreads();
    const double beta = red[nw], tau = red[nw + 1], scl = red[nw + 2];
    // v to the reflector store, zeros below the diagonal of R, w and row k of R
    for (int i = tid; i < n; i += T) {
      double v = i == k ? 1.0 : 0.0;
      if (i > k) {
        v = vcol[i] * scl;
        vcol[i] = v;
        if (i < K) A[(size_t)i * K + k] = 0.0;
      }
      Vt[(size_t)k * n + i] = v;
    }
    for (int c = k + 1 + tid; c < K; c += T) {
      double s = 0.0;
      for (int w = 0; w < nw; ++w) s += wpart[w * K + c];
      const double akc = A[(size_t)k * K + c];
      const double wc = tau * fma(scl, s, akc);
      wv[c] = wc;
      A[(size_t)k * K + c] = akc - wc;
    }
    if (tid == 0) A[(size_t)k * K + k] = beta;
    __syncthreads();
    if (k + 1 < K) {
      const int ql = (K - k - 1 + G - 1) / G;
      double nsq = qr_dispatch<1, NQ, G>(ql, A, n, K, k, vcol, wv, wpart, warp, nw, lane);
      if (lane == 0) red[warp] = nsq;
      __syncthreads();
    }
  }
  if (use_smem) {
    for (int e = tid; e < K * K; e += T) Xg[e] = A[e];
  }
}

// Vectors [c ; 0] through H_0 ... H_{K-1}, four per warp (their dots reduced
// together), a group of gs in shared memory.  grid (S, groups, 2): z = 0 the
// left half (Qx), z = 1 the right one (Qy).  4 n K kc flops per side.
__global__ void __launch_bounds__(128) k_lowrank_expand(LowRankExpandArgs a, int gs) {
  extern __shared__ double V[];                      // [gs][n]
  const int n = a.n, K = a.K, kc = a.kc, side = blockIdx.z, g0 = blockIdx.y * gs;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t it = blockIdx.x, slot = (int64_t)side * a.S + it;
  const int nv = min(gs, kc - g0);
  const double* hc = a.Hc + it * 2 * K * kc + (side ? (size_t)K * kc : 0);
  double* h = a.H + it * 2 * n * kc + (side ? (size_t)n * kc : 0);
  const double* Vt = a.Vt + slot * K * n;
  const double* taus = a.taus + slot * K;
  for (int e = threadIdx.x; e < nv * n; e += blockDim.x) {
    const int q = e / n, i = e - q * n;
    V[e] = i < K ? (side ? hc[(size_t)(g0 + q) * K + i] : hc[(size_t)i * kc + g0 + q]) : 0.0;
  }
  __syncthreads();
  const int a0 = warp * 4;
  if (a0 < nv) {
    double* V0 = V + (size_t)a0 * n;
    const int na = min(4, nv - a0);
    for (int k = K - 1; k >= 0; --k) {
      const double tau = taus[k];
      if (tau == 0.0) continue;
      const double* u = Vt + (size_t)k * n;
      double p0 = 0.0, p1 = 0.0, p2 = 0.0, p3 = 0.0;
      for (int j0 = k + lane; j0 < n; j0 += 256) {     // eight loads of the reflector in flight
        double uu[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) uu[c] = j0 + 32 * c < n ? u[j0 + 32 * c] : 0.0;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const int j = j0 + 32 * c;
          if (j >= n) break;
          p0 = fma(uu[c], V0[j], p0);
          if (na > 1) p1 = fma(uu[c], V0[n + j], p1);
          if (na > 2) p2 = fma(uu[c], V0[2 * n + j], p2);
          if (na > 3) p3 = fma(uu[c], V0[3 * n + j], p3);
        }
      }
      const double t = tau * reduce4(p0, p1, p2, p3, lane);
      const double w0 = __shfl_sync(0xffffffffu, t, 0), w1 = __shfl_sync(0xffffffffu, t, 8);
      const double w2 = __shfl_sync(0xffffffffu, t, 16), w3 = __shfl_sync(0xffffffffu, t, 24);
      for (int j0 = k + lane; j0 < n; j0 += 256) {
        double uu[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) uu[c] = j0 + 32 * c < n ? u[j0 + 32 * c] : 0.0;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const int j = j0 + 32 * c;
          if (j >= n) break;
          V0[j] = fma(-w0, uu[c], V0[j]);
          if (na > 1) V0[n + j] = fma(-w1, uu[c], V0[n + j]);
          if (na > 2) V0[2 * n + j] = fma(-w2, uu[c], V0[2 * n + j]);
          if (na > 3) V0[3 * n + j] = fma(-w3, uu[c], V0[3 * n + j]);
        }
      }
      __syncwarp();
    }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < nv * n; e += blockDim.x) {
    if (side) {
      h[(size_t)g0 * n + e] = V[e];
    } else {
      const int i = e / nv, q = e - i * nv;
      h[(size_t)i * kc + g0 + q] = V[(size_t)q * n + i];
    }
  }
}

template <int NQ, int G>
static cudaError_t launch_qr(const LowRankQrArgs& a, cudaStream_t st) {
  const size_t mat = (size_t)a.n * a.K;
  // few threads where a row group covers the columns: more CTAs an SM
  const int threads = a.n <= 64 && G == 16 ? 64 : (G == 16 ? 128 : 256);
  const size_t aux = qr_aux_doubles(a.n, a.K, threads / 32);
  const int use_smem = (mat + aux) * sizeof(double) <= kQrSmemCap;
  const size_t smem = ((use_smem ? mat : 0) + aux) * sizeof(double);
  static std::atomic<uint64_t> attr{0};
  cudaError_t e = raise_smem_limit(k_lowrank_qr<NQ, G>, (int)kQrSmemCap, attr);
  if (e != cudaSuccess) return e;
  k_lowrank_qr<NQ, G><<<dim3((unsigned)a.S, 2), threads, smem, st>>>(a, use_smem);
  return cudaGetLastError();
}

cudaError_t launch_lowrank_qr(const LowRankQrArgs& a, cudaStream_t st) {
  if (a.S <= 0) return cudaSuccess;
  if (!lowrank_supported(a.n, a.K)) return cudaErrorInvalidValue;
  if (a.K <= 17) return launch_qr<1, 16>(a, st);     // columns right of the first: at most 16
  if (a.K <= 65) return launch_qr<2, 32>(a, st);
  return launch_qr<8, 32>(a, st);
}

cudaError_t launch_lowrank_expand(const LowRankExpandArgs& a, cudaStream_t st) {
  if (a.S <= 0) return cudaSuccess;
  if (!lowrank_supported(a.n, a.K)) return cudaErrorInvalidValue;
  constexpr size_t kCap = 200 * 1024;
  int gs = (size_t)16 * a.n * sizeof(double) <= kCap ? 16 : 8;   // n <= 2304: 8 vectors take 147 KB
  // groups of four, a warp each, where the larger ones are fewer than the SMs (the same quads of vectors; 32
  // matrices of n = 576, 24 vectors: 3.2 -> 3.0 ms, and 1.7 with eight loads of a reflector in flight)
  if ((int64_t)a.S * 2 * ((a.kc + gs - 1) / gs) < 152) gs = 4;
  const size_t smem = (size_t)std::min(gs, a.kc) * a.n * sizeof(double);
  static std::atomic<uint64_t> attr{0};
  cudaError_t e = raise_smem_limit(k_lowrank_expand, (int)kCap, attr);
  if (e != cudaSuccess) return e;
  const dim3 grid((unsigned)a.S, (unsigned)((a.kc + gs - 1) / gs), 2);
  k_lowrank_expand<<<grid, 32 * ((std::min(gs, a.kc) + 3) / 4), smem, st>>>(a, gs);
  return cudaGetLastError();
}

}  // namespace mctrg
