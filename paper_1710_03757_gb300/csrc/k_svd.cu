// K2: batched FP64 one-sided Jacobi SVD (Sec. II, Eq. exactSVD).
//
// Hestenes' method applied to the rows: plane rotations from the left make
// the rows of M mutually orthogonal, J M = B, so the singular values are the
// row norms and the right singular vectors the normalized rows; the left
// vectors of the few kept indices are recovered later as u = M v / s.
// One-sided Jacobi computes small singular values to high relative accuracy,
// which matters here because the sampler divides kept values by inclusion
// rates that scale like s^2.
//
// One CTA per matrix.  The n_pad (even) rows are paired by the round-robin
// ("circle") ordering: n_pad - 1 steps per sweep, n_pad / 2 disjoint pairs per
// step handled by lane groups in parallel.  Rows live in shared memory when
// they fit (n <= 158), otherwise in the caller's global workspace, which the
// batch keeps L2-resident (one matrix per SM).  Stopping rule: a sweep with no
// rotation, where a pair is rotated iff |b_p . b_q| > n_pad 2^-53 |b_p| |b_q|
// (Demmel and Veselic 1992).  Row norms are recomputed exactly at the start
// of every sweep and at the end.  Rows whose norm is below (u/2) |M|_F, u the
// unit roundoff of the arithmetic that produced M (2^-52 for FP64), are
// rounding noise (they always end below the sampler's zero threshold): each
// sweep pairs only the remaining active rows, so a rank-r matrix costs
// O(r^2 n) per sweep instead of O(n^3).
#include <cooperative_groups.h>

#include <algorithm>
#include <cfloat>
#include <cmath>

#include "common.cuh"
#include "kernels.h"

namespace mctrg {

static __device__ __forceinline__ double group_sum(double v, int G) {
  for (int o = G >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Whether rows of squared norms al, be and product g are to be rotated, |g| >
// tol sqrt(al be), and the tangent t and cosine of the rotation that makes them
// orthogonal, in 25 FP64 instructions (three roots and three divisions are 120,
// and each holds the pipe 16 cycles per warp): with h = be - al and q = 2 g, t = sign(h) q / (|h| + sqrt(h^2 +
// q^2)) (Rutishauser's formula multiplied through by |q|).  Products leave the
// exponent range only for rows of extreme scale, which take the root or ratio
// form.  The squared test needs tol^2 al be normal too (tol >= 2^-52): a product
// al be of 2^-800 to 2^1000.  Below, the threshold and g^2 would underflow, which
// left rows of norms near 2^-250 unrotated up to a relative 2^-38.
__device__ __forceinline__ bool rotate_pair(double al, double be, double g, double tol) {
  const double ab = al * be;
  if ((unsigned)(((__double2hiint(ab) >> 20) & 0x7ff) - 223) < 1801u) return g * g > tol * tol * ab;
  return al > 0.0 && be > 0.0 && fabs(g) > tol * sqrt(al) * sqrt(be);
}
__device__ __forceinline__ void rotation(double al, double be, double g, double& t, double& cs) {
  const double h = be - al, q = 2.0 * g, s2 = fma(h, h, q * q);
  if (mid_range(s2)) {
    t = copysign(1.0, h) * q * inv(fabs(h) + s2 * inv_sqrt(s2));
  } else {
    const double zeta = h / q;
    if (fabs(zeta) > 1e150) t = 0.5 / zeta;
    else t = copysign(1.0, zeta) / (fabs(zeta) + sqrt(fma(zeta, zeta, 1.0)));
  }
  cs = inv_sqrt(fma(t, t, 1.0));
}

// n <= 32, one CTA per matrix, the rows in shared memory, G lanes per pair with
// at most two entries of a row each; every pair of a step has its lanes, so a
// step is one chain: dot product, rotation, update, barrier.  Bound by the
// latency of that chain (some thirty dependent FP64 operations): the rows'
// entries stay in registers from the dot product to the update, the next step's
// pair is fetched a step ahead (its place in the round-robin order moves by one),
// and the rotations are counted once a sweep (64 matrices of n = 16 in one launch
// 0.238 -> 0.213 ms).
template <int G>
__global__ void __launch_bounds__(256) k_jacobi(JacobiArgs a) {
  extern __shared__ double smem[];
  const double nu = a.noise_u > 0.0 ? a.noise_u : 0x1.0p-52;
  const int mat = blockIdx.x;
  const int n = a.n, np = a.n_pad;
  double* A = smem;
  double* nrm = smem + (size_t)np * n;
  int* act = (int*)(nrm + np);                      // [np + 1] active rows of a sweep
  const double* Mm = a.M + (size_t)mat * n * n;
  for (int idx = threadIdx.x; idx < np * n; idx += blockDim.x)
    A[idx] = idx < n * n ? Mm[idx] : 0.0;
  __syncthreads();

  const int gl = threadIdx.x & (G - 1);
  const int grp = threadIdx.x / G;
  const int ngrp = blockDim.x / G;
  const bool c0 = gl < n, c1 = gl + G < n;          // this lane's columns
  const double tol = (double)np * 0x1.0p-53;
  bool converged = false;
  __shared__ int s_na;
  __shared__ double s_thr2;

  for (int sweep = 0; sweep < a.max_sweeps && !converged; ++sweep) {
    for (int base = 0; base < np; base += ngrp) {
      int r = base + grp;
      double s = 0.0;
      if (r < np)
        for (int c = gl; c < n; c += G) { double v = A[(size_t)r * n + c]; s = fma(v, v, s); }
      s = group_sum(s, G);
      if (r < np && gl == 0) nrm[r] = s;
    }
    __syncthreads();
    if (threadIdx.x < 32) {                   // np <= 32: lane r holds row r
      const int r = threadIdx.x;
      const double v = r < np ? nrm[r] : 0.0;
      double thr2 = s_thr2;
      if (sweep == 0) {                       // |M|_F^2 is invariant under the rotations
        thr2 = group_sum(v, 32) * (0.25 * nu * nu);
        if (r == 0) s_thr2 = thr2;
      }
      const unsigned m = __ballot_sync(0xffffffffu, v > thr2);
      const int na = __popc(m);
      if (v > thr2) act[__popc(m & ((1u << r) - 1u))] = r;
      if (r == 0) {
        if (na & 1) act[na] = -1;
        s_na = na;
      }
    }
    __syncthreads();
    const int na = s_na, nap = na + (na & 1), npairs = nap >> 1;
    const bool mine = grp < npairs;
    // places of the pair in the order of the rows 1 .. nap-1, which turns by one a step
    int i1 = grp - 1, i2 = nap - 2 - grp, myrot = 0;
    int P = mine ? act[grp == 0 ? 0 : 1 + i1] : -1, Q = mine ? act[1 + i2] : -1;
    for (int step = 0; step + 1 < nap; ++step) {
      const bool act_pair = P >= 0 && Q >= 0;
      const int p = act_pair ? P : 0, q = act_pair ? Q : 0;
      double* ap = A + (size_t)p * n + gl;
      double* aq = A + (size_t)q * n + gl;
      const double x0 = c0 ? ap[0] : 0.0, y0 = c0 ? aq[0] : 0.0, x1 = c1 ? ap[G] : 0.0, y1 = c1 ? aq[G] : 0.0;
      const double al = act_pair ? nrm[p] : 0.0, be = act_pair ? nrm[q] : 0.0;
      if (mine) {                                  // the next step's pair
        if (++i1 == nap - 1) i1 = 0;
        if (++i2 == nap - 1) i2 = 0;
        if (grp > 0) P = act[1 + i1];
        Q = act[1 + i2];
      }
      const double g = group_sum(act_pair ? fma(x1, y1, x0 * y0) : 0.0, G);   // every lane of the warp takes part
      const bool rot = act_pair && rotate_pair(al, be, g, tol);
      double nal = al, nbe = be, u0 = 0.0, u1 = 0.0, v0 = 0.0, v1 = 0.0;
      if (rot) {                                   // uniform within the lane group
        double t, cs;
        rotation(al, be, g, t, cs);
        const double sn = cs * t;
        u0 = fma(-sn, y0, cs * x0);
        u1 = fma(-sn, y1, cs * x1);
        v0 = fma(sn, x0, cs * y0);
        v1 = fma(sn, x1, cs * y1);
        if (c0) { ap[0] = u0; aq[0] = v0; }
        if (c1) { ap[G] = u1; aq[G] = v1; }
        nal = fma(-t, g, al);
        nbe = fma(t, g, be);
        ++myrot;
      }
      // heavy cancellation in the norm update: recompute from the rotated rows
      const bool fixP = rot && nal < 0.01 * al, fixQ = rot && nbe < 0.01 * be;
      if (__any_sync(0xffffffffu, fixP || fixQ)) {
        const double sp = group_sum(fma(u1, u1, u0 * u0), G), sq = group_sum(fma(v1, v1, v0 * v0), G);
        if (fixP) nal = sp;
        if (fixQ) nbe = sq;
      }
      if (rot && gl == 0) { nrm[p] = nal; nrm[q] = nbe; }
      __syncthreads();
    }
    converged = !__syncthreads_or(myrot);
  }

  // exact final norms
  for (int base = 0; base < np; base += ngrp) {
    int r = base + grp;
    double s = 0.0;
    if (r < np)
      for (int c = gl; c < n; c += G) { double v = A[(size_t)r * n + c]; s = fma(v, v, s); }
    s = group_sum(s, G);
    if (r < np && gl == 0) nrm[r] = sqrt(s);
  }
  __syncthreads();
  // rank sort, descending; ties keep row order
  double* sg = a.sig + (size_t)mat * np;
  int* pm = a.perm + (size_t)mat * np;
  for (int r = threadIdx.x; r < np; r += blockDim.x) {
    const double v = nrm[r];
    int rank = 0;
    for (int j = 0; j < np; ++j) {
      const double u = nrm[j];
      rank += (u > v) || (u == v && j < r);
    }
    sg[rank] = v;
    pm[rank] = r;
  }
  double* Wm = a.W + (size_t)mat * np * n;
  for (int idx = threadIdx.x; idx < np * n; idx += blockDim.x) Wm[idx] = A[idx];
  __syncthreads();
  if (threadIdx.x == 0) {
    double s1 = sg[0];
    if (a.lns1) a.lns1[mat] = s1 > 0.0 ? log(s1) : -INFINITY;
    const double tau = (a.zero_rel > 0.0 ? a.zero_rel : (double)n * 0x1.0p-52) * s1;
    int cnt = 0;
    for (int r = 0; r < np; ++r) cnt += sg[r] > tau;
    a.nnz[mat] = s1 > 0.0 ? cnt : 0;
    if (a.mflags && !converged) a.mflags[mat] |= FLAG_NOCONV;
  }
}

// ---------------------------------------------------------------------------
// Warp-batched variant for n > 32 (one lane group = the whole warp).
//
// Each warp takes PW disjoint pairs of a round-robin step.  Their PW dot
// products are reduced together by recursive halving (lane bit 4 picks the
// upper or lower half of the pair set, then bit 3, ...), which costs about
// PW additions per lane instead of 5 PW, and leaves the total of pair
// j = lane >> (5 - log2 PW) in every lane; each lane then computes the
// rotation of "its" pair, so the divisions and square roots are shared by
// the PW pairs.  Rotations use scaled rows (Anda and Park 1994, fast plane
// rotations): the true row is d_r * row_r; the rotation by tangent t,
// cosine c becomes
//   row_p <- row_p - t (d_q / d_p) row_q,  row_q <- row_q + t (d_p / d_q) row_p,
//   d_p <- c d_p,  d_q <- c d_q,
// two FMAs per element instead of four.  With |t| <= 1 each rotation scales
// d by at least 2^-1/2, and the scales are folded back into the rows at every
// sweep start, so d stays above 2^-(n-1)/2.  True squared norms are carried
// separately and recomputed exactly at every sweep start.
template <int PW>
__device__ __forceinline__ double batched_reduce(double (&v)[PW], int lane) {
  int cnt = PW;
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    if (cnt > 1) {
      const int half = cnt >> 1;
      const bool upper = (lane & o) != 0;
#pragma unroll
      for (int k = 0; k < PW / 2; ++k) {
        if (k < half) {
          const double send = upper ? v[k] : v[k + half];
          const double keep = upper ? v[k + half] : v[k];
          v[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
      }
      cnt = half;
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    }
  }
  return v[0];
}

// Householder QR with column pivoting of the np x n row-major matrix A
// (Businger and Golub 1965; norm downdating with the safeguard of LAPACK's
// xLAQP2): A P = Q R, R overwrites A (zeros below the diagonal), Q is not
// formed and colperm[c] = original column of column c.  The singular values
// of R are those of M, and a right singular vector v~ of R gives v = P v~ for
// M.  The rows of R are graded (|r_kk| decreasing), which cuts one-sided
// Jacobi from ~40 sweeps to ~9 on the TRG level matrices (Drmac and Veselic
// 2008, preconditioned Jacobi).
__device__ void qrcp_rows(double* A, int n, int np, int* colperm, double* cn, double* cn0, double* vbuf,
                          double* redv, int* redi) {
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  for (int j = tid; j < n; j += nt) {
    double s = 0.0;
    for (int i = 0; i < np; ++i) { const double v = A[(size_t)i * n + j]; s = fma(v, v, s); }
    cn[j] = sqrt(s);
    cn0[j] = cn[j];
    colperm[j] = j;
  }
  __syncthreads();
  for (int k = 0; k < n; ++k) {
    // pivot: largest remaining column norm, ties to the smallest index
    double best = -1.0;
    int bj = n;
    for (int j = k + tid; j < n; j += nt) {
      const double v = cn[j];
      if (v > best) { best = v; bj = j; }
    }
    for (int o = 16; o > 0; o >>= 1) {
      const double ob = __shfl_xor_sync(0xffffffffu, best, o);
      const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
      if (ob > best || (ob == best && oj < bj)) { best = ob; bj = oj; }
    }
    if (lane == 0) { redv[warp] = best; redi[warp] = bj; }
    __syncthreads();
    if (tid == 0) {
      double b = redv[0];
      int q = redi[0];
      for (int w = 1; w < nw; ++w)
        if (redv[w] > b || (redv[w] == b && redi[w] < q)) { b = redv[w]; q = redi[w]; }
      redi[32] = q;
    }
    __syncthreads();
    const int p = redi[32];
    if (p != k && p < n) {
      for (int i = tid; i < np; i += nt) {
        const double t = A[(size_t)i * n + k];
        A[(size_t)i * n + k] = A[(size_t)i * n + p];
        A[(size_t)i * n + p] = t;
      }
      if (tid == 0) {
        double t = cn[k]; cn[k] = cn[p]; cn[p] = t;
        t = cn0[k]; cn0[k] = cn0[p]; cn0[p] = t;
        const int c = colperm[k]; colperm[k] = colperm[p]; colperm[p] = c;
      }
    }
    __syncthreads();
    // Householder reflector of column k below the diagonal
    double s = 0.0;
    for (int i = k + 1 + tid; i < np; i += nt) { const double v = A[(size_t)i * n + k]; s = fma(v, v, s); }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) redv[warp] = s;
    __syncthreads();
    double xn2 = 0.0;
    for (int w = 0; w < nw; ++w) xn2 += redv[w];
    const double alpha = A[(size_t)k * n + k];
    double tau = 0.0, beta = alpha;
    if (xn2 > 0.0) {
      beta = -copysign(sqrt(fma(alpha, alpha, xn2)), alpha);
      tau = (beta - alpha) / beta;
      const double scal = 1.0 / (alpha - beta);
      for (int i = k + 1 + tid; i < np; i += nt) vbuf[i] = A[(size_t)i * n + k] * scal;
    }
    __syncthreads();
    for (int i = k + 1 + tid; i < np; i += nt) A[(size_t)i * n + k] = 0.0;
    if (tid == 0) A[(size_t)k * n + k] = beta;
    // apply (I - tau v v^T) to the trailing columns and downdate their norms
    for (int j = k + 1 + tid; j < n; j += nt) {
      double akj = A[(size_t)k * n + j];
      if (tau != 0.0) {
        double w = akj;
#pragma unroll 8
        for (int i = k + 1; i < np; ++i) w = fma(vbuf[i], A[(size_t)i * n + j], w);
        w *= tau;
        akj -= w;
        A[(size_t)k * n + j] = akj;
#pragma unroll 8
        for (int i = k + 1; i < np; ++i) A[(size_t)i * n + j] = fma(-vbuf[i], w, A[(size_t)i * n + j]);
      }
      const double c = cn[j];
      if (c != 0.0) {
        double t = fabs(akj) / c;
        t = fmax(0.0, (1.0 - t) * (1.0 + t));
        const double r = c / cn0[j];
        if (t * r * r <= 1.4901161193847656e-08) {
          double s2 = 0.0;
          for (int i = k + 1; i < np; ++i) { const double v = A[(size_t)i * n + j]; s2 = fma(v, v, s2); }
          cn[j] = sqrt(s2);
          cn0[j] = cn[j];
        } else {
          cn[j] = c * sqrt(t);
        }
      }
    }
    __syncthreads();
  }
}

template <int PW>
__global__ void __launch_bounds__(512) k_jacobi_warp(JacobiArgs a, int use_smem) {
  extern __shared__ double smem[];
  const double nu = a.noise_u > 0.0 ? a.noise_u : 0x1.0p-52;
  __shared__ int s_rot, s_na;
  __shared__ double s_thr2;
  constexpr int LOGPW = PW == 1 ? 0 : PW == 2 ? 1 : PW == 4 ? 2 : PW == 8 ? 3 : PW == 16 ? 4 : 5;
  constexpr int SH = 5 - LOGPW;                    // lane >> SH = pair index within the warp
  const int mat = blockIdx.x;
  const int n = a.n, np = a.n_pad;
  double* A = use_smem ? smem : a.W + (size_t)mat * np * n;
  double* nrm = use_smem ? smem + (size_t)np * n : smem;
  double* dsc = nrm + np;                          // [np] row scales
  double* cn = dsc + np;                           // [np] column norms (QR)
  double* cn0 = cn + np;                           // [np] reference norms (QR)
  double* vbuf = cn0 + np;                         // [np] Householder vector
  double* redv = vbuf + np;                        // [33] block reductions
  double* wbuf = redv + 34;                        // global rows: [nwarps][n] row staging
  int* act = (int*)(wbuf + (use_smem ? 0 : (size_t)(blockDim.x >> 5) * n));   // [np + 1] active rows
  int* colperm = act + np + 2;                     // [np] column permutation of R
  int* redi = colperm + np;                        // [33]
  const double* Mm = a.M + (size_t)mat * n * n;
  for (int idx = threadIdx.x; idx < np * n; idx += blockDim.x) A[idx] = idx < n * n ? Mm[idx] : 0.0;
  for (int r = threadIdx.x; r < np; r += blockDim.x) dsc[r] = 1.0;
  __syncthreads();
  qrcp_rows(A, n, np, colperm, cn, cn0, vbuf, redv, redi);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const double tol = (double)np * 0x1.0p-53;
  bool converged = false;

  for (int sweep = 0; sweep < a.max_sweeps && !converged; ++sweep) {
    // fold the scales into the rows and take exact squared norms
    for (int r = warp; r < np; r += nwarps) {
      const double dr = dsc[r];
      double s = 0.0;
      double* row = A + (size_t)r * n;
      for (int c = lane; c < n; c += 32) {
        double v = row[c];
        if (dr != 1.0) { v *= dr; row[c] = v; }
        s = fma(v, v, s);
      }
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) { nrm[r] = s; dsc[r] = 1.0; }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      if (sweep == 0) {
        double f = 0.0;
        for (int r = 0; r < np; ++r) f += nrm[r];
        s_thr2 = f * (0.25 * nu * nu);
      }
      int na = 0;
      for (int r = 0; r < np; ++r)
        if (nrm[r] > s_thr2) act[na++] = r;
      if (na & 1) act[na] = -1;
      s_na = na;
      s_rot = 0;
    }
    __syncthreads();
    const int na = s_na, nap = na + (na & 1), npairs = nap >> 1;
    for (int step = 0; step + 1 < nap; ++step) {
      int myrot = 0;
      for (int base = warp * PW; base < npairs; base += nwarps * PW) {
        int Pj[PW], Qj[PW];
        double g[PW];
#pragma unroll
        for (int j = 0; j < PW; ++j) {
          const int pk = base + j;
          int P = -1, Q = -1;
          if (pk < npairs) {
            P = act[pk == 0 ? 0 : 1 + (pk - 1 + step) % (nap - 1)];
            Q = act[1 + (nap - 2 - pk + step) % (nap - 1)];
          }
          Pj[j] = P; Qj[j] = Q;
          double acc = 0.0;
          if (P >= 0 && Q >= 0) {
            const double* ap = A + (size_t)P * n;
            const double* aq = A + (size_t)Q * n;
            for (int c = lane; c < n; c += 32) acc = fma(ap[c], aq[c], acc);
          }
          g[j] = acc;
        }
        const double gs = batched_reduce<PW>(g, lane);
        // this lane's pair
        const int jm = lane >> SH;
        int P = -1, Q = -1;
#pragma unroll
        for (int j = 0; j < PW; ++j) if (j == jm) { P = Pj[j]; Q = Qj[j]; }
        bool rot = false;
        double mu1 = 0.0, mu2 = 0.0, cs = 1.0, nal = 0.0, nbe = 0.0, al = 0.0, be = 0.0;
        if (P >= 0 && Q >= 0) {
          al = nrm[P]; be = nrm[Q];
          const double dp = dsc[P], dq = dsc[Q];
          const double gam = dp * dq * gs;
          rot = rotate_pair(al, be, gam, tol);
          if (rot) {
            double t;
            rotation(al, be, gam, t, cs);
            mu1 = t * (dq * inv(dp));
            mu2 = t * (dp * inv(dq));
            nal = fma(-t, gam, al);
            nbe = fma(t, gam, be);
          }
        }
        bool fixany = false;
#pragma unroll
        for (int j = 0; j < PW; ++j) {
          const int src = j << SH;
          const bool rj = __shfl_sync(0xffffffffu, rot, src);
          if (!rj) continue;                                   // warp-uniform
          const double m1 = __shfl_sync(0xffffffffu, mu1, src);
          const double m2 = __shfl_sync(0xffffffffu, mu2, src);
          double* ap = A + (size_t)Pj[j] * n;
          double* aq = A + (size_t)Qj[j] * n;
          for (int c = lane; c < n; c += 32) {
            const double x = ap[c], y = aq[c];
            ap[c] = fma(-m1, y, x);
            aq[c] = fma(m2, x, y);
          }
        }
        const bool own = (lane & ((1 << SH) - 1)) == 0;
        const bool fixP = rot && nal < 0.01 * al, fixQ = rot && nbe < 0.01 * be;
        if (own && rot) {
          nrm[P] = nal; nrm[Q] = nbe;
          dsc[P] *= cs; dsc[Q] *= cs;
          ++myrot;
        }
        fixany = __any_sync(0xffffffffu, fixP || fixQ);
        if (fixany) {                                          // rare: recompute from the rows
          __syncwarp();
#pragma unroll
          for (int j = 0; j < PW; ++j) {
            const int src = j << SH;
            const bool fp = __shfl_sync(0xffffffffu, fixP, src), fq = __shfl_sync(0xffffffffu, fixQ, src);
            for (int side = 0; side < 2; ++side) {
              if (!(side == 0 ? fp : fq)) continue;            // warp-uniform
              const int r = side == 0 ? Pj[j] : Qj[j];
              const double* row = A + (size_t)r * n;
              const double dr = dsc[r];
              double s = 0.0;
              for (int c = lane; c < n; c += 32) s = fma(row[c], row[c], s);
              for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
              if (lane == 0) nrm[r] = s * dr * dr;
            }
          }
          __syncwarp();
        }
      }
      if (myrot) atomicAdd(&s_rot, myrot);
      __syncthreads();
    }
    converged = (s_rot == 0);
    __syncthreads();
  }
  // true rows and exact norms
  for (int r = warp; r < np; r += nwarps) {
    const double dr = dsc[r];
    double s = 0.0;
    double* row = A + (size_t)r * n;
    for (int c = lane; c < n; c += 32) {
      double v = row[c];
      if (dr != 1.0) { v *= dr; row[c] = v; }
      s = fma(v, v, s);
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) nrm[r] = sqrt(s);
  }
  __syncthreads();
  double* sg = a.sig + (size_t)mat * np;
  int* pm = a.perm + (size_t)mat * np;
  for (int r = threadIdx.x; r < np; r += blockDim.x) {
    const double v = nrm[r];
    int rank = 0;
    for (int j = 0; j < np; ++j) {
      const double u = nrm[j];
      rank += (u > v) || (u == v && j < r);
    }
    sg[rank] = v;
    pm[rank] = r;
  }
  // rows of W are right vectors of M: undo the column pivoting of R
  if (use_smem) {
    double* Wm = a.W + (size_t)mat * np * n;
    for (int idx = threadIdx.x; idx < np * n; idx += blockDim.x) {
      const int r = idx / n, c = idx - r * n;
      Wm[(size_t)r * n + colperm[c]] = A[idx];
    }
  } else {
    double* buf = wbuf + (size_t)warp * n;
    for (int r = warp; r < np; r += nwarps) {
      double* row = A + (size_t)r * n;
      for (int c = lane; c < n; c += 32) buf[c] = row[c];
      __syncwarp();
      for (int c = lane; c < n; c += 32) row[colperm[c]] = buf[c];
      __syncwarp();
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const double s1 = sg[0];
    if (a.lns1) a.lns1[mat] = s1 > 0.0 ? log(s1) : -INFINITY;
    const double tau = (a.zero_rel > 0.0 ? a.zero_rel : (double)n * 0x1.0p-52) * s1;
    int cnt = 0;
    for (int r = 0; r < np; ++r) cnt += sg[r] > tau;
    a.nnz[mat] = s1 > 0.0 ? cnt : 0;
    if (a.mflags && !converged) a.mflags[mat] |= FLAG_NOCONV;
  }
}

// ---------------------------------------------------------------------------
// Cluster variant for launches of a few matrices (the shared prefix of a
// context: two matrices of up to n = 1024, every nonzero vector needed): eight
// CTAs on eight SMs share one matrix, whose rows stay in the global workspace
// (L2; read past L1, since another SM wrote them a step ago), with the row
// norms and scales in the first CTA's shared memory.  The method is
// k_jacobi_warp's -- QR with column pivoting, then scaled plane rotations -- and
// so is every pair's arithmetic.
//   QR: column j belongs to CTA j mod 8.  One or two cluster barriers per step:
//   after the CTAs have applied the reflector to their columns and offered their
//   largest remaining norm; after a pivot column has been exchanged (rows
//   spread over the CTAs).  Each CTA forms the reflector itself, and column k
//   is overwritten with its part of R after the last step only.
//   Sweeps: the pairs of a step are spread over 8 x 4 warps, one cluster
//   barrier per step; a warp's rows stay in registers between the dot and the
//   rotation where they fit (NQ > 0: sides up to 32 NQ).
// FP64-issue bound in one CTA (225 M FMAs of rotations at n = 256, 54 ms at one
// SM's rate).  The two matrices of n = 256 of a chi = 16 context's last exact
// level (rank 16) and first sampled one (full rank): its set-up 104 -> 23 ms.
constexpr int kJcCtas = 8, kJcThreads = 256, kJcWarps = 4;   // warps that rotate
constexpr int kJcMinN = 64;
namespace cg = cooperative_groups;

struct JacobiClusterShared {
  // (rank 0) largest remaining column norm of each CTA, and its index; the two
  // halves in turn, since a step without an exchange has one barrier only: a
  // CTA may offer step k+1's while another still reads step k's
  double cand[2][kJcCtas];
  int cidx[2][kJcCtas];
  int rot, na;
  double thr2;
};

template <int PW, int NQ>
__global__ void __cluster_dims__(kJcCtas, 1, 1) __launch_bounds__(kJcThreads) k_jacobi_cluster(JacobiArgs a) {
  extern __shared__ double smem[];
  __shared__ JacobiClusterShared sh;
  __shared__ double redv[33];
  __shared__ int redi[33];
  constexpr int LOGPW = PW == 1 ? 0 : PW == 2 ? 1 : PW == 4 ? 2 : PW == 8 ? 3 : 4;
  constexpr int SH = 5 - LOGPW;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank();
  const int mat = blockIdx.x / kJcCtas, n = a.n, np = a.n_pad;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockDim.x, nw = nt >> 5;
  const double nu = a.noise_u > 0.0 ? a.noise_u : 0x1.0p-52;
  double* A = a.W + (size_t)mat * np * n;
  // shared by the cluster, in rank 0: squared norms, scales, column norms, column permutation
  double* nrm_l = smem;
  double* dsc_l = nrm_l + np;
  double* cn_l = dsc_l + np;
  double* cn0_l = cn_l + np;
  int* perm_l = (int*)(cn0_l + np);
  double* vbuf = (double*)(perm_l + np + (np & 1));   // this CTA's copy of the reflector, then row staging
  int* act = (int*)(vbuf + np);                       // [np + 1]
  double* wpart = (double*)(act + np + 2);            // [nw + 1][32 columns] (np is even)
  double* diag = wpart + (nw + 1) * 32;               // [np] diagonal of R
  double* nrm = cl.map_shared_rank(nrm_l, 0);
  double* dsc = cl.map_shared_rank(dsc_l, 0);
  double* cn = cl.map_shared_rank(cn_l, 0);
  double* cn0 = cl.map_shared_rank(cn0_l, 0);
  int* colperm = cl.map_shared_rank(perm_l, 0);
  JacobiClusterShared* s0 = cl.map_shared_rank(&sh, 0);
  const double* Mm = a.M + (size_t)mat * n * n;
  for (int64_t e = rank * nt + tid; e < (int64_t)np * n; e += kJcCtas * nt) A[e] = e < (int64_t)n * n ? Mm[e] : 0.0;
  cl.sync();
  // ---- QR with column pivoting (Businger and Golub; LAPACK xLAQP2's norm downdating)
  for (int j = rank + kJcCtas * tid; j < n; j += kJcCtas * nt) {
    double s = 0.0;
#pragma unroll 8
    for (int i = 0; i < np; ++i) { const double v = __ldcg(A + (size_t)i * n + j); s = fma(v, v, s); }
    const double c = sqrt(s);
    cn[j] = c;
    cn0[j] = c;
    colperm[j] = j;
  }
  cl.sync();
  {  // |M|_F^2, the same sum in every CTA
    double f = 0.0;
    for (int j = tid; j < n; j += nt) f = fma(cn0[j], cn0[j], f);
    for (int o = 16; o > 0; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
    if (lane == 0) redv[warp] = f;
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int w = 0; w < nw; ++w) t += redv[w];
      sh.thr2 = t * (0.25 * nu * nu);
    }
    cl.sync();                                        // all have read cn0 before it is downdated
  }
  int kend = n;                                       // columns of R that have been reached
  for (int k = 0; k < n; ++k) {
    {  // this CTA's largest remaining norm, ties to the smallest index
      double best = -1.0;
      int bj = n;
      for (int j = rank + kJcCtas * tid; j < n; j += kJcCtas * nt) {
        if (j < k) continue;
        const double v = cn[j];
        if (v > best) { best = v; bj = j; }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const double ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
        if (ob > best || (ob == best && oj < bj)) { best = ob; bj = oj; }
      }
      if (lane == 0) { redv[warp] = best; redi[warp] = bj; }
      __syncthreads();
      if (tid == 0) {
        double b = redv[0];
        int q = redi[0];
        for (int w = 1; w < nw; ++w)
          if (redv[w] > b || (redv[w] == b && redi[w] < q)) { b = redv[w]; q = redi[w]; }
        s0->cand[k & 1][rank] = b;
        s0->cidx[k & 1][rank] = q;
      }
    }
    cl.sync();
    if (tid == 0) {
      double b = s0->cand[k & 1][0];
      int q = s0->cidx[k & 1][0];
      for (int w = 1; w < kJcCtas; ++w) {
        const double v = s0->cand[k & 1][w];
        const int i = s0->cidx[k & 1][w];
        if (v > b || (v == b && i < q)) { b = v; q = i; }
      }
      redi[32] = q;
      redv[32] = b;
    }
    __syncthreads();
    // what is left is noise (its rows are below the level that the sweeps leave
    // out): a matrix of rank r needs r steps.  The same decision in every CTA
    if (redv[32] * redv[32] * (double)(n - k) <= sh.thr2) { kend = k; break; }
    const int p = redi[32];
    if (p != k && p < n) {
      for (int i = rank * nt + tid; i < np; i += kJcCtas * nt) {
        const double t = __ldcg(A + (size_t)i * n + k);
        A[(size_t)i * n + k] = __ldcg(A + (size_t)i * n + p);
        A[(size_t)i * n + p] = t;
      }
      if (rank == 0 && tid == 0) {
        double t = cn[k]; cn[k] = cn[p]; cn[p] = t;
        t = cn0[k]; cn0[k] = cn0[p]; cn0[p] = t;
        const int c = colperm[k]; colperm[k] = colperm[p]; colperm[p] = c;
      }
      cl.sync();
    }
    // reflector of column k below the diagonal, formed by every CTA
    double s = 0.0;
    for (int i = k + tid; i < np; i += nt) {
      const double v = __ldcg(A + (size_t)i * n + k);
      vbuf[i] = v;
      if (i > k) s = fma(v, v, s);
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) redv[warp] = s;
    __syncthreads();
    if (tid == 0) {
      double xn2 = 0.0;
      for (int w = 0; w < nw; ++w) xn2 += redv[w];
      const double alpha = vbuf[k];
      double tau = 0.0, beta = alpha, scl = 0.0;
      if (xn2 > 0.0) {
        beta = -copysign(sqrt(fma(alpha, alpha, xn2)), alpha);
        tau = (beta - alpha) / beta;
        scl = 1.0 / (alpha - beta);
      }
      redv[30] = tau; redv[31] = scl; redv[32] = beta;
    }
    __syncthreads();
    const double tau = redv[30], scl = redv[31], beta = redv[32];
    for (int i = k + tid; i < np; i += nt) vbuf[i] = i == k ? 1.0 : vbuf[i] * scl;
    if (tid == 0) diag[k] = beta;
    __syncthreads();
    // own columns, 32 at a time: lane = column, the warps share the rows
    for (int j0 = 0; j0 < n; j0 += 32 * kJcCtas) {
      const int j = j0 + rank + kJcCtas * lane;
      if (j0 + 32 * kJcCtas <= k + 1) continue;       // finished columns
      const bool on = j > k && j < n;
      double w = 0.0;
      if (on && tau != 0.0) {
#pragma unroll 8
        for (int i = k + warp; i < np; i += nw) w = fma(vbuf[i], __ldcg(A + (size_t)i * n + j), w);
      }
      wpart[warp * 32 + lane] = w;
      __syncthreads();
      w = 0.0;
      for (int q = 0; q < nw; ++q) w += wpart[q * 32 + lane];
      w *= tau;
      if (on && tau != 0.0) {
        for (int i0 = k + warp; i0 < np; i0 += 8 * nw) {
          double y[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const int i = i0 + q * nw;
            y[q] = i < np ? fma(-vbuf[i], w, __ldcg(A + (size_t)i * n + j)) : 0.0;
          }
#pragma unroll
          for (int q = 0; q < 8; ++q)
            if (i0 + q * nw < np) A[(size_t)(i0 + q * nw) * n + j] = y[q];
          if (i0 == k) wpart[nw * 32 + lane] = y[0];  // the new entry of row k
        }
      } else if (on && warp == 0) {
        wpart[nw * 32 + lane] = __ldcg(A + (size_t)k * n + j);
      }
      __syncthreads();
      if (on && warp == 0) {                          // downdate the norm
        const double akj = wpart[nw * 32 + lane], c = cn[j];
        if (c != 0.0) {
          double t = fabs(akj) / c;
          t = fmax(0.0, (1.0 - t) * (1.0 + t));
          const double r = c / cn0[j];
          if (t * r * r <= 1.4901161193847656e-08) {
            double s2 = 0.0;
#pragma unroll 8
            for (int i = k + 1; i < np; ++i) { const double v = __ldcg(A + (size_t)i * n + j); s2 = fma(v, v, s2); }
            cn[j] = sqrt(s2);
            cn0[j] = cn[j];
          } else {
            cn[j] = c * sqrt(t);
          }
        }
      }
      __syncthreads();
    }
  }
  cl.sync();
  for (int64_t e = rank * nt + tid; e < (int64_t)np * n; e += kJcCtas * nt) {   // R below and on the diagonal
    const int i = (int)(e / n), j = (int)(e - (int64_t)i * n);
    if (j <= i && j < kend) A[e] = j == i ? diag[j] : 0.0;
  }
  cl.sync();
  // ---- sweeps
  const double tol = (double)np * 0x1.0p-53;
  bool converged = false;
  for (int r = rank * nw + warp; r < np; r += kJcCtas * nw)
    if (lane == 0) dsc[r] = 1.0;
  cl.sync();
  for (int sweep = 0; sweep < a.max_sweeps && !converged; ++sweep) {
    // fold the scales into the rows and take exact squared norms
    for (int r = rank * nw + warp; r < np; r += kJcCtas * nw) {
      const double dr = dsc[r];
      double s = 0.0;
      double* row = A + (size_t)r * n;
      for (int c = lane; c < n; c += 32) {
        double v = __ldcg(row + c);
        if (dr != 1.0) { v *= dr; row[c] = v; }
        s = fma(v, v, s);
      }
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      __syncwarp();
      if (lane == 0) { nrm[r] = s; dsc[r] = 1.0; }
    }
    if (rank == 0 && tid == 0) sh.rot = 0;
    cl.sync();
    // every CTA makes the same list of active rows
    for (int r = tid; r < np; r += nt) vbuf[r] = nrm[r];
    __syncthreads();
    if (tid == 0) {
      if (sweep == 0) {
        double f = 0.0;
        for (int r = 0; r < np; ++r) f += vbuf[r];
        sh.thr2 = f * (0.25 * nu * nu);
      }
      int na = 0;
      for (int r = 0; r < np; ++r)
        if (vbuf[r] > sh.thr2) act[na++] = r;
      if (na & 1) act[na] = -1;
      sh.na = na;
    }
    cl.sync();                                        // every CTA has its list: the norms may change
    const int na = sh.na, nap = na + (na & 1), npairs = nap >> 1;
    for (int step = 0; step + 1 < nap; ++step) {
      int myrot = 0;
      for (int base = (rank * kJcWarps + warp) * PW; warp < kJcWarps && base < npairs;
           base += kJcCtas * kJcWarps * PW) {
        int Pj[PW], Qj[PW];
        double g[PW], xr[PW][NQ > 0 ? NQ : 1], yr[PW][NQ > 0 ? NQ : 1];
#pragma unroll
        for (int j = 0; j < PW; ++j) {
          const int pk = base + j;
          int P = -1, Q = -1;
          if (pk < npairs) {
            P = act[pk == 0 ? 0 : 1 + (pk - 1 + step) % (nap - 1)];
            Q = act[1 + (nap - 2 - pk + step) % (nap - 1)];
          }
          Pj[j] = P; Qj[j] = Q;
          double acc = 0.0;
          const bool in = P >= 0 && Q >= 0;
          const double* ap = A + (size_t)(in ? P : 0) * n;
          const double* aq = A + (size_t)(in ? Q : 0) * n;
          if constexpr (NQ > 0) {
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
              const int c = lane + 32 * q;
              xr[j][q] = in && c < n ? __ldcg(ap + c) : 0.0;
              yr[j][q] = in && c < n ? __ldcg(aq + c) : 0.0;
            }
#pragma unroll
            for (int q = 0; q < NQ; ++q) acc = fma(xr[j][q], yr[j][q], acc);
          } else if (in) {
#pragma unroll 8
            for (int c = lane; c < n; c += 32) acc = fma(__ldcg(ap + c), __ldcg(aq + c), acc);
          }
          g[j] = acc;
        }
        const double gs = batched_reduce<PW>(g, lane);
        const int jm = lane >> SH;                     // this lane's pair
        int P = -1, Q = -1;
#pragma unroll
        for (int j = 0; j < PW; ++j) if (j == jm) { P = Pj[j]; Q = Qj[j]; }
        bool rot = false;
        double mu1 = 0.0, mu2 = 0.0, cs = 1.0, nal = 0.0, nbe = 0.0, al = 0.0, be = 0.0, dp = 1.0, dq = 1.0;
        if (P >= 0 && Q >= 0) {
          al = nrm[P]; be = nrm[Q];
          dp = dsc[P]; dq = dsc[Q];
          const double gam = dp * dq * gs;
          rot = rotate_pair(al, be, gam, tol);
          if (rot) {
            double t;
            rotation(al, be, gam, t, cs);
            mu1 = t * (dq * inv(dp));
            mu2 = t * (dp * inv(dq));
            nal = fma(-t, gam, al);
            nbe = fma(t, gam, be);
          }
        }
#pragma unroll
        for (int j = 0; j < PW; ++j) {
          const int src = j << SH;
          if (!__shfl_sync(0xffffffffu, rot, src)) continue;   // warp-uniform
          const double m1 = __shfl_sync(0xffffffffu, mu1, src);
          const double m2 = __shfl_sync(0xffffffffu, mu2, src);
          double* ap = A + (size_t)Pj[j] * n;
          double* aq = A + (size_t)Qj[j] * n;
          if constexpr (NQ > 0) {
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
              const int c = lane + 32 * q;
              if (c < n) {
                ap[c] = fma(-m1, yr[j][q], xr[j][q]);
                aq[c] = fma(m2, xr[j][q], yr[j][q]);
              }
            }
          } else {
            for (int c0 = lane; c0 < n; c0 += 32 * 8) {
              double x[8], y[8];
#pragma unroll
              for (int q = 0; q < 8; ++q) {
                const int c = c0 + 32 * q;
                x[q] = c < n ? __ldcg(ap + c) : 0.0;
                y[q] = c < n ? __ldcg(aq + c) : 0.0;
              }
#pragma unroll
              for (int q = 0; q < 8; ++q) {
                const int c = c0 + 32 * q;
                if (c < n) {
                  ap[c] = fma(-m1, y[q], x[q]);
                  aq[c] = fma(m2, x[q], y[q]);
                }
              }
            }
          }
        }
        const bool own = (lane & ((1 << SH) - 1)) == 0;
        const bool fixP = rot && nal < 0.01 * al, fixQ = rot && nbe < 0.01 * be;
        __syncwarp();
        if (own && rot) {
          nrm[P] = nal; nrm[Q] = nbe;
          dsc[P] = dp * cs; dsc[Q] = dq * cs;
          ++myrot;
        }
        if (__any_sync(0xffffffffu, fixP || fixQ)) {   // rare: recompute from the rows
#pragma unroll
          for (int j = 0; j < PW; ++j) {
            const int src = j << SH;
            const bool fp = __shfl_sync(0xffffffffu, fixP, src), fq = __shfl_sync(0xffffffffu, fixQ, src);
            const double d1 = __shfl_sync(0xffffffffu, dp * cs, src), d2 = __shfl_sync(0xffffffffu, dq * cs, src);
            for (int side = 0; side < 2; ++side) {
              if (!(side == 0 ? fp : fq)) continue;    // warp-uniform
              const int r = side == 0 ? Pj[j] : Qj[j];
              const double* row = A + (size_t)r * n;
              const double dr = side == 0 ? d1 : d2;
              double s = 0.0;
              for (int c = lane; c < n; c += 32) { const double v = __ldcg(row + c); s = fma(v, v, s); }
              for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
              if (lane == 0) nrm[r] = s * dr * dr;
            }
          }
        }
      }
      if (myrot) atomicAdd(&s0->rot, myrot);
      cl.sync();
    }
    converged = s0->rot == 0;
    cl.sync();                                        // read before the next sweep clears it
  }
  // true rows and exact norms
  for (int r = rank * nw + warp; r < np; r += kJcCtas * nw) {
    const double dr = dsc[r];
    double s = 0.0;
    double* row = A + (size_t)r * n;
    for (int c = lane; c < n; c += 32) {
      double v = __ldcg(row + c);
      if (dr != 1.0) { v *= dr; row[c] = v; }
      s = fma(v, v, s);
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) nrm[r] = sqrt(s);
  }
  cl.sync();
  double* sg = a.sig + (size_t)mat * np;
  int* pm = a.perm + (size_t)mat * np;
  for (int r = tid; r < np; r += nt) vbuf[r] = nrm[r];
  __syncthreads();
  for (int r = rank * nt + tid; r < np; r += kJcCtas * nt) {
    const double v = vbuf[r];
    int pos = 0;
    for (int j = 0; j < np; ++j) {
      const double u = vbuf[j];
      pos += (u > v) || (u == v && j < r);
    }
    sg[pos] = v;
    pm[pos] = r;
  }
  if (rank == 0 && tid == 0) {
    double s1 = 0.0;
    for (int r = 0; r < np; ++r) s1 = fmax(s1, vbuf[r]);
    if (a.lns1) a.lns1[mat] = s1 > 0.0 ? log(s1) : -INFINITY;
    const double tau = (a.zero_rel > 0.0 ? a.zero_rel : (double)n * 0x1.0p-52) * s1;
    int cnt = 0;
    for (int r = 0; r < np; ++r) cnt += vbuf[r] > tau;
    a.nnz[mat] = s1 > 0.0 ? cnt : 0;
    if (a.mflags && !converged) a.mflags[mat] |= FLAG_NOCONV;
  }
  __syncthreads();
  // rows of W are right vectors of M: undo the column pivoting of R
  for (int r = rank; r < np; r += kJcCtas) {
    double* row = A + (size_t)r * n;
    for (int c = tid; c < n; c += nt) vbuf[c] = __ldcg(row + c);
    __syncthreads();
    for (int c = tid; c < n; c += nt) row[colperm[c]] = vbuf[c];
    __syncthreads();
  }
  cl.sync();                                          // rank 0's shared memory stays until all have read it
}

template <int PW, int NQ>
static cudaError_t launch_cluster_variant(const JacobiArgs& a, cudaStream_t st) {
  const size_t np = a.n_pad;
  const size_t smem = (4 * np + 2 * np + (kJcThreads / 32 + 1) * 32) * sizeof(double) + (np + 2 + np + 2) * sizeof(int) + 64;
  static std::atomic<uint64_t> attr{0};
  cudaError_t e = raise_smem_limit(k_jacobi_cluster<PW, NQ>, 100 * 1024, attr);
  if (e != cudaSuccess) return e;
  k_jacobi_cluster<PW, NQ><<<a.S * kJcCtas, kJcThreads, smem, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_jacobi_few(const JacobiArgs& a, cudaStream_t st) {
  if (a.S <= 0) return cudaSuccess;
  // below n = 64 the barriers cost more than seven further SMs give
  if (a.n < kJcMinN || a.n > 1024) return launch_jacobi(a, st);
  const int per = (a.n_pad / 2 + kJcCtas * kJcWarps - 1) / (kJcCtas * kJcWarps);   // pairs per warp
  if (per <= 1) return launch_cluster_variant<1, 2>(a, st);      // n <= 64
  if (per <= 2) return launch_cluster_variant<2, 4>(a, st);      // n <= 128
  if (per <= 4) return launch_cluster_variant<4, 8>(a, st);      // n <= 256
  if (per <= 8) return launch_cluster_variant<8, 0>(a, st);
  return launch_cluster_variant<16, 0>(a, st);
}

template <int PW>
static cudaError_t launch_warp_variant(const JacobiArgs& a, int threads, cudaStream_t st) {
  const int n = a.n, np = a.n_pad;
  const size_t rows_bytes = (size_t)np * n * sizeof(double);
  const size_t aux = (size_t)np * 5 * sizeof(double) + 34 * sizeof(double) +
                     (size_t)(2 * np + 2 + 34) * sizeof(int);
  const int use_smem = (rows_bytes + aux) <= 200 * 1024;
  // Rows in the global workspace: stage one row per warp in shared memory for
  // the final column permutation, and ask for enough shared memory that one
  // CTA runs per SM, so the rows of the resident matrices stay in L2.
  const size_t staging = (size_t)(threads / 32) * n * sizeof(double);
  const size_t smem = use_smem ? rows_bytes + aux : std::max<size_t>(aux + staging, 120 * 1024);
  static std::atomic<uint64_t> attr{0};
  cudaError_t e = raise_smem_limit(k_jacobi_warp<PW>, 200 * 1024 + 64, attr);
  if (e != cudaSuccess) return e;
  k_jacobi_warp<PW><<<a.S, threads, smem, st>>>(a, use_smem);
  return cudaGetLastError();
}

template <int G>
static cudaError_t launch_small(const JacobiArgs& a, cudaStream_t st) {
  const int np = a.n_pad;
  const size_t smem = (size_t)np * a.n * sizeof(double) + (size_t)np * sizeof(double) + (size_t)(np + 2) * sizeof(int);
  k_jacobi<G><<<a.S, std::max(32, (np / 2 * G + 31) / 32 * 32), smem, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_jacobi(const JacobiArgs& a, cudaStream_t st) {
  if (a.S <= 0) return cudaSuccess;
  if (a.n > 32) {
    // pairs per warp so that one pass of the warps covers a step
    const int npairs = a.n_pad / 2;
    const int threads = a.n <= 64 ? 256 : 512;
    const int nw = threads / 32;
    int pw = 1;
    while (pw < 32 && pw * nw < npairs) pw <<= 1;
    switch (pw) {
      case 1: return launch_warp_variant<1>(a, threads, st);
      case 2: return launch_warp_variant<2>(a, threads, st);
      case 4: return launch_warp_variant<4>(a, threads, st);
      case 8: return launch_warp_variant<8>(a, threads, st);
      case 16: return launch_warp_variant<16>(a, threads, st);
      default: return launch_warp_variant<32>(a, threads, st);
    }
  }

  // n <= 32: about two entries of a row per lane, one lane group per pair of a
  // step: a second pass of the groups would double the chain of a step.  With it
  // and the rotation's scalars at a fifth of their FP64 instructions: 64 matrices
  // of n = 16 1.71 -> 0.54 ms, 4096 9.5 -> 4.5, the 4096 cores of an L = 16,
  // chi = 8 run 3.5 -> 1.7
  if (a.n <= 4) return launch_small<2>(a, st);
  if (a.n <= 8) return launch_small<4>(a, st);
  if (a.n <= 16) return launch_small<8>(a, st);
  return launch_small<16>(a, st);
}

}  // namespace mctrg
