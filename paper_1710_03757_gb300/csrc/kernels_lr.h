// Launch interfaces of the low-rank levels' split (K2): the SVD of M = X Yt^T
// through the core of the QR factors of X and Yt, for levels whose inner
// dimension K is smaller than the matrix side n.
#pragma once
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

namespace mctrg {

// M = X Yt^T with X = Qx Rx and Yt = Qy Ry (n x K each): M = Qx (Rx Ry^T) Qy^T,
// so the K x K core C = Rx Ry^T has M's nonzero singular values and its
// vectors are M's in the bases Qx, Qy.
constexpr int kLowRankMaxK = 256;
inline bool lowrank_supported(int n, int K) { return K >= 2 && K < n && K <= kLowRankMaxK && n <= 2304; }

// Householder QR of X and Yt of S items, in place: rows 0 .. K-1 of each
// item's block become R (upper triangular, zeros below), V (unit lower
// trapezoidal) goes to Vt[side][item][K][n], row k holding reflector k over
// all n entries, and tau to taus[side][item][K]; H_k = I - tau_k v_k v_k^T,
// Q = H_0 H_1 ... H_{K-1}.
struct LowRankQrArgs {
  double* X;         // [S][n][K]
  double* Yt;        // [S][n][K]
  double* Vt;        // [2][S][K][n]
  double* taus;      // [2][S][K]
  int n, K, S;
};
cudaError_t launch_lowrank_qr(const LowRankQrArgs& a, cudaStream_t st);

// Halves of the level from those of the core: left = Qx left_c (n x kc),
// right = right_c Qy^T (kc x n), in the sampler's layout (stride 2 n kc, core
// stride 2 K kc).
struct LowRankExpandArgs {
  const double* Vt;
  const double* taus;
  const double* Hc;  // [S]: [left K x kc | right kc x K]
  double* H;         // [S]: [left n x kc | right kc x n]
  int n, K, S, kc;
};
cudaError_t launch_lowrank_expand(const LowRankExpandArgs& a, cudaStream_t st);

// Doubles per item of Vt, taus and the core's halves, in this order.
inline size_t lowrank_vt_doubles(int n, int K) { return (size_t)2 * K * n; }
inline size_t lowrank_tau_doubles(int K) { return (size_t)2 * K; }
inline size_t lowrank_halves_doubles(int K, int kc) { return (size_t)2 * K * kc; }
inline size_t lowrank_item_doubles(int n, int K, int kc) {
  return lowrank_vt_doubles(n, K) + lowrank_tau_doubles(K) + lowrank_halves_doubles(K, kc);
}

}  // namespace mctrg
