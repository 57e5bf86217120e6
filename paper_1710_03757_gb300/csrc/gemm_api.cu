// The plaquette GEMM through the C ABI on its own: M[b] = X[b] Yt[b]^T,
// plain row-major output (the matricization epilogue with parity A is the
// identity map), on the CUDA cores in FP64 or at FP64 accuracy on the tensor
// cores (FP16 digits).
#include <cstdint>

#include "../../include/mctrg.h"
#include "common.cuh"
#include "kernels.h"
#include "kernels_tc.h"

extern "C" int mctrg_contract_batched(const double* X, const double* Yt, int D, int K, int64_t batch, double* M,
                                      int precision, void* stream) {
  if (!X || !Yt || !M || D < 1 || D > 32 || K < 1 || batch < 1 || batch > (1 << 30)) return MCTRG_EINVAL;
  const int n = D * D;
  cudaStream_t st = (cudaStream_t)stream;
  if (precision == MCTRG_FP64) {
    mctrg::GemmArgs gm{};
    gm.X = X; gm.Yt = Yt; gm.M = M; gm.D = D; gm.K = K; gm.c0 = 0; gm.n_items = batch; gm.Nnew = 1;
    gm.L = 2; gm.level_new = 0; gm.fixed_parity = 0;
    if (mctrg::launch_gemm_f64(gm, st) != cudaSuccess) return MCTRG_ECUDA;
    return cudaStreamSynchronize(st) == cudaSuccess ? MCTRG_OK : MCTRG_ECUDA;
  }
  if (precision != MCTRG_FP64TC || !mctrg::gemm_ozaki_supported(n, K)) return MCTRG_EINVAL;
  const int64_t rows = batch * n;
  int* ws = nullptr;                                 // row exponents, then the error word
  int status = MCTRG_ENOMEM;
  if (cudaMalloc(&ws, sizeof(int) * (2 * (size_t)rows + 1)) != cudaSuccess) return status;
  // the kernel reads its operands while it writes: a result over one of them goes through a buffer
  const size_t out = sizeof(double) * (size_t)batch * n * n, in = sizeof(double) * (size_t)batch * n * K;
  auto meets = [&](const double* p) {
    return (uintptr_t)p < (uintptr_t)M + out && (uintptr_t)M < (uintptr_t)p + in;
  };
  double* tmp = nullptr;
  if ((meets(X) || meets(Yt)) && cudaMalloc(&tmp, out) != cudaSuccess) {
    cudaFree(ws);
    return status;
  }
  status = MCTRG_ECUDA;
  uint32_t* err = (uint32_t*)(ws + 2 * rows);
  uint32_t herr = 0;
  mctrg::GemmOzArgs ga{};
  ga.X = X; ga.Y = Yt; ga.M = tmp ? tmp : M; ga.D = D; ga.n = n; ga.K = K; ga.c0 = 0; ga.n_items = batch; ga.Nnew = 1;
  ga.L = 2; ga.level_new = 0; ga.fixed_parity = 0; ga.expX = ws; ga.err = err;
  if (cudaMemsetAsync(err, 0, sizeof(uint32_t), st) == cudaSuccess &&
      mctrg::launch_gemm_ozaki(ga, st) == cudaSuccess &&
      (!tmp || cudaMemcpyAsync(M, tmp, out, cudaMemcpyDeviceToDevice, st) == cudaSuccess) &&
      cudaMemcpyAsync(&herr, err, sizeof(herr), cudaMemcpyDeviceToHost, st) == cudaSuccess &&
      cudaStreamSynchronize(st) == cudaSuccess)
    status = herr ? MCTRG_ECUDA : MCTRG_OK;
  cudaStreamSynchronize(st);
  cudaFree(ws);
  if (tmp) cudaFree(tmp);
  return status;
}
