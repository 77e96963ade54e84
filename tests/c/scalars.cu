/* The square root and the reciprocals on the chains of the QR and the elimination, one per thread. */
#include "ttm_gemm.cuh"
#include "ttm_pre.cuh"

__global__ void scalars_kernel(const double* g, const double* alpha, int n, double* beta, double* vj, double* tau, double* inv) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double b, v, t;
  ttm::qd_scalars(g[i], alpha[i], b, v, t, [](double&, double&) {});
  beta[i] = b;
  vj[i] = v;
  tau[i] = t;
  inv[i] = ttm::pre_pivot_inv(g[i], g[i]);
}
extern "C" int scalars(const double* g, const double* alpha, int n, double* beta, double* vj, double* tau, double* inv) {
  scalars_kernel<<<(n + 127) / 128, 128>>>(g, alpha, n, beta, vj, tau, inv);
  const cudaError_t e = cudaDeviceSynchronize();
  return (int)e;
}
