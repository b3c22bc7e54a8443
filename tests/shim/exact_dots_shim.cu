// k_exact_dots over m vectors of length N (host arrays, hi and lo parts) on the
// grid that the library gives it for P problems.
#include <vector>

#include "blas_kernels.cuh"

extern "C" int shim_exact_blocks(long long N, int P, int m) { return nfs::exact_dots_blocks(N, P, m); }
extern "C" int shim_red_blocks(long long N, int P) { return nfs::red_blocks(N, P); }

extern "C" int shim_exact_dots(const float2* shi, const float2* slo, const float2* whi, const float2* wlo, long long N,
                               int m, int P, double* out) {
  if (N < 2 || N % 2 != 0 || m < 1 || P < 1) return -1;
  const int nb = nfs::exact_dots_blocks(N, P, m);
  float2 *dv[4] = {};
  double *part = nullptr, *fin = nullptr;
  const float2* src[4] = {shi, slo, whi, wlo};
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < 4 && e == cudaSuccess; ++i) {
    const size_t bytes = (size_t)N * (i < 2 ? m : 1) * sizeof(float2);
    e = cudaMalloc(&dv[i], bytes);
    if (e == cudaSuccess) e = cudaMemcpy(dv[i], src[i], bytes, cudaMemcpyHostToDevice);
  }
  if (e == cudaSuccess) e = cudaMalloc(&part, (size_t)m * nb * 2 * sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(&fin, (size_t)m * 2 * sizeof(double));
  if (e == cudaSuccess) {
    nfs::k_exact_dots<<<dim3((m + 1) / 2, nb, 1), nfs::kRedThreads>>>(dv[0], dv[1], (long long)m * N, m, dv[2], dv[3], N,
                                                                      part, nullptr);
    nfs::k_dots_finish<<<dim3(m, 1), nfs::kRedThreads>>>(part, m, nb, fin, nullptr);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(out, fin, (size_t)m * 2 * sizeof(double), cudaMemcpyDeviceToHost);
  for (float2* p : dv) cudaFree(p);
  cudaFree(part);
  cudaFree(fin);
  return (int)e;
}
