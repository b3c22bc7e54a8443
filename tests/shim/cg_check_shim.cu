// One k_cg_check on a state that the caller describes: what the host would read.
#include "blas_kernels.cuh"

namespace {
template <typename R>
int check(double rr_now, const double* part_b, int nb, double tol2, int halt, int broken, int it, int maxit, int* out,
          double* rr) {
  using P = typename nfs::RedAccFor<R>::partial;
  nfs::CGState* h = new nfs::CGState{};
  auto put = [](double v, double& at) {
    if constexpr (sizeof(R) == 4) {
      const float hi = (float)v;
      reinterpret_cast<float2&>(at) = make_float2(hi, (float)(v - (double)hi));
    } else {
      at = v;
    }
  };
  static_assert(sizeof(P) == sizeof(double), "partials are eight bytes");
  for (int i = 0; i < nb; ++i) put(part_b[i], h->part_b[i]);
  put(rr_now, h->rr_now);
  put(tol2, h->tol2);
  h->stop = h->halt = halt;
  h->broken = broken;
  h->it = it;
  h->maxit = maxit;
  nfs::CGState* d = nullptr;
  cudaError_t e = cudaMalloc(&d, sizeof(nfs::CGState));
  if (e == cudaSuccess) e = cudaMemcpy(d, h, sizeof(nfs::CGState), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    nfs::k_cg_check<R><<<1, nfs::kRedThreads>>>(d, nb);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(h, d, sizeof(nfs::CGState), cudaMemcpyDeviceToHost);
  out[0] = h->done;
  out[1] = h->status;
  *rr = h->rr;
  cudaFree(d);
  delete h;
  return (int)e;
}
}  // namespace

extern "C" int shim_cg_check(int single, double rr_now, const double* part_b, int nb, double tol2, int halt, int broken,
                             int it, int maxit, int* out, double* rr) {
  if (nb < 1 || nb > nfs::kMaxPartials) return -1;
  return single ? check<float>(rr_now, part_b, nb, tol2, halt, broken, it, maxit, out, rr)
                : check<double>(rr_now, part_b, nb, tol2, halt, broken, it, maxit, out, rr);
}
