// The kernels around a run of CG steps: the start of an inner solve, and one
// k_cg_check on a state that the caller describes (what the host would read).
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

// r^* r at the start of an inner solve of scale * r64 (N complex numbers).
extern "C" int shim_inner_start(const double2* r64, long long N, double scale, int nb, double* rr0) {
  if (N < 2 || N % 2 != 0 || nb < 1 || nb > nfs::kRedBlocks) return -1;
  char* d = nullptr;
  const size_t vec64 = N * sizeof(double2), vec32 = N * sizeof(float2);
  cudaError_t e = cudaMalloc(&d, vec64 + 3 * vec32 + 2 * sizeof(double) + sizeof(nfs::CGState));
  if (e != cudaSuccess) return (int)e;
  auto* a = reinterpret_cast<double2*>(d);
  auto* r = reinterpret_cast<float2*>(d + vec64);
  auto* small = reinterpret_cast<double*>(d + vec64 + 3 * vec32);
  auto* st = reinterpret_cast<nfs::CGState*>(small + 2);
  const double h[2] = {scale, 0.0};
  nfs::CGState* out = new nfs::CGState{};
  e = cudaMemcpy(a, r64, vec64, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(small, h, sizeof(h), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    nfs::k_inner_start<<<dim3(nb, 1), nfs::kRedThreads>>>(a, small, r, r + N, r + 2 * N, N, st);
    nfs::k_cg_init<float><<<1, nfs::kRedThreads>>>(st, small + 1, false, 1, nb, 1);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(out, st, sizeof(nfs::CGState), cudaMemcpyDeviceToHost);
  *rr0 = out->rr0;
  cudaFree(d);
  delete out;
  return (int)e;
}
