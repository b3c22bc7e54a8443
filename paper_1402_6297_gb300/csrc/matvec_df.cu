// The A_r product in double-single arithmetic (R = df, C = dfc: float pairs
// hi + lo, about 48 bits; see dfloat.cuh).  Used for the FP64-accuracy
// refinement residuals of the mixed-precision path, where it replaces the
// complex128 product: this GPU's FP32 units are far faster than its FP64 ones.
// The row kernels convert complex128 vectors as they load and store them (two
// separate conversion kernels, FP64-pipe bound, took 99 of 650 us at 96^3).
#include "dfloat.cuh"
#include "matvec_impl.cuh"

namespace nfs {

NFS_INSTANTIATE_ROWS(df)  // (the column kernels: matvec_df_columns.cu)

// double -> double-single, `count` reals (the tables of a context)
__global__ void k_double_to_df(const double* __restrict__ in, df* __restrict__ out, long long count) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x)
    out[i] = df(in[i]);
}

cudaError_t double_to_df(const double* in, df* out, long long count, cudaStream_t s) {
  const int blocks = (int)std::min<long long>((count + 255) / 256, 152LL * 16);
  k_double_to_df<<<blocks, 256, 0, s>>>(in, out, count);
  return cudaGetLastError();
}

}  // namespace nfs
