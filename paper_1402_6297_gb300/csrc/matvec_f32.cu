// complex64 instantiation of the A_r product, and the material in the order its
// column kernel reads.
#include "matvec_impl.cuh"

namespace nfs {
NFS_INSTANTIATE_ROWS(float)
NFS_INSTANTIATE_COLUMNS(float)

// pmat and pmu of MatvecArgs: [j][a][x slot][b / 2][z slot], each entry the two
// slots b, b + 1 of y, so that the threads of k_columns (z slot fastest) read
// 16 consecutive bytes each.  Natural index of slot s of a length N1 N2:
// s / N2 + N1 (s % N2).
__global__ void k_pair_material(const double* __restrict__ mat, long long smat, int n1, int N2, int n3, int Z2,
                                int kind, int ax_a, int ax_b, long long gam_len, bool has_mu,
                                float4* __restrict__ pmat, float2* __restrict__ pmu, int P) {
  const long long n = (long long)n1 * n1 * n3;
  const int N1 = n1 / N2, Z1 = n3 / Z2;
  const long long per = 3 * n / 2, total = per * P;
  for (long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x; g < total; g += (long long)gridDim.x * blockDim.x) {
    const double* m = mat + g / per * smat;
    long long r = g % per;
    const int zs = (int)(r % n3);
    r /= n3;
    const int k = (int)(r % (N2 / 2));
    r /= N2 / 2;
    const int xs = (int)(r % n1);
    r /= n1;
    const int a = (int)(r % N1), j = (int)(r / N1);
    const long long z = (zs / Z2 + Z1 * (zs % Z2)), x = (xs / N2 + N1 * (xs % N2));
    const int s = pair_axis(kind, ax_a, ax_b, j);
    float ip[2], gm[2], im[2];
    for (int t = 0; t < 2; ++t) {
      const long long v = (z * n1 + a + N1 * (2 * k + t)) * n1 + x;
      ip[t] = (float)m[j * n + v];
      gm[t] = kind == kMediumChiral ? (float)m[3 * n + j * n + v] : (s == j ? 0.f : (float)m[3 * n + v]);
      im[t] = has_mu ? (float)m[3 * n + gam_len + s * n + v] : 1.f;
    }
    pmat[g] = make_float4(ip[0], gm[0], ip[1], gm[1]);
    if (has_mu) pmu[g] = make_float2(im[0], im[1]);
  }
}

cudaError_t pair_material_launch(const double* mat, long long smat, int n1, int n3, int kind, int ax_a, int ax_b,
                                 long long gam_len, bool has_mu, float4* pmat, float2* pmu, int P,
                                 cudaStream_t stream) {
  const long long total = 3LL * n1 * n1 * n3 / 2 * P;
  const int blocks = (int)std::min<long long>((total + 255) / 256, 152LL * 16);
  int N2 = 0, Z2 = 0;
  switch (n1) {
#define NFS_CASE(N) case N: N2 = PlaneSplit<float, N>::N2; break;
    NFS_FOR_EACH_SIZE(NFS_CASE)
#undef NFS_CASE
  }
  switch (n3) {
#define NFS_CASE(N) case N: Z2 = DepthSplit<float, N>::N2; break;
    NFS_FOR_EACH_SIZE(NFS_CASE)
#undef NFS_CASE
  }
  if (N2 == 0 || Z2 == 0) return cudaErrorInvalidValue;
  k_pair_material<<<blocks, 256, 0, stream>>>(mat, smat, n1, N2, n3, Z2, kind, ax_a, ax_b, gam_len, has_mu, pmat, pmu,
                                              P);
  return cudaGetLastError();
}

bool matvec_supported(int n1, int n2, int n3) {
  auto ok = [](int s) {
    switch (s) {
#define NFS_CASE(N) case N: return true;
      NFS_FOR_EACH_SIZE(NFS_CASE)
#undef NFS_CASE
    }
    return false;
  };
  return n1 == n2 && ok(n1) && ok(n3);
}

}  // namespace nfs
