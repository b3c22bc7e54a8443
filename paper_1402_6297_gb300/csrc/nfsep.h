// Device pieces of the null space free standard problem for any nonsingular
// B (eq. NFSEP_org, Algorithm 1's second branch), complex128 (nfsep.cu):
//
//   M y = [Sigma_r^{1/2} Q_r^* e ; Sigma_r^{1/2} P_r^* h],
//   [e; h] = B^{-1} [P_r Sigma_r^{1/2} y1 ; Q_r Sigma_r^{1/2} y2],
//
// run as the three kernels of the A_r product: k_rows_in (scaling its input by
// Sigma_r^{1/2}), nfsep_columns (the column kernel with B^{-1} per voxel, h in the
// place of p and e in the place of q), k_rows_out (which then has [P_r^* h;
// Q_r^* e], exchanges the halves, scales and optionally subtracts sigma y; see
// KrylovFuse in matvec.h).  B^{-1} is stored per voxel and component as the 2 x 2 block
// coupling (p_c, q_c) to (e_c, h_c): binv[(4 c + t) n + v], t = 00, 01, 10, 11.
#pragma once
#include <cuda_runtime.h>

namespace nfs {

// root[v] = Lambda_q^{1/4}, the diagonal of Sigma_r^{1/2}, per voxel
cudaError_t nfsep_root(const double2* lam, int n1, int n2, int n3, double* root, cudaStream_t s);
cudaError_t nfsep_prepare(int n1, int n3);
cudaError_t nfsep_columns(void* fld, const double2* binv, const double2* tw1, const double2* tw3, int n1, int n3,
                          cudaStream_t s);
// Algorithm 1 (second branch): X = [E; H] = D [e; h] / sqrt(n) from the
// workspace of Sigma_r^{1/2} y after k_rows_in (D: the Bloch twist, from its
// three 1-D diagonals)
cudaError_t nfsep_fields(void* fld, const double2* binv, const double2* tw1, const double2* tw3, const double2* bloch,
                         int n1, int n3, double2* X, cudaStream_t s);

// Long-vector operations of the Krylov drivers (complex128):
// dst = scale * src
cudaError_t zscale_copy(const double2* src, double2* dst, double scale, long long N, cudaStream_t s);
// V_i <- sum_{r<m} V_r Y[r k + i], i < k, in place (Y device interleaved complex)
cudaError_t zrotate(double2* V, int m, const double* Y, int k, long long N, cudaStream_t s);

// Restarted GMRES for the shifted systems (M - sigma I) z = b with the long-
// vector work on the device and no host round trip per step: the two classical
// Gram-Schmidt passes leave their coefficients as partial sums in device memory,
// which the updates add up, and the next product ends the update and
// normalises.  The host reads a batch of Hessenberg columns at once and keeps
// the small least-squares problem (nfs::host::GivensLS, krylov.h).
constexpr int kGmresMax = 128;  // largest restart length
struct GmresDev {
  double2 Hc[kGmresMax * (kGmresMax + 1)];  // column j of H at Hc[j (kGmresMax + 1) + i], i <= j + 1
};

// Chunks (S) of the dot products of vectors of length N, and the blocks (norm
// partials) of gs_finish and gmres_residual.
int gs_chunks(long long N);
int gs_norm_blocks(long long N);
// complex128 elements of the scratch `tmp` that gs_update needs
long long gs_tmp_len(long long N);
// part[(s m + j) 2 + {0, 1}] = chunk s's share of V_j^* w', j < m (m <= kGmresMax),
// w' = w - sum_{g < G} tmp_g, stored in w2 (G = 0: w itself)
cudaError_t gs_dots(const double2* V, int m, const double2* w, const double2* tmp, int G, double2* w2, long long N,
                    double* part, cudaStream_t s);
// tmp_g = the g-th share of sum_{j<m} c_j V_j, c_j = sum_s part[(s m + j)]; *groups = how many
cudaError_t gs_update(const double2* V, int m, long long N, const double* part, int S, double2* tmp, int* groups,
                      cudaStream_t s);
// dst = w - sum_{g < G} tmp_g (dst may be w), and (optional) the partials of |dst|^2
cudaError_t gs_finish(const double2* w, const double2* tmp, int G, double2* dst, long long N, double* nrm_part,
                      cudaStream_t s);
// w = b - w and the partials of ||w||^2
cudaError_t gmres_residual(const double2* b, double2* w, long long N, double* nrm_part, cudaStream_t s);
// Columns j0 .. j0 + nsteps - 1 of H: step t's two passes' partials at
// part + 2 t plen and part + (2 t + 1) plen, its nnrm norm partials at
// nrm + t nlen (the last step's nlast at nrm_last).
cudaError_t gmres_columns(int j0, int nsteps, const double* part, long long plen, int S, const double* nrm,
                          long long nlen, int nnrm, const double* nrm_last, int nlast, GmresDev* st, cudaStream_t s);

}  // namespace nfs
