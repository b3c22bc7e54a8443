// Host-side entry points of the A_r product (matvec_kernels.cuh), instantiated
// for complex64 (matvec_f32.cu), complex128 (matvec_f64.cu) and double-single
// vectors (matvec_df.cu).
#pragma once
#include <cuda_runtime.h>

#include "nfs_complex.cuh"

namespace nfs {

template <typename R>
struct MatView;

// Strides between the problems of a batched launch (P problems of one grid,
// stored back to back): elements for vectors / workspace / tables, reals (pairs
// of voxels in the complex64 order) for the material, ints for the skip flags.
struct BatchStrides {
  long long su = 0;      // u, Au; x, r, p of CG
  long long sfld = 0;    // fld (16-byte elements)
  long long smat = 0;    // inv_phi, gam, inv_mu; pmat, pmu
  long long sbasis = 0;  // basis
  int slam = 0;          // lam
  int sskip = 0;         // skip
};

struct CGState;

// Vectors in memory: complex64, complex128, or (double-single products, whose
// row kernels convert as they load and store) complex128 again.
struct df;
template <typename R> struct VecOf { using type = cplx<R>; };
template <> struct VecOf<df> { using type = double2; };
template <typename R> using vecc = typename VecOf<R>::type;

// The CG step taken by the product's kernels: k_rows_in first forms
// p = r + beta p (in place), k_columns p^* A_r p from the real-space fields,
// k_rows_out x += alpha p and r -= alpha A_r p per voxel (A_r p is never
// stored) and the new r^* r.
template <typename R>
struct CgFuse {
  vecc<R>* x = nullptr;
  vecc<R>* r = nullptr;
  vecc<R>* p = nullptr;
  CGState* st = nullptr;  // per problem: st + prob; nullptr: a plain product
};

// What the row kernels do besides when they form S Q_r^* e | S P_r^* h - sigma v of
// the NFSEP (nfsep.h; complex128, one problem), S = Sigma_r^{1/2}, and the ends of
// a GMRES step around it: k_rows_in scales its input by S; with `tmp` the input
// is u - sum_g tmp_g (the end of the Gram-Schmidt update), stored into v, with
// one partial of its squared norm per CTA.  k_rows_out exchanges the halves of
// the result, scales by S and subtracts sigma v; with nnrm partials of |v|^2 it
// also normalises: v and the result times 1 / |v| (0 for a zero v).
struct KrylovFuse {
  const double* root = nullptr;  // Lambda_q^{1/4} per voxel; nullptr: a plain product
  const double2* tmp = nullptr;  // [groups][4n]
  int groups = 0;
  double2* v = nullptr;          // nullptr: no sigma v
  double* nrm_out = nullptr;     // k_rows_in's partials
  const double* nrm = nullptr;   // k_rows_out: partials to normalise by
  int nnrm = 0;
  double2 sigma = {0.0, 0.0};
};

template <typename R>
struct MatvecArgs {
  const vecc<R>* u;       // 4n, spectral
  vecc<R>* Au;            // 4n, spectral
  void* fld;              // workspace: 6n complex numbers
  const cplx<R>* lam;     // Lambda_1 | Lambda_2 | Lambda_3 (n1 + n2 + n3)
  const cplx<R>* tw1;     // exp(-2 pi i m / n1), m < n1 (n2 = n1)
  const cplx<R>* tw3;     // exp(-2 pi i m / n3), m < n3
  // the material: complex64 products read pmat and pmu (pair_material_launch),
  // the others the natural-order arrays
  const R* inv_phi;
  const R* gam;
  const R* inv_mu;        // nullptr for mu = 1
  const float4* pmat;
  const float2* pmu;      // nullptr for mu = 1
  int kind, ax_a, ax_b;
  int n1, n3;             // grid n1 x n1 x n3
  R alpha, beta;
  const int* skip;        // device flag: when nonzero every kernel returns at once
  // optional table of the per-voxel basis, [c_x, c_y, c_z, x_x, x_y, x_z][n]
  // (spectral order); nullptr: evaluated from the Lambda tables in the kernels
  const cplx<R>* basis;
  cudaStream_t stream;
  bool serial;            // no overlap between kernels: the tables are being written on the stream
  KrylovFuse kr;          // optional (complex128)
  CgFuse<R> cg;           // optional: one CG step (u and Au are then unused)
  // batching: P problems of this grid in one launch (P = 1 for one problem)
  int P;
  BatchStrides bs;
};

// Largest dynamic shared memory a CTA may request on sm_103a.
constexpr size_t kMaxDynSmem = 232448;

// Whether the kernels exist for this grid (n1 = n2 and each size in {8, 12,
// 16, 24, 32, 48, 64, 96, 128}).
bool matvec_supported(int n1, int n2, int n3);
// The row kernels (k_rows_in / k_rows_out) and k_columns; prepare opts the
// kernels of a grid in to their dynamic shared memory (once per device).
template <typename R> cudaError_t rows_prepare(int n1);
template <typename R> cudaError_t rows_launch(const MatvecArgs<R>& a, bool in);
template <typename R> cudaError_t product_columns_prepare(int n1, int n3);
template <typename R> cudaError_t product_columns_launch(const MatvecArgs<R>& a);

template <typename R>
cudaError_t matvec_prepare(int n1, int n3) {
  const cudaError_t e = rows_prepare<R>(n1);
  return e != cudaSuccess ? e : product_columns_prepare<R>(n1, n3);
}
// Selected kernels (bit 0: k_rows_in, bit 1: k_columns, bit 2: k_rows_out).
template <typename R>
cudaError_t matvec_launch_mask(const MatvecArgs<R>& a, int mask) {
  cudaError_t e = cudaSuccess;
  if (mask & 1) e = rows_launch<R>(a, true);
  if (e == cudaSuccess && (mask & 2)) e = product_columns_launch<R>(a);
  if (e == cudaSuccess && (mask & 4)) e = rows_launch<R>(a, false);
  return e;
}
template <typename R> cudaError_t matvec_launch(const MatvecArgs<R>& a) { return matvec_launch_mask<R>(a, 7); }
// Kernels of one whole product.
constexpr int kProductKernels = 3;
// CTAs of k_rows_out per problem: the partials of r^* r that a CG step leaves.
template <typename R> int cg_partials(int n1, int n3);

// The basis table for MatvecArgs<double>::basis: P problems (Lambda tables
// at lam + p * slam, tables at basis + p * sbasis).
cudaError_t basis_table_launch(const double2* lam, int n1, int n2, int n3, double alpha, double beta, double2* basis,
                               int P, int slam, long long sbasis, cudaStream_t stream);

// The material in the order in which the complex64 k_columns meets it: for P
// problems (natural-order FP64 arrays mat + p * smat: inv_phi 3n | gam | inv_mu)
// pmat[p (3n / 2) + ...] = {1/Phi, g} of two neighbouring y slots, pmu = their
// mu^{-1} (has_mu; else nullptr).
cudaError_t pair_material_launch(const double* mat, long long smat, int n1, int n3, int kind, int ax_a, int ax_b,
                                 long long gam_len, bool has_mu, float4* pmat, float2* pmu, int P,
                                 cudaStream_t stream);

// The double-single tables of a context (matvec_df.cu): `count` reals.
cudaError_t double_to_df(const double* in, df* out, long long count, cudaStream_t s);

// Gradient accumulation (complex128 only) from the workspace after k_rows_in:
// per voxel d_eps += scale * dA/deps and dg += the chirality term, 3n doubles
// each (one n per pair) in the column kernel's order; the first vector's call
// (`first`) sets them.  Either may be nullptr.  grad_natural_launch, after the
// last vector, writes the caller's d_eps [3n] and d_gamma (chiral [3n],
// pseudochiral [n]) in natural order.
struct GradArgs {
  void* fld;
  const double2* tw1;
  const double2* tw3;
  const double* inv_phi;
  const double* gam;
  int kind, ax_a, ax_b;
  int n1, n3;
  double scale;
  double* d_eps;
  double* dg;
  bool first;
  cudaStream_t stream;
};
cudaError_t grad_launch(const GradArgs& a);
cudaError_t grad_natural_launch(const GradArgs& a, double* d_eps, double* d_gamma);

// Fields [E; H] = B^{-1} diag(P_r, Q_r) y of one eigenvector from the
// workspace of y after k_rows_in (matvec_f64.cu).
struct FieldsArgs {
  void* fld;
  const double2* tw1;
  const double2* tw3;
  const double2* bloch;   // D_1 | D_2 | D_3 diagonals, n1 + n2 + n3
  const double* inv_phi;
  const double* gam;
  const double* inv_mu;   // nullptr for mu = 1
  int kind, ax_a, ax_b;
  int n1, n3;
  double2* X;             // 6n out: E_x, E_y, E_z, H_x, H_y, H_z
  cudaStream_t stream;
};
cudaError_t fields_launch(const FieldsArgs& a);
// Opt both in to their shared memory.
cudaError_t fields_prepare(int n1, int n3);

// Partial sums of the GEP residual of (omega, x) (matvec_f64.cu).
struct GepResidualArgs {
  const double2* X;       // 6n: E_x, E_y, E_z, H_x, H_y, H_z
  const double* inv_phi;
  const double* gam;
  const double* inv_mu;   // nullptr for mu = 1
  int kind, ax_a, ax_b;
  int n1, n2, n3;
  double inv_delta[3];
  double2 wrap[3];        // exp(i 2 pi k.a_l)
  double omega;
  double* part;           // 2 per block: |residual|^2, |B x|^2
};
cudaError_t gep_residual_launch(const GepResidualArgs& a, int blocks, cudaStream_t stream);

}  // namespace nfs
