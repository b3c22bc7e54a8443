// complex128 instantiation of the A_r product; the eigenvalue gradient and the
// eigenvector fields, which are other per-voxel steps of its column kernel; the
// residual of the original GEP.
#include <algorithm>
#include <cmath>
#include "matvec_impl.cuh"

namespace nfs {
NFS_INSTANTIATE_ROWS(double)
NFS_INSTANTIATE_COLUMNS(double)

// Gradient of omega with respect to the per-component permittivity and the
// chirality, for one eigenvector y of B_r y = theta A_r y (mu = 1):
//   d omega = y^* (dA_r) y / (y^* B_r y),
//   y^* A_r y = sum_c |s_c|^2 / Phi_c + |p_c|^2,  s = xi p + q,
// with (p, q) = (P_r y1, Q_r y2) in real space (eq. factor_mtx with mu = 1,
// zeta = xi^*).  Hence, per voxel and component,
//   d/d eps_c   : -|s_c|^2 / Phi_c^2
//   d/d gamma_c : 2 Re(conj(s_c) i p_c) / Phi_c + 2 gamma_c |s_c|^2 / Phi_c^2   (chiral)
// and for the pseudochiral pair (a, b) with one gamma per voxel the two
// coupled components' terms add (s_a = i gamma p_b + q_a, s_b = i gamma p_a + q_b);
// different CTAs form them, so each pair has its own sums.
// `scale` carries weight / (n y^* B_r y): the DFTs leave sqrt(n) p, sqrt(n) q.
// The sums of several vectors are kept in the order in which the threads of
// k_columns meet the voxels (z slot fastest), where their reads and writes are
// whole lines; k_grad_natural brings them into natural order at the end of a call.
// In natural order every thread's read and write took a sector of its own: the
// gradient of two vectors on one GB300 at 24x24x96 313 us, now 254; 48x48x64 499,
// now 426.
struct GradStep {
  static constexpr bool kForward = false;
  const double* inv_phi;
  const double* gam;
  int kind, ax_a, ax_b;
  long long n;
  double scale;
  double* d_eps;  // slot order: [pair][a][x slot][b][z slot]
  double* dg;
  bool first;     // the sums so far are zero (and not read)
  template <int NB>
  struct Vals {};
  template <int NB>
  __device__ __forceinline__ void load(const ColumnPos&, int, Vals<NB>&) const {}
  template <int NB>
  __device__ __forceinline__ double apply(const ColumnPos& c, int b, const Vals<NB>&, int, double2& p, double2& q) const {
    const long long v = c.voxel(b);
    const long long at = ((((long long)c.j * c.N1 + c.a) * c.n1 + c.xs) * (c.n1 / c.N1) + b) * c.n3 + c.zs;
    const bool chiral = kind == kMediumChiral;
    const bool coupled = chiral || c.j == ax_a || c.j == ax_b;
    const double ip = inv_phi[c.j * n + v];
    const double g = coupled ? gam[(chiral ? c.j * n : 0) + v] : 0.0;
    const double2 s = mk(q.x - g * p.y, q.y + g * p.x);  // q + i g p
    const double s2 = cabs2(s);
    if (d_eps) d_eps[at] = (first ? 0.0 : d_eps[at]) + scale * (-s2 * ip * ip);
    if (dg && coupled) {
      const double2 i_p = cmul_i(p);
      const double re = s.x * i_p.x + s.y * i_p.y;  // Re(conj(s) i p)
      dg[at] = (first ? 0.0 : dg[at]) + scale * (2.0 * re * ip + 2.0 * g * s2 * ip * ip);
    }
    return 0.0;
  }
};

// The slot-order sums of a call in natural order (grid-stride over the voxels);
// pseudochiral: the two coupled pairs' added up.
__global__ void k_grad_natural(const double* __restrict__ eps, const double* __restrict__ g, int n1, int N2, int n3,
                               int Z2, bool chiral, int ax_a, int ax_b, double* __restrict__ d_eps,
                               double* __restrict__ d_gamma) {
  const long long n = (long long)n1 * n1 * n3;
  const int N1 = n1 / N2, Z1 = n3 / Z2;
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(v % n1), y = (int)(v / n1 % n1), z = (int)(v / ((long long)n1 * n1));
    const int xs = x % N1 * N2 + x / N1, zs = z % Z1 * Z2 + z / Z1;
    const long long at = (((long long)(y % N1) * n1 + xs) * N2 + y / N1) * n3 + zs;
    if (d_eps)
      for (int c = 0; c < 3; ++c) d_eps[c * n + v] = eps[c * n + at];
    if (d_gamma && chiral)
      for (int c = 0; c < 3; ++c) d_gamma[c * n + v] = g[c * n + at];
    if (d_gamma && !chiral) d_gamma[v] = g[ax_a * n + at] + g[ax_b * n + at];
  }
}

cudaError_t grad_natural_launch(const GradArgs& a, double* d_eps, double* d_gamma) {
  int N2 = 0, Z2 = 0;
  switch (a.n1) {
#define NFS_CASE(N) case N: N2 = PlaneSplit<double, N>::N2; break;
    NFS_FOR_EACH_SIZE(NFS_CASE)
#undef NFS_CASE
  }
  switch (a.n3) {
#define NFS_CASE(N) case N: Z2 = DepthSplit<double, N>::N2; break;
    NFS_FOR_EACH_SIZE(NFS_CASE)
#undef NFS_CASE
  }
  if (N2 == 0 || Z2 == 0) return cudaErrorInvalidValue;
  const long long n = (long long)a.n1 * a.n1 * a.n3;
  const int blocks = (int)std::min<long long>((n + 255) / 256, 152LL * 16);
  k_grad_natural<<<blocks, 256, 0, a.stream>>>(a.d_eps, a.dg, a.n1, N2, a.n3, Z2, a.kind == kMediumChiral, a.ax_a,
                                               a.ax_b, d_eps, d_gamma);
  return cudaGetLastError();
}

cudaError_t grad_launch(const GradArgs& a) {
  const GradStep step{a.inv_phi, a.gam, a.kind, a.ax_a, a.ax_b, (long long)a.n1 * a.n1 * a.n3, a.scale, a.d_eps, a.dg,
                      a.first};
  return columns_launch<double>(a.fld, step, a.tw1, a.tw3, a.n1, a.n3, 1, nullptr, nullptr, BatchStrides{}, a.stream);
}

// Physical fields of one eigenvector (Algorithm 1, final step):
//   x = [E; H] = B^{-1} diag(P_r, Q_r) y,   B = i [[zeta, mu], [-eps, -xi]].
// By eq. B_inv, B^{-1} [p; q] = [i w; -i f] with the same
//   w = Phi^{-1} (xi mu^{-1} p + q),   f = mu^{-1} (zeta w + p)
// that the middle factors of A_r form, so this is k_rows_in and k_columns up to
// the material step of the product.  The product
// never needs the Bloch twist D of T = n^{-1/2} D U (eq. mtx_T: it cancels
// against T^*); the fields do, so it is applied here from the three 1-D
// diagonals D_l[j] = exp(i 2 pi k.a_l j / n_l).  The two unnormalised DFTs
// leave sqrt(n) p, sqrt(n) q; inv_sqrt_n removes that factor.
struct FieldsStep {
  static constexpr bool kForward = false;
  ProductStep<double> material;  // scale 1 / sqrt(n)
  const double2* bloch;
  double2* X;
  template <int NB>
  using Vals = ProductStep<double>::Vals<NB>;
  template <int NB>
  __device__ __forceinline__ void load(const ColumnPos& c, int b, Vals<NB>& v) const {
    material.load<NB>(c, b, v);
  }
  template <int NB>
  __device__ __forceinline__ double apply(const ColumnPos& c, int b, const Vals<NB>& mv, int k, double2& p, double2& q) const {
    material.apply<NB>(c, b, mv, k, p, q);  // p <- f of axis s(j), q <- w of axis j
    const int y = c.a + c.N1 * b;
    const long long n = material.m.n, v = c.voxel(b);
    const double2 d = cmul(cmul(bloch[c.x], bloch[c.n1 + y]), bloch[2 * c.n1 + c.z]);
    const int s = pair_axis(material.m.kind, material.m.ax_a, material.m.ax_b, c.j);
    X[c.j * n + v] = cmul_i(cmul(d, q));         // E = i D w
    X[(3 + s) * n + v] = cmul_mi(cmul(d, p));    // H = -i D f
    return 0.0;
  }
};

cudaError_t fields_launch(const FieldsArgs& a) {
  const long long n = (long long)a.n1 * a.n1 * a.n3;
  const FieldsStep step{{{a.inv_phi, a.gam, a.inv_mu, nullptr, nullptr, a.kind, a.ax_a, a.ax_b, n},
                         1.0 / std::sqrt((double)n), 0},
                        a.bloch, a.X};
  return columns_launch<double>(a.fld, step, a.tw1, a.tw3, a.n1, a.n3, 1, nullptr, nullptr, BatchStrides{}, a.stream);
}

cudaError_t fields_prepare(int n1, int n3) {
  const cudaError_t e = columns_prepare<double, GradStep>(n1, n3);
  return e != cudaSuccess ? e : columns_prepare<double, FieldsStep>(n1, n3);
}

// Residual of an eigenpair (omega, x = [E; H]) in the GEP of eq.
// discrete_GEP_EH, diag(C, C^*) x = omega B x, with the Yee curl applied as
// its stencil (eqs. mtx_C, mtx_C123, mtx_K_n1): C_l is the forward difference
// along axis l over delta_l, the step past the last cell wrapping to the first
// times exp(i 2 pi k.a_l); C_l^* is the backward difference, wrapping with the
// conjugate phase.  Per voxel
//   B x = i [zeta E + mu H ; -eps E - xi H],
// with eps recovered from the stored 1 / Phi: chiral eps_c = Phi_c + gamma_c^2
// / mu_c, pseudochiral eps_a = Phi_a + gamma^2 / mu_b (and a <-> b).  Each
// block leaves two partial sums, |diag(C, C^*) x - omega B x|^2 and |B x|^2.
__global__ void __launch_bounds__(256) k_gep_residual(GepResidualArgs a) {
  using C = double2;
  const long long n1 = a.n1, n2 = a.n2, n3 = a.n3;
  const long long s3 = n1 * n2, n = s3 * n3;
  const C* X = a.X;
  double racc = 0.0, bacc = 0.0;
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x) {
    const long long i1 = v % n1, i2 = (v / n1) % n2, i3 = v / s3;
    // neighbours: forward (E) and backward (H) along each axis
    const bool fw[3] = {i1 == n1 - 1, i2 == n2 - 1, i3 == n3 - 1};
    const bool bw[3] = {i1 == 0, i2 == 0, i3 == 0};
    const long long step[3] = {1, n1, s3};
    const long long len[3] = {n1, n2, n3};
    C E[3], H[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      E[k] = X[k * n + v];
      H[k] = X[(3 + k) * n + v];
    }
    // fwd(c, l) = (C_l E_c)(v), bwd(c, l) = (C_l^* H_c)(v)
    auto fwd = [&](int c, int l) {
      const long long u = fw[l] ? v - (len[l] - 1) * step[l] : v + step[l];
      C e = X[c * n + u];
      if (fw[l]) e = cmul(a.wrap[l], e);
      return cscale(csub(e, E[c]), a.inv_delta[l]);
    };
    auto bwd = [&](int c, int l) {
      const long long u = bw[l] ? v + (len[l] - 1) * step[l] : v - step[l];
      C h = X[(3 + c) * n + u];
      if (bw[l]) h = cmulc(a.wrap[l], h);
      return cscale(csub(h, H[c]), a.inv_delta[l]);
    };
    const C CE[3] = {csub(fwd(2, 1), fwd(1, 2)), csub(fwd(0, 2), fwd(2, 0)), csub(fwd(1, 0), fwd(0, 1))};
    const C CH[3] = {csub(bwd(1, 2), bwd(2, 1)), csub(bwd(2, 0), bwd(0, 2)), csub(bwd(0, 1), bwd(1, 0))};
    double ip[3], im[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      ip[k] = a.inv_phi[k * n + v];
      im[k] = a.inv_mu ? a.inv_mu[k * n + v] : 1.0;
    }
    C zE[3], xH[3];
    double eps[3];
    if (a.kind == kMediumChiral) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const double g = a.gam[k * n + v];
        eps[k] = 1.0 / ip[k] + g * g * im[k];
        zE[k] = cmul_mi(cscale(E[k], g));  // zeta = -i gamma
        xH[k] = cmul_i(cscale(H[k], g));   // xi = i gamma
      }
    } else {
      const double g = a.gam[v];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int o = k == a.ax_a ? a.ax_b : (k == a.ax_b ? a.ax_a : -1);
        if (o >= 0) {
          eps[k] = 1.0 / ip[k] + g * g * im[o];
          zE[k] = cmul_mi(cscale(E[o], g));
          xH[k] = cmul_i(cscale(H[o], g));
        } else {
          eps[k] = 1.0 / ip[k];
          zE[k] = mk(0.0, 0.0);
          xH[k] = mk(0.0, 0.0);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const C bt = cmul_i(cadd(zE[k], cscale(H[k], 1.0 / im[k])));  // i (zeta E + mu H)
      const C bb = cmul_mi(cadd(cscale(E[k], eps[k]), xH[k]));      // -i (eps E + xi H)
      racc += cabs2(csub(CE[k], cscale(bt, a.omega))) + cabs2(csub(CH[k], cscale(bb, a.omega)));
      bacc += cabs2(bt) + cabs2(bb);
    }
  }
  const double rt = block_sum_dbl<256>(racc);
  const double bt = block_sum_dbl<256>(bacc);
  if (threadIdx.x == 0) {
    a.part[2 * blockIdx.x] = rt;
    a.part[2 * blockIdx.x + 1] = bt;
  }
}

cudaError_t gep_residual_launch(const GepResidualArgs& a, int blocks, cudaStream_t stream) {
  k_gep_residual<<<blocks, 256, 0, stream>>>(a);
  return cudaGetLastError();
}

cudaError_t basis_table_launch(const double2* lam, int n1, int n2, int n3, double alpha, double beta, double2* basis,
                               int P, int slam, long long sbasis, cudaStream_t stream) {
  const long long total = (long long)n1 * n2 * n3 * P;
  const int blocks = (int)std::min<long long>((total + 255) / 256, 152LL * 16);
  k_basis_table<double><<<blocks, 256, 0, stream>>>(lam, n1, n2, n3, alpha, beta, basis, P, slam, sbasis);
  return cudaGetLastError();
}

}  // namespace nfs
