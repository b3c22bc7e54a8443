// Size dispatch and launch of the product's kernels (see matvec_kernels.cuh).
#pragma once
#include <algorithm>

#include "matvec.h"
#include "matvec_kernels.cuh"

namespace nfs {

#define NFS_FOR_EACH_SIZE(M) M(8) M(12) M(16) M(24) M(32) M(48) M(64) M(96) M(128)

constexpr int round32(int x) { return (x + 31) / 32 * 32; }
constexpr int imin(int a, int b) { return a < b ? a : b; }
constexpr int imax(int a, int b) { return a > b ? a : b; }

#ifndef NFS_ROWS_NT
#define NFS_ROWS_NT 192
#endif
// Threads of the row kernels, and CTAs per SM requested from the compiler (its
// registers per thread).  Complex64: 768 threads per SM, 80 registers, which
// holds the 12 element pairs of a stage; 192 threads measured best at 48 to 96
// (96^3 CG iteration 90 us; 288 threads 94, three CTAs of 192 101), 384 at 128
// (245 us; 256 threads 253).  The scalar types take 128 registers.
template <typename R, int N>
struct RowsConfig {
  static constexpr int NF = ElemOf<R>::NF;
  static constexpr int ITEMS = 3 * N;  // of a stage with radix N1
  static constexpr int NT = NF == 2 ? (N == 128 ? 192 : N == 96 ? 160 : imin(96, round32(ITEMS))) : N == 128 ? 384 : N >= 48 ? NFS_ROWS_NT : round32(ITEMS);
  static constexpr int REGS_THREADS = NF == 1 ? 768 : 512;  // threads per SM that the register budget is cut for
  static constexpr int BY_SMEM = (int)(kMaxDynSmem / (rows_smem<R, N>() + 1024));
  static constexpr int MINB = imax(1, imin(imin(BY_SMEM, 12), REGS_THREADS / NT));
};

// Likewise for k_columns: NF L Z2 (or Z1) items in the z stages, X N3 in the y
// stage.
template <typename R, int N2, int X, int N3>
struct ColumnsConfig {
  static constexpr int NF = ElemOf<R>::NF;
  using S = DepthSplit<R, N3>;
  static constexpr int ITEMS = imax(NF * X * N3, NF * N2 * X * S::N2);
  static constexpr int NT = NF == 2 ? imin(128, round32(ITEMS)) : ITEMS <= 192 ? round32(ITEMS) : 128;
  static constexpr int REGS_THREADS = NF == 1 ? (N3 == 128 ? 640 : 768) : 512;  // (128: radix 16 needs 102 registers)
  static constexpr int BY_SMEM = (int)(kMaxDynSmem / (columns_smem<R, N2, X, N3>() + 1024));
  static constexpr int MINB = imax(1, imin(imin(BY_SMEM, 12), REGS_THREADS / NT));
};

template <typename R, int N>
constexpr auto rows_in_kernel() {
  return k_rows_in<R, N, RowsConfig<R, N>::NT, RowsConfig<R, N>::MINB>;
}
template <typename R, int N>
constexpr auto rows_out_kernel() {
  return k_rows_out<R, N, RowsConfig<R, N>::NT, RowsConfig<R, N>::MINB>;
}
template <typename R, class T, int N3, class Step>
constexpr auto columns_kernel() {
  using K = ColumnsConfig<R, T::N2, T::X, N3>;
  return k_columns<R, T::N2, T::X, T::XL, N3, K::NT, K::MINB, Step>;
}

// (up to 48 KB need no opting in, and the call costs a context of a small grid
// more time than its kernels take)
template <typename K>
static cudaError_t allow_smem(K* kernel, size_t bytes) {
  if (bytes <= 48 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// f(tag) with the column tile of plane edge n1: tag::N2, tag::X, tag::XL
template <int N2_, int X_, int XL_>
struct ColumnTile {
  static constexpr int N2 = N2_, X = X_, XL = XL_;
};
template <typename R, typename F>
static cudaError_t with_column_tile(int n1, F f) {
  switch (n1) {
#define NFS_CASE(N) case N: return f(ColumnTile<PlaneSplit<R, N>::N2, PlaneSplit<R, N>::X, PlaneSplit<R, N>::XL>{});
    NFS_FOR_EACH_SIZE(NFS_CASE)
#undef NFS_CASE
  }
  return cudaErrorInvalidValue;
}

// Launch with programmatic stream serialisation (see depend_wait), unless the
// tables were written on the stream a moment ago (`serial`) or it does not pay:
// CTAs that start early are placed on the SMs that happen to be free, which is
// harmless while the kernels are short (complex64 products on GB300, us: 8^3
// 7.0 -> 5.5, 32^3 10.2 -> 8.7, 64^3 22.7 -> 21.3, 96^3 65.6 -> 63.1; but 128^3
// 173.6 -> 177.4) and costly where every SM's share of the FP64 work counts
// (complex128 8^3 15.0 -> 13.3, but 32^3 66 -> 73, 48x48x32 134 -> 191), so the
// scalar types overlap only products with at most one CTA per SM.
template <typename R>
static bool overlap(int n1, int n3, int P) {
  if (ElemOf<R>::NF == 1) return n1 < 128;
  int N2 = 1, X = 1;
  with_column_tile<R>(n1, [&](auto tag) {
    N2 = decltype(tag)::N2;
    X = decltype(tag)::X;
    return cudaSuccess;
  });
  return std::max(2 * N2 * n3, 3 * (n1 / N2) * (n1 / X)) * P <= 152;
}
template <typename... P, typename... A>
static cudaError_t launch_dependent(bool serial, void (*kernel)(P...), dim3 grid, int threads, size_t smem,
                                    cudaStream_t s, A... a) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = serial ? 0 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(a)...);
}

template <typename R, class Step>
static cudaError_t columns_prepare(int n1, int n3) {
  return with_column_tile<R>(n1, [&](auto tag) -> cudaError_t {
    using T = decltype(tag);
    switch (n3) {
#define NFS_CASE(N) case N: return allow_smem(columns_kernel<R, T, N, Step>(), columns_smem<R, T::N2, T::X, N>());
      NFS_FOR_EACH_SIZE(NFS_CASE)
#undef NFS_CASE
    }
    return cudaErrorInvalidValue;
  });
}

template <typename R, class Step>
static cudaError_t columns_launch(void* fld, const Step& step, const cplx<R>* tw1, const cplx<R>* tw3, int n1, int n3,
                                  int P, const int* skip, CGState* st, const BatchStrides& bs, cudaStream_t s,
                                  bool serial = false) {
  return with_column_tile<R>(n1, [&](auto tag) -> cudaError_t {
    using T = decltype(tag);
    const dim3 grid(n1 / T::X, n1 / T::N2, 3 * P);
    auto* f = static_cast<typename ElemOf<R>::E*>(fld);
    switch (n3) {
#define NFS_CASE(N)                                                                              \
  case N:                                                                                        \
    return launch_dependent(serial || !overlap<R>(n1, n3, P), columns_kernel<R, T, N, Step>(), grid, ColumnsConfig<R, T::N2, T::X, N>::NT, \
                            columns_smem<R, T::N2, T::X, N>(), s, f, step, tw1, tw3, skip, st, bs);
      NFS_FOR_EACH_SIZE(NFS_CASE)
#undef NFS_CASE
    }
    return cudaErrorInvalidValue;
  });
}

template <typename R, int N>
static cudaError_t rows_prepare_n() {
  cudaError_t e = allow_smem(rows_in_kernel<R, N>(), rows_smem<R, N>());
  return e != cudaSuccess ? e : allow_smem(rows_out_kernel<R, N>(), rows_smem<R, N>());
}

static inline NoKrylov krylov_of(const KrylovFuse&, NoKrylov) { return {}; }
static inline KrylovFuse krylov_of(const KrylovFuse& k, KrylovFuse) { return k; }

template <typename R, int N>
static cudaError_t rows_launch_n(const MatvecArgs<R>& a, bool in) {
  const dim3 grid(PlaneSplit<R, N>::N2 * ElemOf<R>::NF, a.n3, a.P > 0 ? a.P : 1);
  auto* f = static_cast<typename ElemOf<R>::E*>(a.fld);
  constexpr int NT = RowsConfig<R, N>::NT;
  const auto kr = krylov_of(a.kr, typename KrylovOf<R>::type{});
  const bool serial = a.serial || !overlap<R>(N, a.n3, a.P > 0 ? a.P : 1);
  if (in)
    return launch_dependent(serial, rows_in_kernel<R, N>(), grid, NT, rows_smem<R, N>(), a.stream, a.u, f, a.lam, a.tw1,
                            a.alpha, a.beta, a.kind, a.ax_a, a.ax_b, a.skip, a.basis, a.bs, a.cg, kr);
  return launch_dependent(serial, rows_out_kernel<R, N>(), grid, NT, rows_smem<R, N>(), a.stream, f, a.Au, a.lam, a.tw1,
                          a.alpha, a.beta, a.kind, a.ax_a, a.ax_b, a.skip, a.basis, a.bs, a.cg, kr);
}

template <typename R>
cudaError_t rows_prepare(int n1) {
  switch (n1) {
#define NFS_CASE(N) case N: return rows_prepare_n<R, N>();
    NFS_FOR_EACH_SIZE(NFS_CASE)
#undef NFS_CASE
  }
  return cudaErrorInvalidValue;
}

template <typename R>
cudaError_t rows_launch(const MatvecArgs<R>& a, bool in) {
  switch (a.n1) {
#define NFS_CASE(N) case N: return rows_launch_n<R, N>(a, in);
    NFS_FOR_EACH_SIZE(NFS_CASE)
#undef NFS_CASE
  }
  return cudaErrorInvalidValue;
}

template <typename R>
cudaError_t product_columns_prepare(int n1, int n3) {
  return columns_prepare<R, ProductStep<R>>(n1, n3);
}

template <typename R>
cudaError_t product_columns_launch(const MatvecArgs<R>& a) {
  const long long n = (long long)a.n1 * a.n1 * a.n3;
  const ProductStep<R> step{{a.inv_phi, a.gam, a.inv_mu, a.pmat, a.pmu, a.kind, a.ax_a, a.ax_b, n},
                            (R)(1.0 / (double)n), a.bs.smat};
  return columns_launch<R>(a.fld, step, a.tw1, a.tw3, a.n1, a.n3, a.P > 0 ? a.P : 1, a.skip, a.cg.st, a.bs, a.stream,
                           a.serial);
}

template <typename R>
int cg_partials(int n1, int n3) {
  switch (n1) {
#define NFS_CASE(N) case N: return PlaneSplit<R, N>::N2 * ElemOf<R>::NF * n3;
    NFS_FOR_EACH_SIZE(NFS_CASE)
#undef NFS_CASE
  }
  return 0;
}

// (the two halves may be instantiated in different translation units)
#define NFS_INSTANTIATE_ROWS(R)                                     \
  template int cg_partials<R>(int, int);                            \
  template cudaError_t rows_prepare<R>(int);                        \
  template cudaError_t rows_launch<R>(const MatvecArgs<R>&, bool);
#define NFS_INSTANTIATE_COLUMNS(R)                                  \
  template cudaError_t product_columns_prepare<R>(int, int);        \
  template cudaError_t product_columns_launch<R>(const MatvecArgs<R>&);

}  // namespace nfs
