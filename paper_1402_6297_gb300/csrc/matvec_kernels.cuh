// The A_r matrix-vector product of the HHPD-NFGEP (eq. factor_mtx, applied as
// in eq. spd_LS) in three kernels, for complex64, complex128 and
// double-single vectors.
//
// A line DFT of length N = N1 N2 runs in two register stages.  Inverse:
// stage A forms, for every n2 < N2, the radix-N1 DFT of the elements
// n1 N2 + n2 and the twiddles w_N^{n2 k1}; stage B forms, for every k1 < N1,
// the radix-N2 DFT of the slots k1 N2 + n2.  Both work in place (they write
// the slots they read), which leaves element k1 + N1 k2 in slot k1 N2 + k2;
// nothing in real space cares where an element sits, so it stays there.  The
// forward transform undoes the two stages in turn: A' over the slots of one
// k1, then B' over all k1 at one offset, which ends in natural order.
// No stage has a hazard between its reads and its writes.
//
// Stage A of the y transform needs N1 rows of a plane, stage B then only the
// N2 slots of one k1, so the y transform is split between the kernels and no
// kernel holds a plane:
//
//   k_rows_in   (CTA: z index i3, n2 = b;  the N1 rows y = n1 N2 + b):  CG
//               direction, spectral assembly p^ = P_r-coefficients,
//               q^ = Q_r-coefficients, inverse DFT along x, stage A along y.
//   k_columns   (CTA: pair j, k1 = a, X slots of x;  all z, the N2 slots of
//               a):  inverse DFT along z; then per (z, x) stage B along y, the
//               material product of eq. factor_mtx and stage A' along y, all in
//               registers; forward DFT along z.
//   k_rows_out  (CTA: i3, b;  the N1 rows y = b + N2 k):  stage B' along y,
//               forward DFT along x, the projections P_r^* f, Q_r^* w, and in CG
//               the step x += alpha p, r -= alpha A_r p.
//
// Why this split.  Holding whole xy planes between two plane passes and a z
// pass (the form measured before) took 12 shared-memory round trips per
// element against 10 here, read every input in three CTAs (one per component)
// or exchanged it through a cluster, and needed 149 KB per CTA at 96 x 96, one
// CTA per SM with its loads, transforms and stores one after another.  Here a
// complex64 CTA holds 38.8 KB (rows) or 40.1 KB (columns) at 96^3 (complex128:
// 57.4 and 52.4), several share an SM and overlap, all six fields of a voxel are in one CTA of the row kernels, and on
// small grids the work spreads over more SMs, which is what complex128 needs:
// GB300 retires one FP64 warp instruction per ~16 cycles and SM.
//
// Pairs.  The material couples p and q of one voxel only inside three pairs:
// w_j = Phi_j^{-1} (q_j + i g mu^{-1} p_s(j)) and f_s(j) = mu^{-1} (p_s(j) -
// i g w_j), with s the identity (chiral) or the exchange of the coupled axes
// (pseudochiral; g = 0 for the third).  A CTA of k_columns therefore owns one
// pair.  In complex64 the two fields of a pair also share one element: two
// packed f32x2 registers hold (Re p, Re q) and (Im p, Im q) (fft_pk.cuh), so
// every butterfly treats both lines in one instruction and every shared access
// moves 16 bytes.  The other types keep p and q in separate lines.
//
// Workspace: E fld[j][f][a][x / XL][z][b][x % XL], f < NF.
//
// Basis per spectral voxel (Section 2), with a = (Lambda_1, Lambda_2, Lambda_3),
// t = (alpha, beta, 1), Lambda_p = t x a, Lambda_q = |a|^2:
//   c  = Lambda_p / |Lambda_p|                  (= conj Pi_2, eq. mtx_Pi_2)
//   x  = (a / sqrt(Lambda_q)) x conj(c)          (= Pi_0 x Pi_2 = conj Pi_1)
// so that P_r = (I3 (x) T)[-c, x] and Q_r = (I3 (x) T)[conj x, conj c]
// (eq. mtx_QdPd, SVD theorem thm:svd_C).  x equals conj(Pi_1) because
// Pi_1 = (conj(a) x Lambda_p) / sqrt(Lambda_q |Lambda_p|^2), the unit-norm
// reading of eq. mtx_Pi_1.
//
// The Bloch twist D of T (eq. mtx_T) is a per-voxel unit scalar and commutes
// with the per-voxel material product, so it cancels between T and T^*: the
// kernels run plain DFTs.  The two unnormalised DFTs give a factor n, removed
// in the material step (T = D U / sqrt(n)).
#pragma once
#include <type_traits>

#include "cg_state.cuh"
#include "fft_pk.cuh"
#include "matvec.h"

namespace nfs {

constexpr int kMediumChiral = 0;
constexpr int kMediumPseudochiral = 1;

// Per-voxel real-space material (Section 4.3 with diagonal eps and mu):
//   inv_phi[3][n] = 1 / Phi_c, Phi = eps - xi mu^{-1} zeta (diagonal here)
//   gam     chiral [3][n] gamma_c; pseudochiral [n] gamma
//   inv_mu  [3][n] = 1 / mu_c, or nullptr for mu = 1
// in natural order, or (complex64 products) in the order k_columns meets them:
// pair j, voxel (slot order) -> pmat = {1 / Phi_j, g} for two neighbouring b
// and pmu = mu^{-1}_s(j) likewise (see pair_material_launch).
template <typename R>
struct MatView {
  const R* inv_phi;
  const R* gam;
  const R* inv_mu;
  const float4* pmat;
  const float2* pmu;
  int kind;
  int ax_a, ax_b;
  long long n;
};

// Programmatic dependent launch (the kernels of a product are launched so that
// the next one may start while the last CTAs of the one before still run):
// depend_begin() lets the next kernel of the stream start, depend_wait() waits
// for the one before to end with its writes visible.  Every CTA waits before it
// touches anything but constant tables, and before it returns: a kernel that
// ended earlier would let its successor run ahead of its predecessor.
//
// Such a kernel is alive while its predecessor writes, so what any kernel on the
// stream writes is read by plain loads from plain pointers: __ldg and const
// __restrict__ promise the compiler and the hardware that the data does not
// change during the kernel's life (a load may then move above the wait, whose
// "memory" clobber does not reach a __restrict__ pointer).  Only the tables of
// set-up (lam, tw*, basis, the material) keep them.
__device__ __forceinline__ void depend_begin() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void depend_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Partner axis of pair j: s(j).
__host__ __device__ __forceinline__ int pair_axis(int kind, int ax_a, int ax_b, int j) {
  if (kind == kMediumChiral) return j;
  return j == ax_a ? ax_b : (j == ax_b ? ax_a : j);
}

// Sum of one double per thread over the block (result valid in thread 0).
template <int NT>
__device__ __forceinline__ double block_sum_dbl(double v) {
  __shared__ double sh[NT / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  double r = 0.0;
  if (warp == 0) {
    r = lane < NT / 32 ? sh[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  }
  __syncthreads();
  return r;
}

// ---------------------------------------------------------------------------
// schedule
// ---------------------------------------------------------------------------

// N = N1 N2 of the x and y transforms (N1 rows per CTA of the row kernels, N2
// slots of y per CTA of k_columns), X, the x slots of a CTA of k_columns, and
// XL, the x slots that lie together in the workspace.
// N2 = 8 keeps the items of every stage within a thread's registers up to 128;
// 96 and 48 take 12 in complex64: 8 rows instead of 12 fit four CTAs per SM and
// divide evenly (7.6 CTAs per SM instead of 5.05).  Measured on GB300 at 96^3,
// rows in / columns / rows out in us: 17.7 / 23.2 / 18.9 against 21.7 / 21.6 /
// 19.7 with N2 = 8.  XL = 4: the row kernels reach the workspace in runs of XL
// elements, k_columns in runs of X; XL = X = 2 gave 20.1 / 20.9 / 21.5, XL = 8
// 16.7 / 28.4 / 17.9 (products: 63.8 us with XL = 4, 66.8, 67.5).  X = 2 against
// X = 4: a product of 63.8 against 68.4 us (smaller CTAs, more of them per SM).
// The smallest grids take N2 = 4 and X = 1 to have CTAs for the whole GPU (8^3:
// 32 row CTAs and 48 column CTAs), and complex128 at 32 takes X = 1: with X = 2
// its 192 column CTAs leave one on most SMs and two on some, which take twice as
// long where the FP64 pipe is what counts.  Columns with X = 2 and X = 1 in us:
// 32x32 35.1 and 28.9, 32x96 117.6 and 92.3, 32x128 158 and 121; products: 72.0
// and 65.9, 209 and 183, 269 and 232 (the plane passes before: 90.5, 183, 249).
// At 48 the two are equal, at 64 X = 1 is slower up to 24 of z and 4% faster from
// 48 on; the double-single product gains nothing (80 and 79 us at 32x96).
#ifndef NFS_N2_48
#define NFS_N2_48 12
#endif
#ifndef NFS_N2_96
#define NFS_N2_96 12
#endif
#ifndef NFS_X
#define NFS_X 2
#endif
#ifndef NFS_XL
#define NFS_XL 4
#endif
constexpr int common_divisor(int a, int b) { return b == 0 ? a : common_divisor(b, a % b); }
template <typename R, int N> struct PlaneSplit {
  static constexpr bool F32 = sizeof(cplx<R>) == 8;
  static constexpr int N2 = N < 24 ? 4 : (F32 && N == 48) ? NFS_N2_48 : (F32 && N == 96) ? NFS_N2_96 : 8, N1 = N / N2;
  static constexpr int X = N < 24 || (N == 32 && std::is_same<R, double>::value) ? 1 : NFS_X;
  // (whole runs of whole tiles: the largest part of NFS_XL that divides the
  // edge, but no shorter than a tile.  A run that does not divide it would share
  // its room with the next row's, and leave the workspace at its end)
  static constexpr int RUN = common_divisor(N, NFS_XL);
  static constexpr int XL = RUN % X == 0 ? RUN : X;
  static_assert(N % N2 == 0 && N % XL == 0 && XL % X == 0, "the x slots of a row come in whole runs of whole tiles");
};

// N = N1 N2 of the z transforms.  The packed elements take the shortest lengths
// in one stage; complex128 and double-single ones in two, so that more lanes of
// the few warps work on a small tile (an FP64 warp instruction occupies its
// pipe for ~16 cycles whether 8 or 32 lanes are active).
template <typename R, int N> struct DepthSplit : LineSplit<N> {};
template <> struct DepthSplit<float, 8> { static constexpr int N1 = 8, N2 = 1; };
template <> struct DepthSplit<float, 12> { static constexpr int N1 = 12, N2 = 1; };
template <> struct DepthSplit<float, 16> { static constexpr int N1 = 16, N2 = 1; };

// Elements of the workspace and of shared memory, and how many of them hold
// the two fields of a pair.
template <typename R> struct ElemOf {
  using E = cplx<R>;
  static constexpr int NF = 2;
};
template <> struct ElemOf<float> {
  using E = cp2;
  static constexpr int NF = 1;
};

// One register DFT on elements of either kind.
template <int L, bool INV> __device__ __forceinline__ void edft(cp2* x) { PDFT<L, INV>::run(x); }
template <int L, bool INV, typename C> __device__ __forceinline__ void edft(C* x) { DFT<L, INV>::run(x); }

// Twiddles: the table holds exp(-2 pi i m / N); packed elements keep each one
// as {(cos, cos), (-sin, -sin)}.
__device__ __forceinline__ cp2 tw_entry(float2 w) { return {splat(w.x), splat(w.y)}; }
template <typename C> __device__ __forceinline__ C tw_entry(C w) { return w; }
template <bool INV> __device__ __forceinline__ cp2 etwiddle(cp2 a, cp2 w) { return INV ? pmul_tw_conj(a, w) : pmul_tw(a, w); }
template <bool INV, typename C> __device__ __forceinline__ C etwiddle(C a, C w) { return INV ? cmulc(w, a) : cmul(a, w); }

// Elements of a pair from and to its two complex fields (scalar elements: one
// field per element, `stride` apart).
__device__ __forceinline__ void put_pair(cp2* line0, int stride, float2 p, float2 q) {
  (void)stride;
  *line0 = {f2pk(p.x, q.x), f2pk(p.y, q.y)};
}
template <typename C> __device__ __forceinline__ void put_pair(C* line0, int stride, C p, C q) {
  line0[0] = p;
  line0[stride] = q;
}
__device__ __forceinline__ void get_pair(const cp2* line0, int stride, float2& p, float2& q) {
  (void)stride;
  const cp2 v = *line0;
  const float2 re = pk2f(v.re), im = pk2f(v.im);
  p = mk(re.x, im.x);
  q = mk(re.y, im.y);
}
template <typename C> __device__ __forceinline__ void get_pair(const C* line0, int stride, C& p, C& q) {
  p = line0[0];
  q = line0[stride];
}

// Vector elements in memory to and from the type computed in.
template <typename R, typename V> __device__ __forceinline__ cplx<R> from_vec(V v) {
  if constexpr (std::is_same<cplx<R>, V>::value) return v;
  else return cplx<R>{R(v.x), R(v.y)};
}
template <typename R> __device__ __forceinline__ vecc<R> to_vec(cplx<R> v) {
  if constexpr (std::is_same<cplx<R>, vecc<R>>::value) return v;
  else return vecc<R>{(double)v.x, (double)v.y};
}

template <typename C> __device__ __forceinline__ void cswap(C& a, C& b) {
  const C t = a;
  a = b;
  b = t;
}
// Exchange the entries of the coupled pair (a, b) of a pseudochiral medium.
template <typename C> __device__ __forceinline__ void swap_axes(C* v, int ax_a, int ax_b) {
  const int s = ax_a + ax_b;  // 1: x-y, 2: x-z, 3: y-z
  if (s == 1) cswap(v[0], v[1]);
  else if (s == 2) cswap(v[0], v[2]);
  else cswap(v[1], v[2]);
}

template <typename R>
struct Basis {
  cplx<R> c[3];
  cplx<R> x[3];
};

template <typename R>
__device__ __forceinline__ void make_basis(cplx<R> a1, cplx<R> a2, cplx<R> a3, R al, R be, Basis<R>& B) {
  using C = cplx<R>;
  // Lambda_p = t x a  (eq. mtx_Lambda_p_q)
  const C p1 = mk(be * a3.x - a2.x, be * a3.y - a2.y);
  const C p2 = mk(a1.x - al * a3.x, a1.y - al * a3.y);
  const C p3 = mk(al * a2.x - be * a1.x, al * a2.y - be * a1.y);
  const R lp2 = cabs2(p1) + cabs2(p2) + cabs2(p3);
  const R lq = cabs2(a1) + cabs2(a2) + cabs2(a3);
  const R rp = rsqrt(lp2);
  const R rq = rsqrt(lq);
  B.c[0] = cscale(p1, rp);
  B.c[1] = cscale(p2, rp);
  B.c[2] = cscale(p3, rp);
  // x = (a / sqrt(Lq)) x conj(c):  x_1 = a2 conj(c3) - a3 conj(c2), cyclic
  B.x[0] = cscale(csub(cmulc(B.c[2], a2), cmulc(B.c[1], a3)), rq);
  B.x[1] = cscale(csub(cmulc(B.c[0], a3), cmulc(B.c[2], a1)), rq);
  B.x[2] = cscale(csub(cmulc(B.c[1], a1), cmulc(B.c[0], a2)), rq);
}

// The basis of spectral voxel v: from the table when there is one, else from
// the Lambda tables.
template <typename R>
__device__ __forceinline__ void voxel_basis(const cplx<R>* __restrict__ table, long long n, long long v, cplx<R> a1,
                                            cplx<R> a2, cplx<R> a3, R al, R be, Basis<R>& B) {
  if (table != nullptr) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      B.c[k] = table[k * n + v];
      B.x[k] = table[(3 + k) * n + v];
    }
  } else {
    make_basis<R>(a1, a2, a3, al, be, B);
  }
}

// Table of the basis (complex128 products use it: double-precision square
// roots are scarce on this GPU).  Grid-stride over P x n voxels.
template <typename R>
__global__ void k_basis_table(const cplx<R>* __restrict__ lam, int n1, int n2, int n3, R al, R be,
                              cplx<R>* __restrict__ table, int P, int slam, long long sbasis) {
  const long long n = (long long)n1 * n2 * n3;
  for (long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x; g < n * P; g += (long long)gridDim.x * blockDim.x) {
    const long long p = g / n, v = g % n;
    const int i1 = (int)(v % n1), i2 = (int)((v / n1) % n2), i3 = (int)(v / ((long long)n1 * n2));
    const cplx<R>* L = lam + p * slam;
    Basis<R> B;
    make_basis<R>(L[i1], L[n1 + i2], L[n1 + n2 + i3], al, be, B);
    cplx<R>* t = table + p * sbasis;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      t[k * n + v] = B.c[k];
      t[(3 + k) * n + v] = B.x[k];
    }
  }
}

// ---------------------------------------------------------------------------
// stages over lines in shared memory: element e of line l at buf[l LS + e ES]
// (work items take the line index fastest across threads; the callers'
// pitches are odd, so the 16-byte accesses of 8 neighbouring lanes hit 8
// different bank groups)
// ---------------------------------------------------------------------------

// Inverse stage A (or, FWD = true, forward stage B'): radix N1 over the slots
// n1 N2 + n2 of one n2; the inverse stage multiplies by its twiddles.
template <bool FWD, int N1, int N2, int NLINES, int NT, int LS, int ES, typename E>
__device__ __forceinline__ void stage_strided(E* buf, const E* tw) {
  constexpr int ITEMS = NLINES * N2;
#pragma unroll 1
  for (int it = threadIdx.x; it < ITEMS; it += NT) {
    const int l = it % NLINES, n2 = it / NLINES;
    E* base = buf + l * LS + n2 * ES;
    E r[N1];
#pragma unroll
    for (int n1 = 0; n1 < N1; ++n1) r[n1] = base[n1 * N2 * ES];
    edft<N1, !FWD>(r);
    if (!FWD) {
#pragma unroll
      for (int k1 = 1; k1 < N1; ++k1) r[k1] = etwiddle<true>(r[k1], tw[n2 * k1]);
    }
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) base[k1 * N2 * ES] = r[k1];
  }
}

// Inverse stage B (or, FWD = true, forward stage A'): radix N2 over the slots
// k1 N2 + n2 of one k1; the forward stage multiplies by its twiddles.
template <bool FWD, int N1, int N2, int NLINES, int NT, int LS, int ES, typename E>
__device__ __forceinline__ void stage_group(E* buf, const E* tw) {
  constexpr int ITEMS = NLINES * N1;
#pragma unroll 1
  for (int it = threadIdx.x; it < ITEMS; it += NT) {
    const int l = it % NLINES, k1 = it / NLINES;
    E* base = buf + l * LS + k1 * N2 * ES;
    E r[N2];
#pragma unroll
    for (int i = 0; i < N2; ++i) r[i] = base[i * ES];
    edft<N2, !FWD>(r);
    if (FWD) {
#pragma unroll
      for (int i = 1; i < N2; ++i) r[i] = etwiddle<false>(r[i], tw[k1 * i]);
    }
#pragma unroll
    for (int i = 0; i < N2; ++i) base[i * ES] = r[i];
  }
}

// ---------------------------------------------------------------------------
// k_rows_in: grid (N2 NF, n3, P); scalar elements: a CTA takes one field of
// each pair (P_r u1 or Q_r u2)
// ---------------------------------------------------------------------------
// a - sum_{g < G} tmp[g stride], eight loads in flight at a time
__device__ __forceinline__ double2 minus_groups(double2 a, const double2* tmp, long long stride, int G) {
  for (int g0 = 0; g0 < G; g0 += 8) {
    double2 x[8];
#pragma unroll
    for (int t = 0; t < 8; ++t)
      if (g0 + t < G) x[t] = tmp[(g0 + t) * stride];
#pragma unroll
    for (int t = 0; t < 8; ++t)
      if (g0 + t < G) a = csub(a, x[t]);
  }
  return a;
}

// Whether a thread of the scalar types' kernels fetches all that its items read
// (nv of them, nt threads, `per` items per thread at most) when the kernel
// starts.  The grids this holds for are bound by the chain of latencies from
// one kernel to the next, not by the FP64 pipe: an item's operands fetched where
// they are used add an L2 round trip behind each barrier.  CG iterations in
// complex128 on GB300: 8^3 20.1 -> 19.4 us, 16^3 22.2 -> 21.5.  (On larger grids
// a thread has several items, whose operands would not fit in its registers,
// and other CTAs of the SM fill the gap.)
template <typename R>
__host__ __device__ constexpr bool kAhead(int nv, int nt, int per = 1) {
  return sizeof(cplx<R>) == 16 && nv <= per * nt;
}

// Whether the row kernels of a CG step look whether there is anything left to do
// before they fetch anything else.  The steps of a chunk that are left when a
// solve has converged are empty then; else k_rows_in adds up the partials and
// k_rows_out transforms a workspace for nothing.  An empty step on GB300, us: complex128 32x32x96 21 and 8.5, 48^3 27 and 6.5, 64^3 41 and 8.5;
// complex64 96^3 16 and 8, 128x128x64 24 and 10.  The price is a latency ahead of
// everything in every step: nothing on these grids, but 0.5 us of 69.7 in
// complex128 at 32^3, and in complex64 0.3 of 12.9 at 32^3 and 0.5 of 29 at 64^3,
// more than the empty steps of a solve.  So complex64 edges from 96 on and
// complex128 ones from 32, with workspaces of 8 MB and more.
template <typename R, int N>
__device__ __forceinline__ bool stop_first(int n3) {
  if constexpr (N < (sizeof(cplx<R>) == 8 ? 96 : 32)) return false;
  return 6LL * N * N * n3 * (long long)sizeof(cplx<R>) >= (8LL << 20);
}

// (only complex128 kernels carry the Krylov pieces)
struct NoKrylov {};
template <typename R> struct KrylovOf { using type = NoKrylov; };
template <> struct KrylovOf<double> { using type = KrylovFuse; };

template <typename R, int N>
constexpr size_t rows_smem() {
  return (size_t)(3 * PlaneSplit<R, N>::N1 * (N + 1) + N) * 16;
}

template <typename R, int N, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB)
k_rows_in(const vecc<R>* u, typename ElemOf<R>::E* fld, const cplx<R>* __restrict__ lam,
          const cplx<R>* __restrict__ twx, R alpha, R beta, int kind, int ax_a, int ax_b, const int* skip,
          const cplx<R>* __restrict__ basis, BatchStrides bs, CgFuse<R> cg, typename KrylovOf<R>::type kr) {
  using C = cplx<R>;
  using E = typename ElemOf<R>::E;
  using S = PlaneSplit<R, N>;
  constexpr int NF = ElemOf<R>::NF, N1 = S::N1, N2 = S::N2, X = S::X, XL = S::XL;
  constexpr int PITCH = N + 1;
  constexpr int LINES = 3 * N1;  // line j N1 + row
  extern __shared__ __align__(16) unsigned char smem_raw[];
  E* buf = reinterpret_cast<E*>(smem_raw);
  E* tw = buf + LINES * PITCH;
  const int b = blockIdx.x % N2, fsel = blockIdx.x / N2, i3 = blockIdx.y, prob = blockIdx.z, n3 = gridDim.y;
  for (int i = threadIdx.x; i < N; i += NT) tw[i] = tw_entry(twx[i]);
  depend_wait();
  if (skip != nullptr && skip[(long long)prob * bs.sskip]) return;
  constexpr bool CGT = !std::is_same<R, df>::value;  // (the double-single product never runs CG)
  CGState* st = (CGT && cg.st != nullptr) ? cg.st + prob : nullptr;
  if (st != nullptr && stop_first<R, N>(n3) && st->halt) {
    if (blockIdx.x == 0 && i3 == 0 && threadIdx.x == 0) st->stop = 1;
    return;
  }
  if (st != nullptr) u = cg.p;
  u += prob * bs.su;
  fld += prob * bs.sfld;
  lam += (long long)prob * bs.slam;
  if (basis != nullptr) basis += prob * bs.sbasis;
  const vecc<R>* r_in = st != nullptr ? cg.r + prob * bs.su : nullptr;
  const long long n = (long long)N * N * n3;
  // the quarters of u that this CTA needs: all, or the two of its field
  constexpr int NQ = 4 / NF;
  const int q0 = NF == 1 ? 0 : 2 * fsel;
  // the first voxel's inputs are on their way while (in CG) the partials of
  // r^* r are summed; each later voxel's while the one before it is assembled
  constexpr int NV = N1 * N;
  vecc<R> v[NQ], g[NQ];
  auto fetch = [&](int vi) {
    if (vi < NV) {
      const long long e = ((long long)i3 * N + (vi / N) * N2 + b) * N + vi % N + q0 * n;
#pragma unroll
      for (int q = 0; q < NQ; ++q) v[q] = u[q * n + e];
      if (r_in != nullptr) {
#pragma unroll
        for (int q = 0; q < NQ; ++q) g[q] = r_in[q * n + e];
      }
    }
  };
  fetch(threadIdx.x);
  // (one voxel per thread: its basis too; see kAhead)
  constexpr bool AHEAD = kAhead<R>(NV, NT);
  Basis<R> B;
  if constexpr (AHEAD) {
    if (threadIdx.x < NV) {
      const int x = threadIdx.x % N, y = threadIdx.x / N * N2 + b;
      voxel_basis<R>(basis, n, ((long long)i3 * N + y) * N + x, lam[x], lam[N + y], lam[2 * N + i3], alpha, beta, B);
    }
  }
  R bt = (R)0;
  if constexpr (CGT) {
    if (st != nullptr) {
      using P = typename RedAccFor<R>::partial;
      const P tol2 = *reinterpret_cast<const P*>(&st->tol2), last = *reinterpret_cast<const P*>(&st->rr_last);
      const bool over = (st->halt != 0) | (st->it >= st->maxit);
      const P rr = sum_partials_all<R, NT>(st->part_b, gridDim.x * n3);
      const bool stop = over || scalar_nan(rr) || scalar_le(rr, tol2);
      if (blockIdx.x == 0 && i3 == 0 && threadIdx.x == 0) {
        st->stop = stop;
        *reinterpret_cast<P*>(&st->rr_now) = rr;
      }
      if (stop) return;
      bt = (R)scalar_ratio(rr, last);
    }
  }
  const C a3 = lam[2 * N + i3];
  RedAccFor<R> nrm_acc;
#pragma unroll 1
  for (int vi = threadIdx.x; vi < NV; vi += NT) {
    const int row = vi / N, x = vi % N, y = row * N2 + b;
    const long long e = ((long long)i3 * N + y) * N + x;
    C w[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) w[q] = from_vec<R>(v[q]);
    if constexpr (CGT) {
      if (r_in != nullptr) {
        // CG direction p = r + beta p, stored back
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          w[q] = mk(g[q].x + bt * w[q].x, g[q].y + bt * w[q].y);
          const_cast<C*>(u)[(q0 + q) * n + e] = w[q];
        }
      }
    }
    fetch(vi + NT);
    if constexpr (std::is_same<R, double>::value) {
      if (kr.root != nullptr) {
        const double s = kr.root[e];
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          const long long at = (q0 + q) * n + e;
          if (kr.tmp != nullptr) {
            w[q] = minus_groups(w[q], kr.tmp + at, 4 * n, kr.groups);
            kr.v[at] = w[q];
            nrm_acc.add(cabs2(w[q]));
          }
          w[q] = cscale(w[q], s);
        }
      }
    }
    if constexpr (!AHEAD) voxel_basis<R>(basis, n, e, lam[x], lam[N + y], a3, alpha, beta, B);
    E* cell = buf + row * PITCH + x;
    if constexpr (NF == 1) {
      C p[3], q[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        p[k] = csub(cmul(B.x[k], w[1]), cmul(B.c[k], w[0]));   // p^ = -c u1a + x u1b
        q[k] = cadd(cmulc(B.x[k], w[2]), cmulc(B.c[k], w[3]));  // q^ = conj(x) u2a + conj(c) u2b
      }
      if (kind != kMediumChiral) swap_axes(p, ax_a, ax_b);
#pragma unroll
      for (int j = 0; j < 3; ++j) put_pair(cell + j * N1 * PITCH, 0, p[j], q[j]);
    } else {
      C o[3];
      if (fsel == 0) {
#pragma unroll
        for (int k = 0; k < 3; ++k) o[k] = csub(cmul(B.x[k], w[1]), cmul(B.c[k], w[0]));
        if (kind != kMediumChiral) swap_axes(o, ax_a, ax_b);
      } else {
#pragma unroll
        for (int k = 0; k < 3; ++k) o[k] = cadd(cmulc(B.x[k], w[0]), cmulc(B.c[k], w[1]));
      }
#pragma unroll
      for (int j = 0; j < 3; ++j) cell[j * N1 * PITCH] = o[j];
    }
  }
  if constexpr (std::is_same<R, double>::value) {
    if (kr.tmp != nullptr) {
      const double part = nrm_acc.template block_total<NT>();
      if (threadIdx.x == 0) kr.nrm_out[i3 * gridDim.x + blockIdx.x] = part;
    }
  }
  __syncthreads();
  stage_strided<false, N1, N2, LINES, NT, PITCH, 1>(buf, tw);  // along x
  __syncthreads();
  stage_group<false, N1, N2, LINES, NT, PITCH, 1>(buf, tw);
  __syncthreads();
  depend_begin();
  // stage A along y over the rows, results to the workspace
#pragma unroll 1
  for (int it = threadIdx.x; it < 3 * N; it += NT) {
    const int j = it / N, x = it % N;
    E r[N1];
#pragma unroll
    for (int k = 0; k < N1; ++k) r[k] = buf[(j * N1 + k) * PITCH + x];
    edft<N1, true>(r);
    E* o = fld + (long long)(j * NF + fsel) * n + ((long long)(x / XL) * n3 + i3) * (N2 * XL) + b * XL + x % XL;
#pragma unroll
    for (int a = 0; a < N1; ++a) {
      if (a > 0) r[a] = etwiddle<true>(r[a], tw[a * b]);
      o[(long long)a * N * n3 * N2] = r[a];
    }
  }
}

// ---------------------------------------------------------------------------
// k_columns: grid (N / X, N1, 3 P)
// ---------------------------------------------------------------------------

// The voxel whose fields a column CTA holds at slot (a, b) of y, slot xs of x
// and slot zs of z (natural index).
template <int N2>
__device__ __forceinline__ int slot_index(int s, int N1) { return s / N2 + N1 * (s % N2); }

// Where a column CTA sits, for the per-voxel steps.
struct ColumnPos {
  int j, a, xs, zs, prob;  // pair, k1 of y, slot of x, slot of z, problem
  int x, z;                // natural indices of xs and zs
  int n1, N1, n3;          // plane edge, its first factor, z length
  __device__ __forceinline__ long long voxel(int b) const { return ((long long)z * n1 + a + N1 * b) * n1 + x; }
};

// The material product of a pair at one voxel:
//   w = 1/Phi (q + i g im p),  f = im (p - i g w),  both times `scale`;
// returns Re(conj(p) f + conj(q) w) for the CG curvature.
template <typename R>
__device__ __forceinline__ R pair_material(R ip, R g, R im, R scale, cplx<R>& p, cplx<R>& q) {
  const R gi = g * im;
  const cplx<R> wc = cscale(mk(q.x - gi * p.y, q.y + gi * p.x), ip);
  const cplx<R> fc = mk(p.x + g * wc.y, p.y - g * wc.x);
  const cplx<R> w = cscale(wc, scale), f = cscale(fc, im * scale);
  const R s = p.x * f.x + p.y * f.y + q.x * w.x + q.y * w.y;
  p = f;
  q = w;
  return s;
}

// The step of the A_r product: load() fetches the material of the NB voxels
// from slot b of y on, ahead of its use; apply() forms the product of the voxel
// at slot b, entry k of the loaded values.
template <typename R>
struct ProductStep {
  static constexpr bool kForward = true;
  MatView<R> m;
  R inv_n;
  long long smat;
  template <int NB>
  struct Vals {
    R ip[NB], g[NB], im[NB];
  };
  template <int NB>
  __device__ __forceinline__ void load(const ColumnPos& c, int b, Vals<NB>& v) const {
    if constexpr (std::is_same<R, float>::value) {
      // [j][a][x][b / 2][z]: {1/Phi, g} of b and b + 1
      const long long at = (((long long)(c.j * c.N1 + c.a) * c.n1 + c.xs) * (NB / 2)) * c.n3 + c.zs;
      const float4* t = m.pmat + c.prob * smat + at;
#pragma unroll
      for (int k = 0; k < NB / 2; ++k) {
        const float4 w = __ldg(t + (long long)k * c.n3);
        v.ip[2 * k] = w.x;
        v.g[2 * k] = w.y;
        v.ip[2 * k + 1] = w.z;
        v.g[2 * k + 1] = w.w;
      }
      if (m.pmu != nullptr) {
        const float2* s = m.pmu + c.prob * smat + at;
#pragma unroll
        for (int k = 0; k < NB / 2; ++k) {
          const float2 w = __ldg(s + (long long)k * c.n3);
          v.im[2 * k] = w.x;
          v.im[2 * k + 1] = w.y;
        }
      } else {
#pragma unroll
        for (int k = 0; k < NB; ++k) v.im[k] = 1.0f;
      }
    } else {
      const int s = pair_axis(m.kind, m.ax_a, m.ax_b, c.j);
      const bool none = m.kind != kMediumChiral && s == c.j;  // the uncoupled component
#pragma unroll
      for (int k = 0; k < NB; ++k) {
        const long long vox = c.voxel(b + k);
        v.ip[k] = m.inv_phi[c.prob * smat + c.j * m.n + vox];
        v.im[k] = m.inv_mu ? m.inv_mu[c.prob * smat + s * m.n + vox] : (R)1;
        v.g[k] = none ? (R)0 : m.gam[c.prob * smat + (m.kind == kMediumChiral ? c.j * m.n : 0) + vox];
      }
    }
  }
  template <int NB>
  __device__ __forceinline__ R apply(const ColumnPos&, int, const Vals<NB>& v, int k, cplx<R>& p, cplx<R>& q) const {
    return pair_material<R>(v.ip[k], v.g[k], v.im[k], inv_n, p, q);
  }
};

template <typename R, int N2, int X, int N3>
constexpr size_t columns_smem() {
  return (size_t)(N3 * (ElemOf<R>::NF * N2 * X + 1) + N3 + N2) * 16;
}

// The plane edge N1 N2 is a run-time value (it only sets strides).
template <typename R, int N2, int X, int XL, int N3, int NT, int MINB, class Step>
__global__ void __launch_bounds__(NT, MINB)
k_columns(typename ElemOf<R>::E* fld, Step step, const cplx<R>* __restrict__ twy, const cplx<R>* __restrict__ twz,
          const int* skip, CGState* st, BatchStrides bs) {
  using C = cplx<R>;
  using E = typename ElemOf<R>::E;
  using S = DepthSplit<R, N3>;
  constexpr int NF = ElemOf<R>::NF, Z1 = S::N1, Z2 = S::N2;
  constexpr int L = N2 * X;
  constexpr int LINES = NF * L;  // line f L + b X + x % X
  constexpr int PITCH = LINES + 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  E* buf = reinterpret_cast<E*>(smem_raw);
  E* tz = buf + N3 * PITCH;
  E* ty = tz + N3;  // w_N^{a b}, b < N2
  const int xt = blockIdx.x, a = blockIdx.y, j = blockIdx.z % 3, prob = blockIdx.z / 3;
  for (int i = threadIdx.x; i < N3; i += NT) tz[i] = tw_entry(twz[i]);
  if (threadIdx.x < N2) ty[threadIdx.x] = tw_entry(twy[a * threadIdx.x]);
  depend_wait();
  if (skip != nullptr && skip[(long long)prob * bs.sskip]) return;
  const int stop = st != nullptr ? st[prob].stop : 0;
  const int N1 = gridDim.y, N = N1 * N2;
  const long long n = (long long)N * N * N3;
  E* tile = fld + prob * bs.sfld + (long long)j * NF * n + ((long long)a * N + xt * X / XL * XL) * (N3 * N2) + xt * X % XL;
  auto gaddr = [&](int l, int z) { return tile + (l / L) * n + z * (N2 * XL) + l % L / X * XL + l % X; };
  if (stop) return;
  auto position = [&](int xi, int zs) {
    return ColumnPos{j,  a, xt * X + xi, zs, prob, slot_index<N2>(xt * X + xi, N1), slot_index<Z2>(zs, Z1), N, N1, N3};
  };
  constexpr int VITEMS = L * N3;
  constexpr bool AHEAD = NF == 2 && kAhead<R>(VITEMS, NT, 2);
  typename Step::template Vals<1> ahead[2];
  if constexpr (AHEAD) {
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int it = threadIdx.x + t * NT;
      if (it < VITEMS) step.template load<1>(position(it / N3 % X, it % N3), it / N3 / X, ahead[t]);
    }
  }
  __syncthreads();  // twiddles
  // inverse stage A along z from the workspace
  {
    constexpr int ITEMS = LINES * Z2;
#pragma unroll 1
    for (int it = threadIdx.x; it < ITEMS; it += NT) {
      const int l = it % LINES, n2 = it / LINES;
      const E* g = gaddr(l, n2);
      E r[Z1];
#pragma unroll
      for (int k = 0; k < Z1; ++k) r[k] = g[k * Z2 * (N2 * XL)];
      edft<Z1, true>(r);
      E* o = buf + n2 * PITCH + l;
#pragma unroll
      for (int k = 0; k < Z1; ++k) o[k * Z2 * PITCH] = (k > 0 && Z2 > 1) ? etwiddle<true>(r[k], tz[n2 * k]) : r[k];
    }
  }
  __syncthreads();
  if constexpr (Z2 > 1) {
    stage_group<false, Z1, Z2, LINES, NT, 1, PITCH>(buf, tz);
    __syncthreads();
  }
  // stage B along y, the material step, stage A' along y
  RedAccFor<R> dot;
  if constexpr (NF == 1) {
    // all in registers: items (x slot, z slot), the z slot fastest across
    // threads (odd pitch)
    constexpr int ITEMS = X * N3;
#pragma unroll 1
    for (int it = threadIdx.x; it < ITEMS; it += NT) {
      const int xi = it / N3, zs = it % N3;
      const ColumnPos pos = position(xi, zs);
      typename Step::template Vals<N2> mv;
      step.template load<N2>(pos, 0, mv);
      E* cell = buf + zs * PITCH + xi;
      E v[N2];
#pragma unroll
      for (int k = 0; k < N2; ++k) v[k] = cell[k * X];
      edft<N2, true>(v);
      R sacc = (R)0;
#pragma unroll
      for (int k = 0; k < N2; ++k) {
        C p, q;
        get_pair(&v[k], 0, p, q);
        const R s = step.template apply<N2>(pos, k, mv, k, p, q);
        if (st != nullptr) sacc = sacc + s;
        put_pair(&v[k], 0, p, q);
      }
      if (st != nullptr) dot.add(static_cast<typename RedAccFor<R>::value_type>(sacc));
      edft<N2, false>(v);
#pragma unroll
      for (int k = 0; k < N2; ++k) cell[k * X] = k > 0 ? etwiddle<false>(v[k], ty[k]) : v[k];
    }
  } else {
    // one step after the other over the tile, each with as many items as it
    // has: these types are bound by their arithmetic, and a small tile leaves
    // most lanes of a warp idle when one item does all three (8^3 complex128,
    // whose 48 CTAs have 8 such items each)
    constexpr int DITEMS = NF * X * N3;
#pragma unroll 1
    for (int it = threadIdx.x; it < DITEMS; it += NT) {
      E* cell = buf + (it % N3) * PITCH + it / N3 % X + it / (N3 * X) * L;
      E v[N2];
#pragma unroll
      for (int k = 0; k < N2; ++k) v[k] = cell[k * X];
      edft<N2, true>(v);
#pragma unroll
      for (int k = 0; k < N2; ++k) cell[k * X] = v[k];
    }
    __syncthreads();
    auto voxel_step = [&](int it, typename Step::template Vals<1>& mv) {
      const int zs = it % N3, l = it / N3;
      const ColumnPos pos = position(l % X, zs);
      if constexpr (!AHEAD) step.template load<1>(pos, l / X, mv);
      E* cell = buf + zs * PITCH + l;
      C p = cell[0], q = cell[L];
      const R s = step.template apply<1>(pos, l / X, mv, 0, p, q);
      if (st != nullptr) dot.add(static_cast<typename RedAccFor<R>::value_type>(s));
      cell[0] = p;
      cell[L] = q;
    };
    if constexpr (AHEAD) {
#pragma unroll
      for (int t = 0; t < 2; ++t)
        if (threadIdx.x + t * NT < VITEMS) voxel_step(threadIdx.x + t * NT, ahead[t]);
    } else {
#pragma unroll 1
      for (int it = threadIdx.x; it < VITEMS; it += NT) {
        typename Step::template Vals<1> mv;
        voxel_step(it, mv);
      }
    }
    if constexpr (Step::kForward) {
      __syncthreads();
#pragma unroll 1
      for (int it = threadIdx.x; it < DITEMS; it += NT) {
        E* cell = buf + (it % N3) * PITCH + it / N3 % X + it / (N3 * X) * L;
        E v[N2];
#pragma unroll
        for (int k = 0; k < N2; ++k) v[k] = cell[k * X];
        edft<N2, false>(v);
#pragma unroll
        for (int k = 0; k < N2; ++k) cell[k * X] = k > 0 ? etwiddle<false>(v[k], ty[k]) : v[k];
      }
    }
  }
  if constexpr (Step::kForward) {
    if (st != nullptr) {
      // this CTA's share of p^* A_r p (Parseval: from the real-space fields; the
      // DFTs carry the factor n that the step removes)
      const auto tot = dot.template block_total<NT>();
      if (threadIdx.x == 0)
        reinterpret_cast<typename RedAccFor<R>::partial*>(st[prob].part_a)[(j * gridDim.y + a) * gridDim.x + xt] = tot;
      if (NT == 32) __syncthreads();  // (otherwise block_total's barriers order the tile's writes)
    } else {
      __syncthreads();
    }
    if constexpr (Z2 > 1) {
      stage_group<true, Z1, Z2, LINES, NT, 1, PITCH>(buf, tz);
      __syncthreads();
    }
    depend_begin();
    // forward stage B' along z, results to the workspace
    constexpr int ITEMS = LINES * Z2;
#pragma unroll 1
    for (int it = threadIdx.x; it < ITEMS; it += NT) {
      const int l = it % LINES, n2 = it / LINES;
      const E* s = buf + n2 * PITCH + l;
      E r[Z1];
#pragma unroll
      for (int k = 0; k < Z1; ++k) r[k] = s[k * Z2 * PITCH];
      edft<Z1, false>(r);
      E* g = gaddr(l, n2);
#pragma unroll
      for (int k = 0; k < Z1; ++k) g[k * Z2 * (N2 * XL)] = r[k];
    }
  }
}

// ---------------------------------------------------------------------------
// k_rows_out: grid (N2 NF, n3, P), as k_rows_in
// ---------------------------------------------------------------------------
template <typename R, int N, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB)
k_rows_out(const typename ElemOf<R>::E* fld, vecc<R>* Au, const cplx<R>* __restrict__ lam,
           const cplx<R>* __restrict__ twx, R alpha, R beta, int kind, int ax_a, int ax_b, const int* skip,
           const cplx<R>* __restrict__ basis, BatchStrides bs, CgFuse<R> cg, typename KrylovOf<R>::type kr) {
  using C = cplx<R>;
  using E = typename ElemOf<R>::E;
  using S = PlaneSplit<R, N>;
  constexpr int NF = ElemOf<R>::NF, N1 = S::N1, N2 = S::N2, X = S::X, XL = S::XL;
  constexpr int PITCH = N + 1;
  constexpr int LINES = 3 * N1;
  constexpr int NV = N1 * N;
  static_assert(3 * N1 * (N / X) <= kMaxPartials, "one partial of p^* A p per CTA of k_columns");
  static_assert(N2 * NF * 128 <= kMaxPartials, "one partial of r^* r per CTA of this kernel, up to 128 of z");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  E* buf = reinterpret_cast<E*>(smem_raw);
  E* tw = buf + LINES * PITCH;
  const int b = blockIdx.x % N2, fsel = blockIdx.x / N2, i3 = blockIdx.y, prob = blockIdx.z, n3 = gridDim.y;
  for (int i = threadIdx.x; i < N; i += NT) tw[i] = tw_entry(twx[i]);
  depend_wait();
  if (skip != nullptr && skip[(long long)prob * bs.sskip]) return;
  constexpr bool CGT = !std::is_same<R, df>::value;  // (the double-single product never runs CG)
  CGState* st = (CGT && cg.st != nullptr) ? cg.st + prob : nullptr;
  const bool first = blockIdx.x == 0 && i3 == 0 && threadIdx.x == 0;
  const long long n = (long long)N * N * n3;
  constexpr int NQ = 4 / NF;  // quarters of the result that this CTA forms, from q0 on
  const int q0 = NF == 1 ? 0 : 2 * fsel;
  int stop = 0;
  RedAccFor<R> pap_acc;
  if constexpr (CGT) {
    if (st != nullptr) {
      stop = st->stop;
      if (stop_first<R, N>(n3) && stop) {
        if (first) st->halt = 1;
        return;
      }
      cg.x += prob * bs.su + q0 * n;
      cg.r += prob * bs.su + q0 * n;
      cg.p += prob * bs.su + q0 * n;
      const auto* pa = reinterpret_cast<const typename RedAccFor<R>::partial*>(st->part_a);
#pragma unroll 2
      for (int i = threadIdx.x; i < 3 * N1 * (N / X); i += NT) pap_acc.add_partial(pa[i]);
    }
  }
  double inv_h = 1.0;
  if constexpr (std::is_same<R, double>::value) {
    if (kr.nnrm > 0) {
      RedAcc<double> acc;
      for (int i = threadIdx.x; i < kr.nnrm; i += NT) acc.add(kr.nrm[i]);
      const double ss = acc.template block_total<NT>();
      inv_h = ss > 0.0 ? ::rsqrt(ss) : 0.0;  // (a zero vector stays zero)
    }
  }
  fld += prob * bs.sfld;
  Au += prob * bs.su;
  lam += (long long)prob * bs.slam;
  if (basis != nullptr) basis += prob * bs.sbasis;
  // one voxel per thread: the operands of the last step (see kAhead)
  constexpr bool AHEAD = kAhead<R>(NV, NT);
  Basis<R> B;
  vecc<R> pv[NQ], xv[NQ], rv[NQ];
  if constexpr (AHEAD) {
    if (threadIdx.x < NV) {
      const int x = threadIdx.x % N, y = b + N2 * (threadIdx.x / N);
      const long long e = ((long long)i3 * N + y) * N + x;
      if constexpr (CGT) {
        if (st != nullptr) {
#pragma unroll
          for (int q = 0; q < NQ; ++q) {
            pv[q] = cg.p[e + q * n];
            rv[q] = cg.r[e + q * n];
            xv[q] = cg.x[e + q * n];
          }
        }
      }
      voxel_basis<R>(basis, n, e, lam[x], lam[N + y], lam[2 * N + i3], alpha, beta, B);
    }
  }
  // stage B' along y from the workspace: row k of the CTA is y = b + N2 k
#pragma unroll 1
  for (int it = threadIdx.x; it < 3 * N; it += NT) {
    const int j = it / N, x = it % N;
    const E* g = fld + (long long)(j * NF + fsel) * n + ((long long)(x / XL) * n3 + i3) * (N2 * XL) + b * XL + x % XL;
    E r[N1];
#pragma unroll
    for (int a = 0; a < N1; ++a) r[a] = g[(long long)a * N * n3 * N2];
    edft<N1, false>(r);
#pragma unroll
    for (int k = 0; k < N1; ++k) buf[(j * N1 + k) * PITCH + x] = r[k];
  }
  if (stop) {
    if (first) st->halt = 1;
    return;
  }
  __syncthreads();
  stage_group<true, N1, N2, LINES, NT, PITCH, 1>(buf, tw);  // along x
  __syncthreads();
  stage_strided<true, N1, N2, LINES, NT, PITCH, 1>(buf, tw);
  R cg_al = (R)0;
  bool ok = false;
  if constexpr (CGT) {
    if (st != nullptr) {
      using P = typename RedAccFor<R>::partial;
      const P pAp = pap_acc.template block_total<NT>();
      const P rr = *reinterpret_cast<const P*>(&st->rr_now);
      cg_al = (R)scalar_ratio(rr, pAp);
      ok = scalar_positive(pAp) && cg_al == cg_al;  // also catches NaN
      if (first) {
        if (ok) {
          st->it += 1;
          *reinterpret_cast<P*>(&st->rr_last) = rr;
        } else {
          st->broken = st->halt = 1;  // breakdown: x, r left untouched
        }
      }
      if (!ok) return;
    }
  }
  __syncthreads();
  depend_begin();
  RedAccFor<R> rr_acc;
  const C a3 = lam[2 * N + i3];
#pragma unroll 1
  for (int vi = threadIdx.x; vi < NV; vi += NT) {
    const int row = vi / N, x = vi % N, y = b + N2 * row;
    const long long e = ((long long)i3 * N + y) * N + x;
    if constexpr (CGT && !AHEAD) {
      if (ok) {
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          pv[q] = cg.p[e + q * n];
          rv[q] = cg.r[e + q * n];
          xv[q] = cg.x[e + q * n];
        }
      }
    }
    if constexpr (!AHEAD) voxel_basis<R>(basis, n, e, lam[x], lam[N + y], a3, alpha, beta, B);
    // P_r^* f = [-sum conj(c) f ; sum conj(x) f],  Q_r^* w = [sum x w ; sum c w]
    const E* cell = buf + row * PITCH + x;
    C o[NQ];
    C f[3], w[3];
    if constexpr (NF == 1) {
#pragma unroll
      for (int j = 0; j < 3; ++j) get_pair(cell + j * N1 * PITCH, 0, f[j], w[j]);
    } else {
#pragma unroll
      for (int j = 0; j < 3; ++j) f[j] = w[j] = cell[j * N1 * PITCH];
    }
    if (NF == 1 || fsel == 0) {
      if (kind != kMediumChiral) swap_axes(f, ax_a, ax_b);
      o[0] = cneg(cadd(cadd(cmulc(B.c[0], f[0]), cmulc(B.c[1], f[1])), cmulc(B.c[2], f[2])));
      o[1] = cadd(cadd(cmulc(B.x[0], f[0]), cmulc(B.x[1], f[1])), cmulc(B.x[2], f[2]));
    }
    if (NF == 1 || fsel == 1) {
      o[NQ - 2] = cadd(cadd(cmul(B.x[0], w[0]), cmul(B.x[1], w[1])), cmul(B.x[2], w[2]));
      o[NQ - 1] = cadd(cadd(cmul(B.c[0], w[0]), cmul(B.c[1], w[1])), cmul(B.c[2], w[2]));
    }
    if (ok) {
      if constexpr (CGT) {
        R s = (R)0;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          xv[q] = mk(xv[q].x + cg_al * pv[q].x, xv[q].y + cg_al * pv[q].y);
          rv[q] = mk(rv[q].x - cg_al * o[q].x, rv[q].y - cg_al * o[q].y);
          cg.x[e + q * n] = xv[q];
          cg.r[e + q * n] = rv[q];
          s += rv[q].x * rv[q].x + rv[q].y * rv[q].y;
        }
        rr_acc.add(s);
      }
      continue;
    }
    if constexpr (std::is_same<R, double>::value) {
      if (kr.root != nullptr) {
        const double s = kr.root[e] * inv_h;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          const long long at = ((q0 + q + 2) & 3) * n + e;
          double2 out = cscale(o[q], s);
          if (kr.v != nullptr) {
            double2 vv = kr.v[at];
            if (kr.nnrm > 0) {
              vv = cscale(vv, inv_h);
              kr.v[at] = vv;
            }
            out = csub(out, cmul(kr.sigma, vv));
          }
          Au[at] = out;
        }
        continue;
      }
    }
#pragma unroll
    for (int q = 0; q < NQ; ++q) Au[(q0 + q) * n + e] = to_vec<R>(o[q]);
  }
  if constexpr (CGT) {
    if (st != nullptr) {
      const auto part = rr_acc.template block_total<NT>();
      if (threadIdx.x == 0) reinterpret_cast<typename RedAccFor<R>::partial*>(st->part_b)[i3 * gridDim.x + blockIdx.x] = part;
    }
  }
}

}  // namespace nfs
