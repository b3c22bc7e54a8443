// Vector kernels of the CG and Lanczos loops (Section 4.2: CG on A_r u = b;
// invert Lanczos on (B_r, A_r)), batched over the P problems of one context:
// problem p's vectors sit at base + p * N (N = 4n), and the problem index comes
// from a grid dimension, so a launch serves every problem at once.
//
// Reductions are deterministic: a grid of blocks per problem fixed by the
// vector length and the problem count (at most kRedBlocks) writes one
// partial per block, and a one-block kernel, the host or (in CG) every block of
// the next kernel sums the partials in a fixed order.
#pragma once
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "cg_state.cuh"
#include "nfs_complex.cuh"

namespace nfs {

// Blocks per problem of the reductions over P problems' vectors of length N.
// Never more blocks than the vector has threads' worth of elements (empty
// blocks add exact zeros: a single problem's sums are the same at any larger
// count); for batches, fewer, with at least 32 elements per thread, as long
// as all problems together still have kRedBlocks blocks.  Each block ends in
// FP64 block sums, which GB300 retires at about one warp instruction per 17
// SM cycles: a full grid per problem over the short vectors of a batch of
// small grids made those epilogues, not the data, the cost of a reduction.
inline int red_blocks(long long N, int P) {
  long long nb = std::min<long long>(kRedBlocks, (N + kRedThreads - 1) / kRedThreads);
  if (P > 1) {
    const long long per32 = (N + (long long)kRedThreads * 32 - 1) / ((long long)kRedThreads * 32);
    nb = std::min(nb, std::max<long long>(per32, (kRedBlocks + P - 1) / P));
  }
  return (int)std::max<long long>(1, nb);
}

// Blocks per problem and pair of k_exact_dots over m vectors: with many vectors
// half of them, for fewer FP64 ends of blocks.  A thread's FP32 sums are then as
// long as those of one element at a time over all the blocks, since it keeps two
// of each.  52 vectors on one GB300, with k_dots_finish, all blocks and half of
// them: 96^3 636 and 594 us, 64^3 271 and 217, 32^3 137 and 82, 16 problems of
// 32^3 428 and 383.
inline int exact_dots_blocks(long long N, int P, int m) {
  const int nb = red_blocks(N, P);
  return m < 16 ? nb : (nb + 1) / 2;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum over the block; the result is valid in thread 0 (and warp 0) only.
template <int NT>
__device__ __forceinline__ double block_sum(double v) {
  __shared__ double sh[NT / 32];
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  double r = 0.0;
  if (warp == 0) {
    r = lane < NT / 32 ? sh[lane] : 0.0;
    r = warp_sum(r);
  }
  __syncthreads();
  return r;
}

// part[p * pstride + b] = block b's share of Re(conj(x_p) y_p); grid (blocks, P).
__global__ void __launch_bounds__(kRedThreads)
k_dot_re(const double2* __restrict__ x, const double2* __restrict__ y, long long N, double* __restrict__ part,
         long long pstride) {
  const int p = blockIdx.y;
  x += (long long)p * N;
  y += (long long)p * N;
  double acc = 0.0;
  for (long long i = (long long)blockIdx.x * kRedThreads + threadIdx.x; i < N; i += (long long)gridDim.x * kRedThreads) {
    const double2 a = x[i], b = y[i];
    acc += a.x * b.x + a.y * b.y;
  }
  const double s = block_sum<kRedThreads>(acc);
  if (threadIdx.x == 0) part[(long long)p * pstride + blockIdx.x] = s;
}

// Partials of |Ay - omega By|^2 and |y|^2 for one eigenpair (the residual
// of the HHPD-NFGEP, B_r y = omega^{-1} A_r y scaled by omega): block b writes
// part[2b], part[2b + 1]; grid kRedBlocks.
__global__ void __launch_bounds__(kRedThreads)
k_residual_parts(const double2* __restrict__ Ay, const double2* __restrict__ By, const double2* __restrict__ y,
                 double omega, long long N, double* __restrict__ part) {
  double rr = 0.0, yy = 0.0;
  for (long long i = (long long)blockIdx.x * kRedThreads + threadIdx.x; i < N; i += (long long)gridDim.x * kRedThreads) {
    const double2 a = Ay[i], b = By[i], v = y[i];
    const double dx = a.x - omega * b.x, dy = a.y - omega * b.y;
    rr += dx * dx + dy * dy;
    yy += v.x * v.x + v.y * v.y;
  }
  rr = block_sum<kRedThreads>(rr);
  yy = block_sum<kRedThreads>(yy);
  if (threadIdx.x == 0) {
    part[2 * blockIdx.x] = rr;
    part[2 * blockIdx.x + 1] = yy;
  }
}

// CG start, one block per problem: r^* r = the sum of the nred partials in
// part_a (k_dot_re, k_inner_start, k_solve_start) becomes the only partial of the
// nb in part_b; tol2 is the threshold, or (relative) its ratio to r^* r.  An
// infinite one, or an r^* r that is not positive, means nothing to solve.
template <typename R>
__global__ void __launch_bounds__(kRedThreads)
k_cg_init(CGState* st, const double* __restrict__ tol2, bool relative, int maxit, int nred, int nb) {
  using P = typename RedAccFor<R>::partial;
  st += blockIdx.x;
  const P rr = sum_partials_all<R, kRedThreads>(st->part_a, nred);
  P* pb = reinterpret_cast<P*>(st->part_b);
  for (int i = threadIdx.x; i < nb; i += kRedThreads) {
    P v = rr;
    if (i > 0) scalar_from(0.0, v);
    pb[i] = v;
  }
  if (threadIdx.x == 0) {
    const double r2 = scalar_double(rr);
    double tol = tol2[blockIdx.x];
    if (relative) tol = r2 > 0.0 && tol < (double)INFINITY ? tol * r2 : (double)INFINITY;
    st->rr = st->rr0 = r2;
    st->it = 0;
    st->maxit = maxit;
    st->done = st->status = 0;
    st->stop = st->halt = st->broken = 0;
    scalar_from((double)INFINITY, *reinterpret_cast<P*>(&st->rr_last));
    scalar_from(tol, *reinterpret_cast<P*>(&st->tol2));
  }
}

// End of a chunk of CG steps, one block per problem: the state that the host
// reads, from the nb partials of r^* r.  Where the steps have stopped, r^* r is
// the sum that k_rows_in stopped them by: its blocks add the partials up in
// another order, which may round to the other side of the threshold, and a state
// that steps no more has to be done.
template <typename R>
__global__ void __launch_bounds__(kRedThreads) k_cg_check(CGState* st, int nb) {
  using P = typename RedAccFor<R>::partial;
  st += blockIdx.x;
  const P sum = sum_partials_all<R, kRedThreads>(st->part_b, nb);
  if (threadIdx.x == 0) {
    const P rr = st->halt ? *reinterpret_cast<const P*>(&st->rr_now) : sum;
    st->rr = scalar_double(rr);
    const bool bad = st->broken || scalar_nan(rr);
    const bool conv = scalar_le(rr, *reinterpret_cast<const P*>(&st->tol2));
    st->status = bad ? -7 : conv ? 0 : st->it >= st->maxit ? -6 : 0;
    st->done = bad || conv || st->it >= st->maxit;
  }
}

// ---------------------------------------------------------------------------
// Elementwise helpers over all P problems (flat index i, problem i / N)
// ---------------------------------------------------------------------------

template <typename C>
__global__ void k_sub(const C* __restrict__ a, const C* __restrict__ b, C* __restrict__ y, long long total) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x)
    y[i] = csub(a[i], b[i]);
}

// *mark = 1 if an entry of x is not zero (a NaN is not)
__global__ void k_mark_nonzero(const double2* __restrict__ x, long long total, int* mark) {
  bool any = false;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const double2 v = x[i];
    any = any || !(v.x == 0.0) || !(v.y == 0.0);
  }
  if (any) *mark = 1;
}

// Refinement residual per problem p (skip64, skip32: the masks of the two
// products just launched): r_p = b_p - Ap64_p where the double-single product ran
// (!skip64[p]), else r_p -= s_p Ap32_p where the complex64 product of the
// correction ran (!skip32[p]), else r_p is left.  Grid-stride over P x N.
__global__ void k_refine_residual(double2* __restrict__ r, const double2* __restrict__ b,
                                  const double2* __restrict__ Ap64, const float2* __restrict__ Ap32,
                                  const double* __restrict__ s, const int* __restrict__ skip64,
                                  const int* __restrict__ skip32, long long N, long long total) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const long long p = i / N;
    if (!skip64[p]) {
      r[i] = csub(b[i], Ap64[i]);
    } else if (!skip32[p]) {
      const float2 a = Ap32[i];
      const double f = s[p];
      double2 ri = r[i];
      ri.x -= f * (double)a.x;
      ri.y -= f * (double)a.y;
      r[i] = ri;
    }
  }
}

// Start of an inner solve: r32 = s[problem] r64 rounded to complex64, zero iterate
// and direction, and the partials of r32^* r32 (part_a; grid (blocks, P)).  One
// kernel instead of the conversion, two memsets and a dot product: 30 instead of
// 66 us at 96^3, bound by the FP64 pipe (two products and two conversions per
// element).
__global__ void __launch_bounds__(kRedThreads)
k_inner_start(const double2* __restrict__ r64, const double* __restrict__ s, float2* __restrict__ r32,
              float2* __restrict__ x32, float2* __restrict__ p32, long long N, CGState* st) {
  const int p = blockIdx.y;
  const double f = s[p];
  const double2* a = r64 + (long long)p * N;
  float4* r = reinterpret_cast<float4*>(r32 + (long long)p * N);
  float4* x = reinterpret_cast<float4*>(x32 + (long long)p * N);
  float4* d = reinterpret_cast<float4*>(p32 + (long long)p * N);
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  RedAcc<float> acc;
  for (long long i = (long long)blockIdx.x * kRedThreads + threadIdx.x; i < N / 2; i += (long long)gridDim.x * kRedThreads) {
    const double2 v0 = a[2 * i], v1 = a[2 * i + 1];
    const float4 o = make_float4((float)(v0.x * f), (float)(v0.y * f), (float)(v1.x * f), (float)(v1.y * f));
    r[i] = o;
    x[i] = zero;
    d[i] = zero;
    acc.add(o.x * o.x + o.y * o.y);  // (one sum in FP32 for both elements would lose the smaller's low bits)
    acc.add(o.z * o.z + o.w * o.w);
  }
  const float2 t = acc.block_total<kRedThreads>();
  if (threadIdx.x == 0) reinterpret_cast<float2*>(st[p].part_a)[blockIdx.x] = t;
}

// Likewise of a complex128 solve from x = 0: r = b.
__global__ void __launch_bounds__(kRedThreads)
k_solve_start(const double2* __restrict__ b, double2* __restrict__ r, double2* __restrict__ x, double2* __restrict__ d,
              long long N, CGState* st) {
  const long long off = (long long)blockIdx.y * N;
  const double2 zero = make_double2(0.0, 0.0);
  RedAcc<double> acc;
  for (long long i = (long long)blockIdx.x * kRedThreads + threadIdx.x; i < N; i += (long long)gridDim.x * kRedThreads) {
    const double2 v = b[off + i];
    r[off + i] = v;
    x[off + i] = zero;
    d[off + i] = zero;
    acc.add(v.x * v.x + v.y * v.y);
  }
  const double t = acc.block_total<kRedThreads>();
  if (threadIdx.x == 0) st[blockIdx.y].part_a[blockIdx.x] = t;
}

// x += s[problem] * complex128(d)
__global__ void k_axpy_promote(double2* __restrict__ x, const double* __restrict__ s, const float2* __restrict__ d,
                               long long N, long long total) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const float2 v = d[i];
    const double f = s[i / N];
    double2 xi = x[i];
    xi.x += f * (double)v.x;
    xi.y += f * (double)v.y;
    x[i] = xi;
  }
}

// B_r v = i [Sigma^{-1} v2 ; -Sigma^{-1} v1], Sigma_r = diag(sqrt(Lq), sqrt(Lq))
// (eq. NFSEP_spd_1).  lam holds Lambda_1 | Lambda_2 | Lambda_3 per problem
// (stride n1 + n2 + n3); v and out hold P vectors of 4n.
__global__ void k_apply_Br(const double2* __restrict__ v, double2* __restrict__ out, const double2* __restrict__ lam,
                           int n1, int n2, int n3, int P, long long vstride = -1) {
  const long long n = (long long)n1 * n2 * n3;
  const int nl = n1 + n2 + n3;
  for (long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x; g < n * P; g += (long long)gridDim.x * blockDim.x) {
    const long long p = g / n, e = g % n;
    const int i1 = (int)(e % n1);
    const int i2 = (int)((e / n1) % n2);
    const int i3 = (int)(e / ((long long)n1 * n2));
    const double2* L = lam + p * nl;
    const double lq = cabs2(L[i1]) + cabs2(L[n1 + i2]) + cabs2(L[n1 + n2 + i3]);
    const double is = 1.0 / sqrt(lq);
    const double2* vp = v + p * (vstride >= 0 ? vstride : 4 * n);  // problem p's input (e.g. a basis column)
    double2* op = out + p * 4 * n;
    const double2 v1a = vp[e], v1b = vp[n + e], v2a = vp[2 * n + e], v2b = vp[3 * n + e];
    op[e] = cmul_i(cscale(v2a, is));
    op[n + e] = cmul_i(cscale(v2b, is));
    op[2 * n + e] = cmul_mi(cscale(v1a, is));
    op[3 * n + e] = cmul_mi(cscale(v1b, is));
  }
}

// Counter-based uniform numbers in [-1, 1) (splitmix64 finaliser of the
// element index and seed): the Lanczos starting vectors.
__device__ __forceinline__ double u01_hash(unsigned long long x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  x ^= x >> 31;
  return (double)(x >> 11) * (1.0 / 9007199254740992.0) * 2.0 - 1.0;
}

// Problem p's starting vector at v + p * vstride (N entries).
__global__ void k_random_fill(double2* __restrict__ v, long long N, long long vstride, int P, unsigned long long seed) {
  for (long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x; g < N * P; g += (long long)gridDim.x * blockDim.x) {
    const long long p = g / N, i = g % N;
    const unsigned long long k = (unsigned long long)i * 2ull + seed * 0x632BE59BD9B4E019ull;
    v[p * vstride + i] = make_double2(u01_hash(k), u01_hash(k + 1));
  }
}

// ---------------------------------------------------------------------------
// Lanczos.  Problem p's basis: vector j at V + p * vstride + j * N (complex128),
// its new vector w at w + p * N.  Coefficients per problem at c + p * m * 2.
// ---------------------------------------------------------------------------

// part[((p * gridDim.x + b) * m + j) * 2 + {0,1}] = block b's share of
// conj(V_pj)^T w_p, j < m; grid (blocks, P).
template <int NT>
__global__ void __launch_bounds__(NT)
k_multi_dot(const double2* __restrict__ V, long long vstride, int m, const double2* __restrict__ w, long long N,
            double* __restrict__ part, const int* __restrict__ active) {
  constexpr int EPT = 4;  // elements of w per thread and pass
  const int p = blockIdx.y;
  if (active && !active[p]) return;
  V += (long long)p * vstride;
  w += (long long)p * N;
  double* pp = part + ((long long)p * gridDim.x + blockIdx.x) * m * 2;
  for (int j0 = 0; j0 < m; ++j0) {
    double re = 0.0, im = 0.0;
    for (long long base = (long long)blockIdx.x * NT * EPT; base < N; base += (long long)gridDim.x * NT * EPT) {
#pragma unroll
      for (int t = 0; t < EPT; ++t) {
        const long long i = base + (long long)t * NT + threadIdx.x;
        if (i < N) {
          const double2 a = V[(long long)j0 * N + i], b = w[i];
          re += a.x * b.x + a.y * b.y;
          im += a.x * b.y - a.y * b.x;
        }
      }
    }
    re = block_sum<NT>(re);
    im = block_sum<NT>(im);
    if (threadIdx.x == 0) {
      pp[j0 * 2 + 0] = re;
      pp[j0 * 2 + 1] = im;
    }
  }
}

// out[(p * m + j) * 2 + {0,1}] = sum over nb blocks; grid (m, P)
__global__ void __launch_bounds__(kRedThreads)
k_multi_dot_finish(const double* __restrict__ part, int m, int nb, double* __restrict__ out,
                   const int* __restrict__ active) {
  const int j = blockIdx.x, p = blockIdx.y;
  if (active && !active[p]) return;
  double re = 0.0, im = 0.0;
  for (int b = threadIdx.x; b < nb; b += kRedThreads) {
    re += part[(((long long)p * nb + b) * m + j) * 2 + 0];
    im += part[(((long long)p * nb + b) * m + j) * 2 + 1];
  }
  re = block_sum<kRedThreads>(re);
  im = block_sum<kRedThreads>(im);
  if (threadIdx.x == 0) {
    out[((long long)p * m + j) * 2] = re;
    out[((long long)p * m + j) * 2 + 1] = im;
  }
}

// w_p -= sum_j c_pj V_pj ; Mw_p -= sum_j c_pj MV_pj; grid (blocks, P).
__global__ void k_multi_axpy(double2* __restrict__ w, double2* __restrict__ Mw, const double2* __restrict__ V,
                             const double2* __restrict__ MV, long long vstride, const double* __restrict__ c, int m,
                             long long N, const int* __restrict__ active) {
  const int p = blockIdx.y;
  if (active && !active[p]) return;
  w += (long long)p * N;
  Mw += (long long)p * N;
  V += (long long)p * vstride;
  MV += (long long)p * vstride;
  c += (long long)p * m * 2;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
    double2 a = w[i], b = Mw[i];
    for (int j = 0; j < m; ++j) {
      const double2 cj = make_double2(c[2 * j], c[2 * j + 1]);
      const double2 v = V[(long long)j * N + i], mv = MV[(long long)j * N + i];
      a = csub(a, cmul(cj, v));
      b = csub(b, cmul(cj, mv));
    }
    w[i] = a;
    Mw[i] = b;
  }
}

// Re-orthogonalisation through the shadows: w_p -= sum_j d_pj V32_pj and
// Mw_p -= sum_j d_pj MV32_pj for j < m, with d (layout of k_dots_finish, on the
// device) exact A_r inner products.  It runs only when the loss of
// orthogonality is small (|d| ~ 1e-8 of |w|), so the update is formed in FP32
// arithmetic from the FP32 shadows: its error is ~1e-8 * 6e-8 of |w|.
// Grid (blocks, P); problems with a zero flag are skipped.
__global__ void k_shadow_axpy(double2* __restrict__ w, double2* __restrict__ Mw, const float2* __restrict__ V32,
                              const float2* __restrict__ MV32, long long vstride, const double* __restrict__ d, int m,
                              long long N, const int* __restrict__ active) {
  const int p = blockIdx.y;
  if (active && !active[p]) return;
  w += (long long)p * N;
  Mw += (long long)p * N;
  V32 += (long long)p * vstride;
  MV32 += (long long)p * vstride;
  d += (long long)p * m * 2;
  // the coefficients as floats, converted once per block (double-precision
  // conversions run at the FP64 rate)
  extern __shared__ float2 sd[];
  for (int j = threadIdx.x; j < m; j += blockDim.x) sd[j] = make_float2((float)d[2 * j], (float)d[2 * j + 1]);
  __syncthreads();
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x) {
    float2 a = make_float2(0.f, 0.f), b = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int j = 0; j < m; ++j) {
      const float2 cj = sd[j];
      const float2 v = V32[(long long)j * N + i], mv = MV32[(long long)j * N + i];
      a = cadd(a, cmul(cj, v));
      b = cadd(b, cmul(cj, mv));
    }
    double2 wi = w[i], mi = Mw[i];
    wi.x -= (double)a.x;
    wi.y -= (double)a.y;
    mi.x -= (double)b.x;
    mi.y -= (double)b.y;
    w[i] = wi;
    Mw[i] = mi;
  }
}

// ---------------------------------------------------------------------------
// Exact A_r inner products on the FP32 units.  A_r is ill-conditioned
// (|A v| |w| >> |v|_A |w|_A), so single-precision inner products carry an
// absolute error near 1e-8 |w|_A: the level of orthogonality Lanczos needs to
// keep.  Here every operand is split into two floats (hi + lo, the lo part
// holding the FP64 remainder), the hi x hi products are formed exactly
// (TwoProduct by FMA) and summed exactly (TwoSum, Knuth), the small hi x lo
// and lo x hi terms and the rounding errors go to an ordinary FP32 sum, and
// the block sums are FP64: about 1e-14 of sum |terms|.  Double-precision
// arithmetic, scarce on this GPU, is used only for the per-block totals.
// ---------------------------------------------------------------------------

// Error-free transformations (TwoProduct by FMA; TwoSum, Knuth) on (real,
// imaginary) pairs, both halves in one packed f32x2 instruction:
// p + e = a * b and s + e = a + b exactly, per half.
__device__ __forceinline__ void two_prod_x2(float2 a, float2 b, float2& p, float2& e) {
  p = mul_x2(a, b);
  e = fma_x2(a, b, make_float2(-p.x, -p.y));
}
__device__ __forceinline__ void two_sum_x2(float2 a, float2 b, float2& s, float2& e) {
  s = add_x2(a, b);
  const float2 bb = sub_x2(s, a);
  e = add_x2(sub_x2(a, sub_x2(s, bb)), sub_x2(b, bb));
}
struct DSAccX2 {
  float2 hi = make_float2(0.f, 0.f), lo = make_float2(0.f, 0.f);
  __device__ __forceinline__ void add(float2 x) {
    float2 e;
    two_sum_x2(hi, x, hi, e);
    lo = add_x2(lo, e);
  }
};

__device__ __forceinline__ float2 split_lo(double2 v, float2 hi) {
  return make_float2((float)(v.x - (double)hi.x), (float)(v.y - (double)hi.y));
}

// In-place basis rotation V_p[:, 0:k] = V_p[:, 0:m] Y_p (Y_p real, m x k,
// column-major), in double-single arithmetic on the FP32 units: Y is given
// as float pairs Yhl[p m k + col m + j] = (hi, lo) with hi + lo = Y to ~1e-15,
// each block stages TE elements of all m vectors in shared memory split the
// same way, and every product hi x hi is formed exactly (TwoProduct) and
// summed exactly (TwoSum) with the cross terms and rounding errors in an
// ordinary FP32 sum: ~1e-14 of sum |terms|, at a small fraction of the cost
// of FP64 arithmetic (m k FP64 FMAs per element otherwise).  A thread forms
// CPT columns of one element.  Grid (blocks, P); problems with a zero flag
// are skipped.
template <int TE, int CPT>
__global__ void __launch_bounds__(256)
k_rotate_basis(double2* __restrict__ V, long long vstride, int m, const float2* __restrict__ Yhl, int k, long long N,
               const int* __restrict__ active) {
  const int p = blockIdx.y;
  if (active && !active[p]) return;
  V += (long long)p * vstride;
  Yhl += (long long)p * m * k;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float4* tile = reinterpret_cast<float4*>(smem_raw);  // [m][TE]: (re hi, im hi, re lo, im lo)
  const int groups = (k + CPT - 1) / CPT;
  for (long long base = (long long)blockIdx.x * TE; base < N; base += (long long)gridDim.x * TE) {
    for (int idx = threadIdx.x; idx < m * TE; idx += blockDim.x) {
      const int j = idx / TE, t = idx % TE;
      const long long i = base + t;
      const double2 v = i < N ? V[(long long)j * N + i] : make_double2(0.0, 0.0);
      const float2 h = make_float2((float)v.x, (float)v.y);
      const float2 l = split_lo(v, h);
      tile[idx] = make_float4(h.x, h.y, l.x, l.y);
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < groups * TE; idx += blockDim.x) {
      const int g = idx / TE, t = idx % TE;
      const long long i = base + t;
      DSAccX2 acc[CPT];
      float2 small[CPT];
      const float2* yc[CPT];
#pragma unroll
      for (int q = 0; q < CPT; ++q) {
        small[q] = make_float2(0.f, 0.f);
        yc[q] = Yhl + (long long)min(g * CPT + q, k - 1) * m;  // columns past k: computed, not stored
      }
      for (int j = 0; j < m; ++j) {
        const float4 v = tile[j * TE + t];
        const float2 vh = make_float2(v.x, v.y), vl = make_float2(v.z, v.w);
#pragma unroll
        for (int q = 0; q < CPT; ++q) {
          const float2 y = __ldg(yc[q] + j);
          const float2 yh = make_float2(y.x, y.x), yl = make_float2(y.y, y.y);
          float2 pr, e;
          two_prod_x2(yh, vh, pr, e);
          acc[q].add(pr);
          small[q] = add_x2(small[q], fma_x2(yh, vl, fma_x2(yl, vh, e)));
        }
      }
      if (i < N) {
#pragma unroll
        for (int q = 0; q < CPT; ++q) {
          const int col = g * CPT + q;
          if (col < k)
            V[(long long)col * N + i] =
                make_double2((double)acc[q].hi.x + ((double)acc[q].lo.x + (double)small[q].x),
                             (double)acc[q].hi.y + ((double)acc[q].lo.y + (double)small[q].y));
        }
      }
    }
    __syncthreads();
  }
}

// out[(p * m + j) * 2 + {0,1}] = sum over the nb block partials of k_exact_dots; grid (m, P)
__global__ void __launch_bounds__(kRedThreads)
k_dots_finish(const double* __restrict__ part, int m, int nb, double* __restrict__ out, const int* __restrict__ active) {
  const int j = blockIdx.x, p = blockIdx.y;
  if (active && !active[p]) return;
  double re = 0.0, im = 0.0;
  for (int b = threadIdx.x; b < nb; b += kRedThreads) {
    re += part[(((long long)p * m + j) * nb + b) * 2 + 0];
    im += part[(((long long)p * m + j) * nb + b) * 2 + 1];
  }
  re = block_sum<kRedThreads>(re);
  im = block_sum<kRedThreads>(im);
  if (threadIdx.x == 0) {
    out[((long long)p * m + j) * 2] = re;
    out[((long long)p * m + j) * 2 + 1] = im;
  }
}

// part[(((p * m + j) * gridDim.y) + b) * 2 + {0, 1}] = block b's share of
// conj(S_pj)^T w_p (S = Shi + Slo, w = whi + wlo) for the two vectors
// j = 2 blockIdx.x, 2 blockIdx.x + 1 < m; grid (ceil(m / 2), blocks, P).  A thread
// takes two neighbouring elements at a time (N is even): six 16-byte loads in
// flight.  Bound by memory, 16 bytes per element and vector: all pairs of one
// range of elements run together (their w is read from L2) and few blocks per
// pair, whose FP64 ends (a pair sum per value, then the block's) would otherwise
// show.  One GB300, 52 vectors, with k_dots_finish: 752 us at 96^3 and 174 at 32^3
// with 304 blocks per pair, 8-byte loads, a full block sum per value and the
// blocks of one pair together (w from memory again for every pair), 594 and 82 now
// (430 at 96^3 at the copy rate).  The error against 64 bits, rms of 40 products of
// random vectors over the sum of the terms' magnitudes: 3.8e-18 then and 3.9e-18
// now at 96^3, 7.8e-18 and 8.0e-18 at 32^3; with one FP32 sum for both elements of
// the pair 1.2e-17 at 32^3.
__global__ void __launch_bounds__(kRedThreads)
k_exact_dots(const float2* __restrict__ Shi, const float2* __restrict__ Slo, long long sstride, int m,
             const float2* __restrict__ whi, const float2* __restrict__ wlo, long long N, double* __restrict__ part,
             const int* __restrict__ active) {
  constexpr int G = 2;
  const int p = blockIdx.z;
  if (active && !active[p]) return;
  const int j0 = blockIdx.x * G;
  const int j1 = min(j0 + 1, m - 1);  // (an odd last vector is done twice and stored once)
  const float4* wh4 = reinterpret_cast<const float4*>(whi + (long long)p * N);
  const float4* wl4 = reinterpret_cast<const float4*>(wlo + (long long)p * N);
  const float4* sh4[G] = {reinterpret_cast<const float4*>(Shi + p * sstride + j0 * N),
                          reinterpret_cast<const float4*>(Shi + p * sstride + j1 * N)};
  const float4* sl4[G] = {reinterpret_cast<const float4*>(Slo + p * sstride + j0 * N),
                          reinterpret_cast<const float4*>(Slo + p * sstride + j1 * N)};
  // per vector and element of the pair: the exact sum of the hi x hi products
  // (real, imaginary) and an ordinary sum of their rounding errors and the hi x
  // lo, lo x hi terms.  (Apart for the two elements: the error of the ordinary
  // sums grows with their length.)
  DSAccX2 acc[G][2];
  float2 small[G][2];
#pragma unroll
  for (int g = 0; g < G; ++g) small[g][0] = small[g][1] = make_float2(0.f, 0.f);
  for (long long i = (long long)blockIdx.y * kRedThreads + threadIdx.x; i < N / 2; i += (long long)gridDim.y * kRedThreads) {
    const float4 bh4 = wh4[i], bl4 = wl4[i];
    float4 ah4[G], al4[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      ah4[g] = __ldcs(sh4[g] + i);
      al4[g] = __ldcs(sl4[g] + i);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float2 bh = h == 0 ? make_float2(bh4.x, bh4.y) : make_float2(bh4.z, bh4.w);
      const float2 bl = h == 0 ? make_float2(bl4.x, bl4.y) : make_float2(bl4.z, bl4.w);
      // conj(a) b = (ar br + ai bi, ar bi - ai br) = ar (br, bi) + ai (bi, -br)
      const float2 bh2 = make_float2(bh.y, -bh.x), bl2 = make_float2(bl.y, -bl.x);
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const float2 ah = h == 0 ? make_float2(ah4[g].x, ah4[g].y) : make_float2(ah4[g].z, ah4[g].w);
        const float2 al = h == 0 ? make_float2(al4[g].x, al4[g].y) : make_float2(al4[g].z, al4[g].w);
        const float2 ax = make_float2(ah.x, ah.x), ay = make_float2(ah.y, ah.y);
        float2 p1, e1, p2, e2;
        two_prod_x2(ax, bh, p1, e1);
        two_prod_x2(ay, bh2, p2, e2);
        acc[g][h].add(p1);
        acc[g][h].add(p2);
        float2 t = add_x2(e1, e2);
        t = fma_x2(ax, bl, t);
        t = fma_x2(make_float2(al.x, al.x), bh, t);
        t = fma_x2(ay, bl2, t);
        t = fma_x2(make_float2(al.y, al.y), bh2, t);
        small[g][h] = add_x2(small[g][h], t);
      }
    }
  }
#pragma unroll
  for (int g = 0; g < G; ++g) {
    acc[g][0].add(acc[g][1].hi);
    acc[g][0].lo = add_x2(acc[g][0].lo, acc[g][1].lo);
    small[g][0] = add_x2(small[g][0], small[g][1]);
  }
  // block sums in FP64.  (Double-single sums on the FP32 units lost the
  // accuracy the monitor needs on homogeneous media at symmetric k-points:
  // spurious losses of 1e-6 and wrong degenerate eigenvalues.)  The four values
  // of a warp at once: two halving exchanges leave each eight lanes with one of
  // them, three more steps complete it (six FP64 additions instead of twenty).
  double v[2 * G];
#pragma unroll
  for (int g = 0; g < G; ++g) {
    v[2 * g] = (double)acc[g][0].hi.x + (double)acc[g][0].lo.x + (double)small[g][0].x;
    v[2 * g + 1] = (double)acc[g][0].hi.y + (double)acc[g][0].lo.y + (double)small[g][0].y;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int h = G, o = 16; h >= 1; h >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int t = 0; t < h; ++t) {
      const double keep = up ? v[t + h] : v[t], give = up ? v[t] : v[t + h];
      v[t] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
  __shared__ double sh[kRedThreads / 32][2 * G];
  if ((lane & 7) == 0) sh[warp][((lane >> 4) & 1) * 2 + ((lane >> 3) & 1)] = v[0];
  __syncthreads();
  if (threadIdx.x < 2 * G && j0 + (int)threadIdx.x / 2 < m) {
    double t = sh[0][threadIdx.x];
#pragma unroll
    for (int w = 1; w < kRedThreads / 32; ++w) t += sh[w][threadIdx.x];
    part[(((long long)p * m + j0 + threadIdx.x / 2) * gridDim.y + blockIdx.y) * 2 + threadIdx.x % 2] = t;
  }
}

// w -> (whi, wlo) floats with whi + wlo = w to ~1e-15 (once per vector, so
// that the inner-product kernel runs no double-precision arithmetic)
__global__ void k_split_hi_lo(const double2* __restrict__ w, float2* __restrict__ whi, float2* __restrict__ wlo,
                              long long total) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const double2 v = w[i];
    const float2 h = make_float2((float)v.x, (float)v.y);
    whi[i] = h;
    wlo[i] = split_lo(v, h);
  }
}

// New basis vector j of every active problem: V_pj = s_p w_p, MV_pj = s_p Mw_p
// in FP64, plus their complex64 shadows and the FP64 remainder of the MV
// shadow (MV = MV32 + MV32lo to ~1e-15).
__global__ void k_store_basis_vector(const double2* __restrict__ w, const double2* __restrict__ Mw,
                                     const double* __restrict__ s, double2* __restrict__ V, double2* __restrict__ MV,
                                     float2* __restrict__ V32, float2* __restrict__ MV32, float2* __restrict__ MV32lo,
                                     long long vstride, int j, long long N, int P, const int* __restrict__ active) {
  for (long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x; g < N * P; g += (long long)gridDim.x * blockDim.x) {
    const long long p = g / N, i = g % N;
    if (active && !active[p]) continue;
    const double f = s[p];
    const double2 a = cscale(w[g], f), b = cscale(Mw[g], f);
    const long long o = p * vstride + (long long)j * N + i;
    V[o] = a;
    MV[o] = b;
    V32[o] = make_float2((float)a.x, (float)a.y);
    const float2 bh = make_float2((float)b.x, (float)b.y);
    MV32[o] = bh;
    MV32lo[o] = split_lo(b, bh);
  }
}

// Shadows of vectors [first, first + count) of every problem (after a basis
// rotation): V32, MV32 and MV32lo from V and MV.
__global__ void k_refresh_shadows(const double2* __restrict__ V, const double2* __restrict__ MV,
                                  float2* __restrict__ V32, float2* __restrict__ MV32, float2* __restrict__ MV32lo,
                                  long long vstride, long long len, int P) {
  for (long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x; g < len * P; g += (long long)gridDim.x * blockDim.x) {
    const long long p = g / len, i = g % len;
    const long long o = p * vstride + i;
    const double2 a = V[o], b = MV[o];
    V32[o] = make_float2((float)a.x, (float)a.y);
    const float2 bh = make_float2((float)b.x, (float)b.y);
    MV32[o] = bh;
    MV32lo[o] = split_lo(b, bh);
  }
}

}  // namespace nfs
