// Device-resident CG state and the accumulator of the vector reductions,
// shared by the vector kernels (blas_kernels.cuh) and the product's kernels,
// which take the CG step themselves (matvec_kernels.cuh).  Declarations only.
#pragma once
#include <type_traits>

#include "nfs_complex.cuh"

namespace nfs {

constexpr int kRedBlocks = 304;   // two blocks per SM on a 152-SM GB300
constexpr int kRedThreads = 256;
constexpr int kMaxPartials = 3072;  // >= kRedBlocks and the CTAs of one problem in any kernel of the product

// CG state of one problem, device resident (an array of P).  The scalars of
// the recurrence come from per-CTA partial sums that every CTA of the next
// kernel adds up itself, in the same order (so all agree): a last CTA that
// sums for the others (an atomic count, the form measured before) costs each
// kernel a fence, an atomic and a serial sum at its end, about 4 us each on the
// 48^3 kernels that take 5 us without it.  One CTA records what the later
// kernels need.  Flags are written only by kernels that do not read them, so
// every CTA of a launch sees the same value:
//   stop   k_rows_in writes, k_columns and k_rows_out read: nothing left to do
//   halt   k_rows_out writes, k_rows_in and k_cg_check read: stop was set, or a
//          breakdown
// `partial` values are doubles (complex128) or (hi, lo) float pairs
// (complex64), eight bytes either way.
struct CGState {
  // what the host reads (set by k_cg_check at the end of a chunk)
  double rr;        // r^* r of the current residual
  double rr0;       // and of the one at the start (set by k_cg_init)
  int it, maxit;    // steps taken, and how many are allowed
  int done;         // 1: converged, broken down or out of iterations
  int status;       // 0, -6 (no convergence) or -7 (breakdown)
  // the recurrence
  int stop, halt, broken, pad;
  double rr_now;    // r^* r of this step's residual (k_rows_in; a `partial`)
  double rr_last;   // of the step before (k_rows_out; infinite at the start: beta = 0)
  double tol2;      // stop when r^* r <= tol2 (a `partial`)
  double part_a[kMaxPartials];  // p^* A p, one per CTA of k_columns (at the start: of r^* r)
  double part_b[kMaxPartials];  // r^* r, one per CTA of k_rows_out
};
constexpr long long kStateDoubles = sizeof(CGState) / sizeof(double);
static_assert(sizeof(CGState) % sizeof(double) == 0, "CGState must be a whole number of doubles");

// Per-thread accumulator and block sum of the CG reductions (the partials
// of p^* A p and r^* r).  Complex64 runs accumulate in double-single
// arithmetic on the FP32 units (hi + lo floats, TwoSum: ~1e-14 of the sum of
// the terms' magnitudes) and complex128 runs in FP64.  FP64 arithmetic is
// scarce on this GPU: a block sum of doubles in every CTA of a pass keeps
// the SM's FP64 pipe busy for microseconds.
template <typename T>
struct RedAcc;
template <>
struct RedAcc<double> {
  using value_type = double;
  using partial = double;
  double v = 0.0;
  __device__ __forceinline__ void add(double x) { v += x; }
  __device__ __forceinline__ void add_partial(double x) { v += x; }
  // the block's total, valid in every thread; all threads must call it
  template <int NT>
  __device__ __forceinline__ double block_total() {
    __shared__ double sh[NT / 32];
    double t = v;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (NT == 32) return t;
    __syncthreads();  // sh may still be read by an earlier call
    if (lane == 0) sh[warp] = t;
    __syncthreads();
    double r = sh[0];
#pragma unroll
    for (int w = 1; w < NT / 32; ++w) r += sh[w];
    return r;
  }
};
template <>
struct RedAcc<float> {
  using value_type = float;
  using partial = float2;
  float hi = 0.f, lo = 0.f;
  // (hi, lo) += (bh, bl): TwoSum of the high parts, the rest to the error, renormalised
  __device__ __forceinline__ static void ds_add(float& hi, float& lo, float bh, float bl) {
    const float s = hi + bh;
    const float bb = s - hi;
    const float e = ((hi - (s - bb)) + (bh - bb)) + (lo + bl);
    hi = s + e;
    lo = e - (hi - s);
  }
  __device__ __forceinline__ void add(float x) {
    const float s = hi + x;
    const float bb = s - hi;
    lo += (hi - (s - bb)) + (x - bb);
    hi = s;
  }
  __device__ __forceinline__ void add_partial(float2 x) { ds_add(hi, lo, x.x, x.y); }
  template <int NT>
  __device__ __forceinline__ float2 block_total() {
    __shared__ float2 sh[NT / 32];
    float th = hi, tl = lo;
    ds_add(th, tl, 0.f, 0.f);  // renormalise
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      ds_add(th, tl, __shfl_xor_sync(0xffffffffu, th, o), __shfl_xor_sync(0xffffffffu, tl, o));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (NT == 32) return make_float2(th, tl);
    __syncthreads();  // sh may still be read by an earlier call
    if (lane == 0) sh[warp] = make_float2(th, tl);
    __syncthreads();
    float rh = sh[0].x, rl = sh[0].y;
#pragma unroll
    for (int w = 1; w < NT / 32; ++w) ds_add(rh, rl, sh[w].x, sh[w].y);
    return make_float2(rh, rl);
  }
};
// the accumulator for data of real type R (complex64 or complex128 runs)
template <typename R>
using RedAccFor = RedAcc<typename std::conditional<std::is_same<R, float>::value, float, double>::type>;

// The block's sum of n partials, in every thread, the same in every block of
// the same size.
template <typename R, int NT>
__device__ __forceinline__ typename RedAccFor<R>::partial sum_partials_all(const double* part, int n) {
  using P = typename RedAccFor<R>::partial;
  const P* q = reinterpret_cast<const P*>(part);
  RedAccFor<R> acc;
#pragma unroll 4
  for (int i = threadIdx.x; i < n; i += NT) acc.add_partial(q[i]);
  return acc.template block_total<NT>();
}
// Scalars of the recurrence in either form.
__device__ __forceinline__ double scalar_ratio(double a, double b) { return a / b; }
// a / b of float pairs: the quotient of the high parts and one correction
// step, rounded to float at the end (b infinite: 0)
__device__ __forceinline__ float scalar_ratio(float2 a, float2 b) {
  const float q = a.x / b.x;
  if (!(fabsf(b.x) <= 3.4e38f)) return q;
  const float rem = fmaf(-q, b.x, a.x) + (a.y - q * b.y);
  return q + rem / b.x;
}
__device__ __forceinline__ bool scalar_le(double a, double b) { return a <= b; }
__device__ __forceinline__ bool scalar_le(float2 a, float2 b) { return a.x < b.x || (a.x == b.x && a.y <= b.y); }
__device__ __forceinline__ bool scalar_nan(double a) { return !(a == a); }
__device__ __forceinline__ bool scalar_nan(float2 a) { return !(a.x == a.x); }
__device__ __forceinline__ bool scalar_positive(double a) { return a > 0.0; }
__device__ __forceinline__ bool scalar_positive(float2 a) { return a.x > 0.f; }
__device__ __forceinline__ double scalar_double(double a) { return a; }
__device__ __forceinline__ double scalar_double(float2 a) { return (double)a.x + (double)a.y; }
__device__ __forceinline__ void scalar_from(double v, double& out) { out = v; }
__device__ __forceinline__ void scalar_from(double v, float2& out) {
  const float h = (float)v;
  const double d = v - (double)h;
  out = make_float2(h, d == d ? (float)d : 0.f);  // (an infinite v has no low part)
}

}  // namespace nfs
