// Kernels of the null space free standard problem for any nonsingular B
// (see nfsep.h).  The DFT kernels are those of the A_r product
// (matvec_kernels.cuh); only the per-voxel step of the column kernel and the
// scalings around the product differ.
#include <algorithm>
#include <cmath>

#include "matvec_impl.cuh"
#include "nfsep.h"

namespace nfs {

namespace {

__global__ void k_nfsep_root(const double2* __restrict__ lam, int n1, int n2, long long n, double* __restrict__ root) {
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    const int i1 = (int)(e % n1);
    const int i2 = (int)((e / n1) % n2);
    const int i3 = (int)(e / ((long long)n1 * n2));
    const double lq = cabs2(lam[i1]) + cabs2(lam[n1 + i2]) + cabs2(lam[n1 + n2 + i3]);
    root[e] = sqrt(sqrt(lq));
  }
}

// (e_c, h_c) = B_c^{-1} (p_c, q_c) for component c = the pair of one voxel
struct BinvStep {
  const double2* binv;
  long long n;
  double scale;
  template <int NB>
  struct Vals {};
  template <int NB>
  __device__ __forceinline__ void load(const ColumnPos&, int, Vals<NB>&) const {}
  __device__ __forceinline__ void solve(const ColumnPos& c, long long v, double2 p, double2 q, double2& e,
                                        double2& h) const {
    const double2* b = binv + 4 * c.j * n + v;
    e = cscale(cadd(cmul(b[0], p), cmul(b[n], q)), scale);
    h = cscale(cadd(cmul(b[2 * n], p), cmul(b[3 * n], q)), scale);
  }
};

struct NfsepStep : BinvStep {
  static constexpr bool kForward = true;
  template <int NB>
  __device__ __forceinline__ double apply(const ColumnPos& c, int b, const Vals<NB>&, int, double2& p, double2& q) const {
    double2 e, h;
    solve(c, c.voxel(b), p, q, e, h);
    p = h;  // projected by P_r^*
    q = e;  // projected by Q_r^*
    return 0.0;
  }
};

struct NfsepFieldsStep : BinvStep {
  static constexpr bool kForward = false;
  const double2* bloch;
  double2* X;
  template <int NB>
  __device__ __forceinline__ double apply(const ColumnPos& c, int b, const Vals<NB>&, int, double2& p, double2& q) const {
    const long long v = c.voxel(b);
    double2 e, h;
    solve(c, v, p, q, e, h);
    const double2 d = cmul(cmul(bloch[c.x], bloch[c.n1 + c.a + c.N1 * b]), bloch[2 * c.n1 + c.z]);
    X[c.j * n + v] = cmul(d, e);
    X[(3 + c.j) * n + v] = cmul(d, h);
    return 0.0;
  }
};

__global__ void k_zscale_copy(const double2* __restrict__ src, double2* __restrict__ dst, double scale, long long N) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (long long)gridDim.x * blockDim.x)
    dst[i] = cscale(src[i], scale);
}

// in place: a tile of TE elements of all m vectors in shared memory, then the
// k combinations written back
template <int TE>
__global__ void k_zrotate(double2* __restrict__ V, int m, const double* __restrict__ Y, int k, long long N) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* tile = reinterpret_cast<double2*>(smem_raw);  // [m][TE]
  for (long long base = (long long)blockIdx.x * TE; base < N; base += (long long)gridDim.x * TE) {
    for (int idx = threadIdx.x; idx < m * TE; idx += blockDim.x) {
      const int j = idx / TE, t = idx % TE;
      const long long i = base + t;
      tile[idx] = i < N ? V[(long long)j * N + i] : make_double2(0.0, 0.0);
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < k * TE; idx += blockDim.x) {
      const int o = idx / TE, t = idx % TE;
      const long long i = base + t;
      double2 acc = make_double2(0.0, 0.0);
      for (int r = 0; r < m; ++r) {
        const double2 y = make_double2(Y[2 * ((long long)r * k + o)], Y[2 * ((long long)r * k + o) + 1]);
        acc = cadd(acc, cmul(tile[r * TE + t], y));
      }
      if (i < N) V[(long long)o * N + i] = acc;
    }
    __syncthreads();
  }
}

// --- device-resident GMRES -------------------------------------------------
//
// A step is seven kernels: the three of the product (which also end the
// Gram-Schmidt update of the step before and normalise its vector, KrylovFuse)
// and dots, update, dots, update.  At 8^3 (2048 elements, up to 101 basis
// vectors) every one is a chain of latencies and FP64 instructions, so the work
// is spread over as many SMs as the vectors allow: the dots over element tiles
// and groups of 8 vectors, the updates over elements and groups of vectors,
// whose partial sums the next kernel adds up (w - sum_g tmp_g).  One GB300, a
// step at 8^3: 62 us with fourteen kernels (separate scalings, sums over the
// groups, norm column and store; 78 with the product they were written for), 39
// us now; at 16^3 104.

constexpr int kGsThreads = 256;
constexpr int kGsTile = 128;      // elements of w that a block of k_gs_dots holds
constexpr int kGsMaxChunks = 64;
constexpr int kGsPerWarp = 2;     // vectors per warp (4: the FP64 work of a block takes 3 us instead of 1.9)

// grid (S, ceil(m / 8)): part[(s m + j) 2 + {0, 1}] = chunk s's share of
// V_j^* w', w' = w - sum_{g < G} tmp_g (written to w2 when G > 0)
__global__ void __launch_bounds__(kGsTile)
k_gs_dots(const double2* V, int m, const double2* w, const double2* tmp, int G, double2* w2, long long N,
          long long chunk, double* part) {
  constexpr int PER = kGsTile / 32;  // elements of a tile per lane
  __shared__ double2 ws[kGsTile];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int j0 = (blockIdx.y * (kGsTile / 32) + warp) * kGsPerWarp;
  const int s = blockIdx.x;
  const long long i0 = (long long)s * chunk, i1 = min(N, i0 + chunk);
  double2 x[kGsPerWarp][PER];
  auto fetch = [&](long long base) {
#pragma unroll
    for (int t = 0; t < kGsPerWarp; ++t)
      if (j0 + t < m)
#pragma unroll
        for (int k = 0; k < PER; ++k) {
          const long long i = base + k * 32 + lane;
          x[t][k] = i < i1 ? V[(long long)(j0 + t) * N + i] : make_double2(0.0, 0.0);
        }
  };
  depend_wait();
  fetch(i0);
  double acc[2 * kGsPerWarp];
#pragma unroll
  for (int t = 0; t < 2 * kGsPerWarp; ++t) acc[t] = 0.0;
  for (long long base = i0; base < i1; base += kGsTile) {
    const long long i = base + threadIdx.x;
    // (before w' is formed and stored: plain loads stay behind the store)
    if (base > i0) fetch(base);
    double2 a = make_double2(0.0, 0.0);
    if (i < i1) {
      a = minus_groups(w[i], tmp + i, N, G);
      if (G > 0 && blockIdx.y == 0) w2[i] = a;
    }
    if (base > i0) __syncthreads();  // the tile before has been read
    ws[threadIdx.x] = a;
    __syncthreads();
#pragma unroll
    for (int t = 0; t < kGsPerWarp; ++t)
      if (j0 + t < m)
#pragma unroll
        for (int k = 0; k < PER; ++k) {
          const double2 v = x[t][k], y = ws[k * 32 + lane];
          acc[2 * t] += v.x * y.x + v.y * y.y;
          acc[2 * t + 1] += v.x * y.y - v.y * y.x;
        }
  }
  depend_begin();
  // the four sums over the 32 lanes at once: two halving exchanges leave each
  // eight lanes with one of the four values, three more steps complete it (six
  // FP64 additions instead of twenty)
#pragma unroll
  for (int h = kGsPerWarp, o = 16; h >= 1; h >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int t = 0; t < h; ++t) {
      const double keep = up ? acc[t + h] : acc[t], give = up ? acc[t] : acc[t + h];
      acc[t] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
  static_assert(kGsPerWarp == 2, "two exchanges");
  const int which = ((lane >> 4) & 1) * 2 + ((lane >> 3) & 1);
  if ((lane & 7) == 0 && j0 + which / 2 < m) part[((long long)s * m + j0) * 2 + which] = acc[0];
}

// grid (ceil(N / NT), G): tmp[g N + i] = sum over the g-th group of VB basis
// vectors of c_j V_j[i], c_j = sum over the S chunks' partials
template <int NT>
__global__ void __launch_bounds__(NT)
k_gs_update(const double2* V, long long N, int m, int VB, const double* part, int S, double2* tmp) {
  constexpr int AHEAD = 12;  // vectors fetched before the coefficients are summed
  __shared__ double2 cs[kGmresMax];
  const int j0 = blockIdx.y * VB, nj = min(VB, m - j0);
  const long long i = (long long)blockIdx.x * NT + threadIdx.x;
  const double2* v = V + (long long)j0 * N + (i < N ? i : 0);
  double2 x[AHEAD];
  depend_wait();
#pragma unroll
  for (int t = 0; t < AHEAD; ++t)
    if (t < nj) x[t] = v[(long long)t * N];
  // four threads add up one coefficient
  for (int t = threadIdx.x; t < (nj + NT / 4 - 1) / (NT / 4) * NT; t += NT) {
    const int j = t / 4;
    double re = 0.0, im = 0.0;
    if (j < nj) {
      const double2* p = reinterpret_cast<const double2*>(part) + j0 + j;
#pragma unroll 4
      for (int q = t % 4; q < S; q += 4) {
        const double2 y = p[(long long)q * m];
        re += y.x;
        im += y.y;
      }
    }
#pragma unroll
    for (int o = 2; o > 0; o >>= 1) {
      re += __shfl_xor_sync(0xffffffffu, re, o);
      im += __shfl_xor_sync(0xffffffffu, im, o);
    }
    if (t % 4 == 0 && j < nj) cs[j] = make_double2(re, im);
  }
  __syncthreads();
  depend_begin();
  if (i >= N) return;
  double2 a0 = make_double2(0.0, 0.0), a1 = a0;
#pragma unroll
  for (int t = 0; t < AHEAD; t += 2) {
    if (t < nj) a0 = cadd(a0, cmul(cs[t], x[t]));
    if (t + 1 < nj) a1 = cadd(a1, cmul(cs[t + 1], x[t + 1]));
  }
  int j = AHEAD;
  for (; j + 8 <= nj; j += 8) {
    double2 y[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) y[t] = v[(long long)(j + t) * N];
#pragma unroll
    for (int t = 0; t < 8; t += 2) {
      a0 = cadd(a0, cmul(cs[j + t], y[t]));
      a1 = cadd(a1, cmul(cs[j + t + 1], y[t + 1]));
    }
  }
  for (; j < nj; ++j) a0 = cadd(a0, cmul(cs[j], v[(long long)j * N]));
  tmp[(long long)blockIdx.y * N + i] = cadd(a0, a1);
}

// sum over the block (blockDim.x = kGsThreads); the result in every thread
__device__ __forceinline__ double gs_block_sum(double v) {
  RedAcc<double> a;
  a.v = v;
  return a.block_total<kGsThreads>();
}

// dst = w - sum_g tmp_g, and (nrm_part != nullptr) the partials of |dst|^2
__global__ void __launch_bounds__(kGsThreads)
k_gs_finish(const double2* w, const double2* tmp, int G, double2* dst, long long N, double* nrm_part) {
  depend_wait();
  double nr = 0.0;
  for (long long i = (long long)blockIdx.x * kGsThreads + threadIdx.x; i < N; i += (long long)gridDim.x * kGsThreads) {
    const double2 a = minus_groups(w[i], tmp + i, N, G);
    dst[i] = a;
    nr += cabs2(a);
  }
  depend_begin();
  if (nrm_part) {
    nr = gs_block_sum(nr);
    if (threadIdx.x == 0) nrm_part[blockIdx.x] = nr;
  }
}

__global__ void __launch_bounds__(kGsThreads)
k_gmres_residual(const double2* __restrict__ b, double2* __restrict__ w, long long N, double* __restrict__ nrm_part) {
  double nr = 0.0;
  for (long long i = (long long)blockIdx.x * kGsThreads + threadIdx.x; i < N; i += (long long)gridDim.x * kGsThreads) {
    const double2 a = csub(b[i], w[i]);
    w[i] = a;
    nr += cabs2(a);
  }
  nr = gs_block_sum(nr);
  if (threadIdx.x == 0) nrm_part[blockIdx.x] = nr;
}

// Columns j0 .. j0 + gridDim.x - 1 of H from their steps' partials: step t's
// two passes at part + 2 t plen (and + plen), its norm partials at nrm + t nlen
// (nnrm of them; the last step's at nrm_last, nlast of them).
__global__ void __launch_bounds__(kGsThreads)
k_gmres_columns(int j0, const double* part, long long plen, int S, const double* nrm, long long nlen, int nnrm,
                const double* nrm_last, int nlast, GmresDev* st) {
  depend_wait();
  depend_begin();
  const int t = blockIdx.x, j = j0 + t, m = j + 1;
  const double* p1 = part + 2 * t * plen;
  const double* p2 = p1 + plen;
  double2* col = st->Hc + (long long)j * (kGmresMax + 1);
  for (int i = threadIdx.x; i < m; i += kGsThreads) {
    double re = 0.0, im = 0.0;
#pragma unroll 4
    for (int q = 0; q < S; ++q) {
      const double2 x = reinterpret_cast<const double2*>(p1)[(long long)q * m + i];
      const double2 y = reinterpret_cast<const double2*>(p2)[(long long)q * m + i];
      re += x.x + y.x;
      im += x.y + y.y;
    }
    col[i] = make_double2(re, im);
  }
  const bool last = t == (int)gridDim.x - 1;
  const double* np = last ? nrm_last : nrm + t * nlen;
  double h = 0.0;
  for (int i = threadIdx.x; i < (last ? nlast : nnrm); i += kGsThreads) h += np[i];
  h = sqrt(fmax(gs_block_sum(h), 0.0));
  if (threadIdx.x == 0) col[j + 1] = make_double2(h, 0.0);
}

int blocks_for(long long work) { return (int)std::max<long long>(1, std::min<long long>((work + 255) / 256, 152LL * 16)); }

}  // namespace

cudaError_t nfsep_root(const double2* lam, int n1, int n2, int n3, double* root, cudaStream_t s) {
  const long long n = (long long)n1 * n2 * n3;
  k_nfsep_root<<<blocks_for(n), 256, 0, s>>>(lam, n1, n2, n, root);
  return cudaGetLastError();
}

cudaError_t nfsep_prepare(int n1, int n3) {
  const cudaError_t e = columns_prepare<double, NfsepStep>(n1, n3);
  return e != cudaSuccess ? e : columns_prepare<double, NfsepFieldsStep>(n1, n3);
}

cudaError_t nfsep_columns(void* fld, const double2* binv, const double2* tw1, const double2* tw3, int n1, int n3,
                          cudaStream_t s) {
  const long long n = (long long)n1 * n1 * n3;
  NfsepStep step;
  step.binv = binv;
  step.n = n;
  step.scale = 1.0 / (double)n;
  return columns_launch<double>(fld, step, tw1, tw3, n1, n3, 1, nullptr, nullptr, BatchStrides{}, s);
}

cudaError_t nfsep_fields(void* fld, const double2* binv, const double2* tw1, const double2* tw3, const double2* bloch,
                         int n1, int n3, double2* X, cudaStream_t s) {
  const long long n = (long long)n1 * n1 * n3;
  NfsepFieldsStep step;
  step.binv = binv;
  step.n = n;
  step.scale = 1.0 / std::sqrt((double)n);
  step.bloch = bloch;
  step.X = X;
  return columns_launch<double>(fld, step, tw1, tw3, n1, n3, 1, nullptr, nullptr, BatchStrides{}, s);
}

cudaError_t zscale_copy(const double2* src, double2* dst, double scale, long long N, cudaStream_t s) {
  k_zscale_copy<<<blocks_for(N), 256, 0, s>>>(src, dst, scale, N);
  return cudaGetLastError();
}

cudaError_t zrotate(double2* V, int m, const double* Y, int k, long long N, cudaStream_t s) {
  constexpr int TE = 32;
  const size_t smem = (size_t)m * TE * sizeof(double2);
  cudaError_t e = cudaFuncSetAttribute(k_zrotate<TE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int blocks = (int)std::max<long long>(1, std::min<long long>((N + TE - 1) / TE, 152LL * 8));
  k_zrotate<TE><<<blocks, 256, smem, s>>>(V, m, Y, k, N);
  return cudaGetLastError();
}

int gs_chunks(long long N) {
  return (int)std::min<long long>(kGsMaxChunks, (N + kGsTile - 1) / kGsTile);
}
int gs_norm_blocks(long long N) { return blocks_for(N); }

// Vector groups of the update: enough that the GPU has about four warps per SM
// (grids up to 24^3 or so), one for longer vectors
static int gs_groups(long long N, int m) {
  const long long warps = (N + 31) / 32;
  return (int)std::max<long long>(1, std::min<long long>((m + 7) / 8, 152 * 4 / warps));
}
long long gs_tmp_len(long long N) { return (long long)gs_groups(N, kGmresMax) * N; }
// kernels of vectors this short overlap (see depend_wait)
static bool gs_serial(long long N) { return N >= 152LL * 256; }

cudaError_t gs_dots(const double2* V, int m, const double2* w, const double2* tmp, int G, double2* w2, long long N,
                    double* part, cudaStream_t s) {
  if (m <= 0 || m > kGmresMax) return cudaErrorInvalidValue;
  const int S = gs_chunks(N);
  const long long chunk = ((N + S - 1) / S + kGsTile - 1) / kGsTile * kGsTile;
  return launch_dependent(gs_serial(N), k_gs_dots, dim3(S, (m + 7) / 8), kGsTile, 0, s, V, m, w, tmp, G, w2, N,
                          chunk, part);
}

cudaError_t gs_update(const double2* V, int m, long long N, const double* part, int S, double2* tmp, int* groups,
                      cudaStream_t s) {
  if (m <= 0 || m > kGmresMax) return cudaErrorInvalidValue;
  const int VB = (m + gs_groups(N, m) - 1) / gs_groups(N, m);
  const int G = (m + VB - 1) / VB;
  *groups = G;
  if (gs_serial(N))
    return launch_dependent(true, k_gs_update<256>, dim3((unsigned)((N + 255) / 256), G), 256, 0, s, V, N, m, VB, part,
                            S, tmp);
  return launch_dependent(false, k_gs_update<64>, dim3((unsigned)((N + 63) / 64), G), 64, 0, s, V, N, m, VB, part, S,
                          tmp);
}

cudaError_t gs_finish(const double2* w, const double2* tmp, int G, double2* dst, long long N, double* nrm_part,
                      cudaStream_t s) {
  return launch_dependent(gs_serial(N), k_gs_finish, dim3(gs_norm_blocks(N)), kGsThreads, 0, s, w, tmp, G, dst, N,
                          nrm_part);
}

cudaError_t gmres_residual(const double2* b, double2* w, long long N, double* nrm_part, cudaStream_t s) {
  k_gmres_residual<<<gs_norm_blocks(N), kGsThreads, 0, s>>>(b, w, N, nrm_part);
  return cudaGetLastError();
}

cudaError_t gmres_columns(int j0, int nsteps, const double* part, long long plen, int S, const double* nrm,
                          long long nlen, int nnrm, const double* nrm_last, int nlast, GmresDev* st, cudaStream_t s) {
  if (j0 < 0 || j0 + nsteps > kGmresMax) return cudaErrorInvalidValue;
  return launch_dependent(false, k_gmres_columns, dim3(nsteps), kGsThreads, 0, s, j0, part, plen, S, nrm, nlen, nnrm,
                          nrm_last, nlast, st);
}

}  // namespace nfs

