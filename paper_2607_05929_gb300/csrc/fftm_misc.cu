// Reductions, Anderson acceleration on p, and field (un)packing.
//
// Anderson acceleration on p (Sec. 2.3, Algorithm 1).  With couples (q_j, g_j),
// g_j = p_{j+1} the polarisation divergence produced by the transformed field
// q_j, the residual of a couple is f_j = g_j - q_j and the accelerated field
// is sum_j c_j g_j with c = argmin || sum_j c_j f_j ||_2, sum_j c_j = 1.  Since
// the Green operator inverts div(R0 : grad .) exactly on the transformed
// fields, q_j = div(R0 : grad u^{j+1}) and f_j = -D^{j+1}: the same step reads
// u_new = sum_k c_k u^k - Gamma(sum_k c_k D^k) with c = argmin ||sum_k c_k D^k||
// over the last iterates u^k and their residuals D^k.  That is the form used
// here (it keeps the rounding of the update relative to the residual).  The
// normal equations of the differences D_k - D_last are accumulated in FP64
// and solved by Cholesky in FP64 by one thread; a pivot below `pivot_tol`
// times its diagonal entry rejects the step (c = e_last).
#include <math_constants.h>

#include <algorithm>

#include "fftm_internal.cuh"

namespace fftm {

// Sum `nvals` doubles over `nblocks` rows (fixed order: deterministic).  One warp per column:
// FP64 adds issue at one warp instruction in 16 cycles per SM here, so the sums are arranged
// for few of them (a lane's rows, then five shuffles per column).
__global__ void k_reduce(const double* __restrict__ partial, int nblocks, int nvals, double* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  for (int v = threadIdx.x >> 5; v < nvals; v += blockDim.x >> 5) {
    double s = 0.0;
#pragma unroll 4
    for (int b = lane; b < nblocks; b += 32) s += partial[(size_t)b * nvals + v];
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) out[v] = s;
  }
}

// S_D and S_P over the residual's block partials (rows of two), in one block: NORM_THREADS
// threads read a row at a time, several in flight; valid in thread 0.
constexpr int NORM_THREADS = 256;
__device__ __forceinline__ double2 norm_sums(const double* __restrict__ partial, int nblocks) {
  __shared__ double2 red[NORM_THREADS / 32];
  const double2* rows = reinterpret_cast<const double2*>(partial);
  double2 s = make_double2(0.0, 0.0);
#pragma unroll 8
  for (int b = threadIdx.x; b < nblocks; b += NORM_THREADS) {
    const double2 r = rows[b];
    s.x += r.x;
    s.y += r.y;
  }
  const int lane = threadIdx.x & 31;
  for (int off = 16; off > 0; off >>= 1) {
    s.x += __shfl_xor_sync(0xffffffffu, s.x, off);
    s.y += __shfl_xor_sync(0xffffffffu, s.y, off);
  }
  if (lane == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0)
    for (int w = 1; w < NORM_THREADS / 32; ++w) {
      s.x += red[w].x;
      s.y += red[w].y;
    }
  return s;
}

// err = h1 sqrt(S_D / S_P) (Eq. equilibrium_condition; +inf while S_P is 0 under a non-zero S_D)
__device__ __forceinline__ double norm_error(double2 s, double h1) {
  return s.y > 0.0 ? h1 * sqrt(s.x / s.y) : (s.x == 0.0 ? 0.0 : CUDART_INF);
}

// sums[0..1] = S_D, S_P and, with err_too, sums[2] = err
__global__ void __launch_bounds__(NORM_THREADS) k_norms(const double* __restrict__ partial, int nblocks,
                                                        double* __restrict__ sums, int err_too, double h1,
                                                        const int* __restrict__ stop) {
  if (stop && *stop) return;
  const double2 s = norm_sums(partial, nblocks);
  if (threadIdx.x != 0) return;
  sums[0] = s.x;
  sums[1] = s.y;
  if (err_too) sums[2] = norm_error(s, h1);
}

cudaError_t launch_norms(const double* partial, int nblocks, double* sums, bool err_too, double h1, cudaStream_t s,
                         const int* stop) {
  k_norms<<<1, NORM_THREADS, 0, s>>>(partial, nblocks, sums, err_too ? 1 : 0, h1, stop);
  return cudaGetLastError();
}

cudaError_t launch_reduce_sums(const double* partial, int nblocks, int nvals, double* out, cudaStream_t s) {
  k_reduce<<<1, 32 * (nvals < 32 ? nvals : 32), 0, s>>>(partial, nblocks, nvals, out);
  return cudaGetLastError();
}

// The norms and the convergence test of Algorithm 1 on the device, in one launch (the sum of
// the partials and the test were two: 10 + 4 us per iteration, now 5-8 with the same sums): err
// (Eq. equilibrium_condition; +inf only means "not yet") is recorded at err_hist[m]; the step
// stops when err < tol (1), on a non-finite norm (2) or at the iteration limit (3), else the
// next iteration is m + 1.
__global__ void __launch_bounds__(NORM_THREADS) k_check(const double* __restrict__ partial, int nblocks,
                                                        double* __restrict__ sums, int* __restrict__ ctl,
                                                        double* __restrict__ err_hist, double tol, int max_iter,
                                                        double h1) {
  if (ctl[0]) return;
  const double2 s = norm_sums(partial, nblocks);
  if (threadIdx.x != 0) return;
  const int m = ctl[1];
  const double err = norm_error(s, h1);
  sums[0] = s.x;
  sums[1] = s.y;
  err_hist[m] = err;
  ctl[2] = m;
  if (isnan(err) || isinf(s.x) || isinf(s.y) || isnan(s.x) || isnan(s.y)) ctl[0] = 2;
  else if (err < tol) ctl[0] = 1;
  else if (m >= max_iter) ctl[0] = 3;
  else ctl[1] = m + 1;
}

cudaError_t launch_check(const double* partial, int nblocks, double* sums, int* ctl, double* err_hist, double tol,
                         int max_iter, double h1, cudaStream_t s) {
  k_check<<<1, NORM_THREADS, 0, s>>>(partial, nblocks, sums, ctl, err_hist, tol, max_iter, h1);
  return cudaGetLastError();
}

template <typename T>
__global__ void k_copy(T* d0, T* d1, T* d2, const T* s0, const T* s1, const T* s2, long long count) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
       i += (long long)gridDim.x * blockDim.x) {
    d0[i] = s0[i];
    d1[i] = s1[i];
    d2[i] = s2[i];
  }
}

template <typename T>
cudaError_t launch_copy_fields(T* const dst[3], const T* const src[3], long long count, cudaStream_t s) {
  k_copy<T><<<152 * 8, 256, 0, s>>>(dst[0], dst[1], dst[2], src[0], src[1], src[2], count);
  return cudaGetLastError();
}

template <typename T>
__global__ void k_axpy(T* d0, T* d1, T* d2, const T* a0, const T* a1, const T* a2, const T* b0, const T* b1,
                       const T* b2, T alpha, long long count) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
       i += (long long)gridDim.x * blockDim.x) {
    d0[i] = a0[i] + alpha * b0[i];
    d1[i] = a1[i] + alpha * b1[i];
    d2[i] = a2[i] + alpha * b2[i];
  }
}

template <typename T>
cudaError_t launch_axpy_fields(T* const dst[3], const T* const a[3], const T* const b[3], T alpha, long long count,
                               cudaStream_t s) {
  k_axpy<T><<<152 * 8, 256, 0, s>>>(dst[0], dst[1], dst[2], a[0], a[1], a[2], b[0], b[1], b[2], alpha, count);
  return cudaGetLastError();
}

// Four blocks per SM, and no more than one element per thread needs: a block ends with 9 FP64
// warp sums whatever it read (at 32^3 608 blocks took 22 us, 148 take 16).
int gram_blocks(long long count) { return (int)std::min<long long>(152 * 4, (count + 255) / 256); }

// Normal matrix of the residual differences d_k = D_k - D_last (k < last) and
// the right-hand side <d_k, D_last>, formed from explicit differences (no
// Gram-entry cancellation) and reduced in FP64 across threads and blocks.
template <typename T>
struct GramArgs {
  const T* D[4][3];
};

// Accumulator of a sum of products: FP64 for double data; for float data an unevaluated pair
// (hi, lo) of floats updated with error-free transformations (TwoProduct through fma, TwoSum),
// which keeps about twice FP32's precision without the FP64 pipe (whose rate is a small fraction of
// FP32's on this GPU).  Float data go two neighbouring nodes at a time in packed FP32x2
// instructions, each with its own pair: ten instructions for two products.  256^3, four sets: 249 ->
// 200 us (the reads alone 120); 128^3 58 -> 56.
template <typename T>
struct DotAcc;
template <>
struct DotAcc<double> {
  using V = double;  // a thread's nodes of one step
  double s = 0.0;
  __device__ __forceinline__ void add(double a, double b) { s += a * b; }
  __device__ __forceinline__ double value() const { return s; }
};
template <>
struct DotAcc<float> {
  using V = float2;
  float2 hi = {0.f, 0.f}, lo = {0.f, 0.f};
  static __device__ __forceinline__ float2 sub(float2 a, float2 b) {
    return __ffma2_rn(b, make_float2(-1.f, -1.f), a);
  }
  __device__ __forceinline__ void add(float2 a, float2 b) {
    const float2 p = __fmul2_rn(a, b);
    const float2 pe = __ffma2_rn(a, b, make_float2(-p.x, -p.y));  // exact error of the product
    const float2 s = __fadd2_rn(hi, p);
    const float2 bb = sub(s, hi);
    const float2 se = __fadd2_rn(sub(hi, sub(s, bb)), sub(p, bb));  // exact error of the sum
    hi = s;
    lo = __fadd2_rn(lo, __fadd2_rn(se, pe));
  }
  __device__ __forceinline__ double value() const {
    return ((double)hi.x + (double)lo.x) + ((double)hi.y + (double)lo.y);
  }
};
__device__ __forceinline__ double v_sub(double a, double b) { return a - b; }
__device__ __forceinline__ float2 v_sub(float2 a, float2 b) { return DotAcc<float>::sub(a, b); }

// (four resident blocks: 64 registers of FP32 accumulators and loads, of which the instance for four
// sets spills 132 bytes a thread; two to three blocks leave too few loads in flight, 265 us, five spill
// more, 421 us)
template <typename T, int M>
__global__ void __launch_bounds__(256, 4) k_gram(GramArgs<T> A, long long count, double* __restrict__ partial,
                                              const int* __restrict__ stop) {
  if (stop && *stop) return;
  using V = typename DotAcc<T>::V;
  constexpr int L = M - 1, W = sizeof(V) / sizeof(T);
  __shared__ double red[8][9];
  DotAcc<T> acc[9];
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i * W < count;
       i += (long long)gridDim.x * blockDim.x) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      V v[M], d[3];
#pragma unroll
      for (int j = 0; j < M; ++j) v[j] = reinterpret_cast<const V*>(A.D[j][c])[i];
#pragma unroll
      for (int j = 0; j < L; ++j) d[j] = v_sub(v[j], v[L]);
      int k = 0;
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = a; b < 3; ++b, ++k)
          if (b < L) acc[k].add(d[a], d[b]);
#pragma unroll
      for (int a = 0; a < L; ++a) acc[6 + a].add(d[a], v[L]);
    }
  }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    double v = acc[k].value();
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if (l == 0) red[w][k] = v;
  }
  __syncthreads();
  if (threadIdx.x < 9) {
    double t = 0.0;
    for (int i = 0; i < 8; ++i) t += red[i][threadIdx.x];
    partial[(size_t)blockIdx.x * 9 + threadIdx.x] = t;
  }
}

// (a component, its padding included, is a multiple of 64 elements and starts at one: count is even
// and pairs of nodes are aligned)
template <typename T>
cudaError_t launch_gram(const T* const D[4][3], int m, long long count, double* partial, int nblocks,
                        cudaStream_t s, const int* stop) {
  GramArgs<T> A;
  for (int j = 0; j < 4; ++j)
    for (int c = 0; c < 3; ++c) A.D[j][c] = (j < m) ? D[j][c] : D[0][c];
  if (m <= 1) k_gram<T, 1><<<nblocks, 256, 0, s>>>(A, count, partial, stop);
  else if (m == 2) k_gram<T, 2><<<nblocks, 256, 0, s>>>(A, count, partial, stop);
  else if (m == 3) k_gram<T, 3><<<nblocks, 256, 0, s>>>(A, count, partial, stop);
  else k_gram<T, 4><<<nblocks, 256, 0, s>>>(A, count, partial, stop);
  return cudaGetLastError();
}

// Reduce the partials (one warp per sum, its rows in flight together: a single warp that walked
// them in a chain of dependent loads took 49-57 us at any grid size, this takes 12-13); solve
// (d^T d) gamma = -(d^T D_last) by Cholesky in FP64;
// c_k = gamma_k (k < last), c_last = 1 - sum gamma.  A pivot below pivot_tol
// times its diagonal entry rejects the step: c = e_last.
__global__ void __launch_bounds__(288) k_anderson_solve(const double* __restrict__ partial, int nblocks, int m,
                                                        double pivot_tol, double* __restrict__ coef,
                                                        int* __restrict__ accepted, const int* __restrict__ ctl) {
  if (ctl && ctl[0]) return;
  if (ctl) accepted += ctl[2];
  __shared__ double g[9];
  {
    const int v = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double t = 0.0;
#pragma unroll 8
    for (int b = lane; b < nblocks; b += 32) t += partial[(size_t)b * 9 + v];
    for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
    if (lane == 0) g[v] = t;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  const double A[3][3] = {{g[0], g[1], g[2]}, {g[1], g[3], g[4]}, {g[2], g[4], g[5]}};
  const double rhs[3] = {-g[6], -g[7], -g[8]};
  const int d = m - 1;
  double Lc[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
  bool ok = d > 0;
  for (int c = 0; c < d && ok; ++c) {
    double s = A[c][c];
    for (int j = 0; j < c; ++j) s -= Lc[c][j] * Lc[c][j];
    if (!(A[c][c] > 0.0) || !(s > pivot_tol * A[c][c])) {
      ok = false;
      break;
    }
    Lc[c][c] = sqrt(s);
    for (int i = c + 1; i < d; ++i) {
      double t = A[i][c];
      for (int j = 0; j < c; ++j) t -= Lc[i][j] * Lc[c][j];
      Lc[i][c] = t / Lc[c][c];
    }
  }
  double cf[4] = {0.0, 0.0, 0.0, 0.0};
  if (ok) {
    double y[3] = {0, 0, 0}, gam[3] = {0, 0, 0};
    for (int i = 0; i < d; ++i) {
      double t = rhs[i];
      for (int j = 0; j < i; ++j) t -= Lc[i][j] * y[j];
      y[i] = t / Lc[i][i];
    }
    for (int i = d - 1; i >= 0; --i) {
      double t = y[i];
      for (int j = i + 1; j < d; ++j) t -= Lc[j][i] * gam[j];
      gam[i] = t / Lc[i][i];
    }
    double sum = 0.0;
    for (int i = 0; i < d; ++i) {
      cf[i] = gam[i];
      sum += gam[i];
    }
    cf[d] = 1.0 - sum;
  } else {
    cf[d] = 1.0;
  }
  for (int i = 0; i < 4; ++i) coef[i] = cf[i];
  *accepted = ok ? 1 : 0;
}

cudaError_t launch_anderson_solve(const double* partial, int nblocks, int m, double pivot_tol, double* coef,
                                  int* accepted, cudaStream_t s, const int* ctl) {
  k_anderson_solve<<<1, 288, 0, s>>>(partial, nblocks, m, pivot_tol, coef, accepted, ctl);
  return cudaGetLastError();
}

template <typename T>
struct CombArgs {
  T* dst[3];
  T* bh[3];
  T* bl[3];
  const T* D[4][3];
  const T* uh[4][3];
  const T* ul[4][3];
};

// Dbar = sum_k c_k D_k; ubar = u_last + sum_{k<last} c_k (u_k - u_last) (the
// differences of nearby iterates are formed first, then added to u_last with
// an error-free sum when the low parts are present).  Every operand of an element is
// loaded before the first store, so that the loads of all three components are in
// flight together (the output arrays may alias nothing the compiler can see).
template <typename T, bool LO>
__global__ void k_combine(CombArgs<T> A, int m, const double* __restrict__ coef, long long count,
                          const int* __restrict__ stop) {
  if (stop && *stop) return;
  T c[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) c[j] = (j < m) ? (T)coef[j] : T(0);
  const int L = m - 1;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
       i += (long long)gridDim.x * blockDim.x) {
    T Dv[3][4], Uh[3][4], Ul[3][4];
#pragma unroll
    for (int q = 0; q < 3; ++q)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        Dv[q][j] = (j < m) ? __ldg(A.D[j][q] + i) : T(0);
        Uh[q][j] = (j < m) ? __ldg(A.uh[j][q] + i) : T(0);
        Ul[q][j] = (LO && j < m) ? __ldg(A.ul[j][q] + i) : T(0);
      }
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      T s = T(0);
#pragma unroll
      for (int j = 0; j < 4; ++j) s += c[j] * Dv[q][j];
      T uL = Uh[q][0], lL = Ul[q][0];
#pragma unroll
      for (int j = 1; j < 4; ++j)
        if (j == L) {
          uL = Uh[q][j];
          lL = Ul[q][j];
        }
      T corr = T(0);
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        if (j < L) {
          T dj = Uh[q][j] - uL;
          if (LO) dj += Ul[q][j] - lL;
          corr += c[j] * dj;
        }
      }
      A.dst[q][i] = s;
      if (LO) {
        const T s1 = uL + corr;
        const T bb = s1 - uL;
        const T e = (uL - (s1 - bb)) + (corr - bb);
        const T t = lL + e;
        const T h = s1 + t;
        A.bh[q][i] = h;
        A.bl[q][i] = t - (h - s1);
      } else {
        A.bh[q][i] = uL + corr;
      }
    }
  }
}

template <typename T>
cudaError_t launch_combine(T* const dst[3], T* const bh[3], T* const bl[3], const T* const D[4][3],
                           const T* const uh[4][3], const T* const ul[4][3], int m, const double* coef,
                           long long count, cudaStream_t s, const int* stop) {
  CombArgs<T> A;
  const bool lo = bl != nullptr && bl[0] != nullptr;
  for (int q = 0; q < 3; ++q) {
    A.dst[q] = dst[q];
    A.bh[q] = bh[q];
    A.bl[q] = lo ? bl[q] : nullptr;
    for (int j = 0; j < 4; ++j) {
      const int jj = j < m ? j : 0;
      A.D[j][q] = D[jj][q];
      A.uh[j][q] = uh[jj][q];
      A.ul[j][q] = lo ? ul[jj][q] : nullptr;
    }
  }
  if (lo) k_combine<T, true><<<152 * 8, 256, 0, s>>>(A, m, coef, count, stop);
  else k_combine<T, false><<<152 * 8, 256, 0, s>>>(A, m, coef, count, stop);
  return cudaGetLastError();
}

// ---- arithmetic peak probe --------------------------------------------------------------
// Eight independent chains of fused multiply-adds per thread (enough to cover the FMA
// latency), `iters` rounds; the result is written so the chains are not removed.
template <typename T>
__global__ void __launch_bounds__(256) k_fma_peak(T* __restrict__ sink, int iters, T a, T b) {
  T x[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) x[k] = T(threadIdx.x + k) * T(1e-3);
  for (int i = 0; i < iters; ++i) {
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = x[k] * a + b;
  }
  T t = T(0);
#pragma unroll
  for (int k = 0; k < 8; ++k) t += x[k];
  if (t == T(-1.2345)) sink[blockIdx.x] = t;  // practically never: keeps the chains live
}

double fma_peak_flops(int fp64) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return -1.0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int blocks = (sms > 0 ? sms : 152) * 8, threads = 256;
  const int iters = fp64 ? 4096 : 65536;
  void* sink = nullptr;
  if (cudaMalloc(&sink, blocks * sizeof(double)) != cudaSuccess) return -1.0;
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  double best = -1.0;
  for (int rep = 0; rep < 4; ++rep) {
    cudaEventRecord(e0, 0);
    if (fp64) k_fma_peak<double><<<blocks, threads>>>((double*)sink, iters, 0.999999, 1e-7);
    else k_fma_peak<float><<<blocks, threads>>>((float*)sink, iters, 0.999999f, 1e-7f);
    cudaEventRecord(e1, 0);
    cudaEventSynchronize(e1);
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess && ms > 0.f && rep > 0) {
      const double flops = 2.0 * 8.0 * (double)iters * blocks * threads / (ms * 1e-3);
      if (flops > best) best = flops;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaFree(sink);
  return cudaGetLastError() == cudaSuccess ? best : -1.0;
}

// Dense [q][z][y][x] <-> pitched component arrays.  A warp copies a row (one division per row:
// an index decomposition per element cost 64-bit divisions and ran at 0.2 of the copy rate,
// 292 us for the FP32 node field of a 256^3 grid), PACK_UNROLL elements a lane in flight.  When
// writing the component arrays, elements outside the node range [lo, hi) are stored as zero.
template <typename T>
struct PackArgs {
  T* f[3];
  T* dense;
  int N1, N2, N3;
  long long sy, sz;
  int lo[3][3], hi[3][3];
};
constexpr int PACK_UNROLL = 4, PACK_WARPS = 8;

template <typename T, bool UNPACK>
__global__ void __launch_bounds__(32 * PACK_WARPS) k_pack(PackArgs<T> A) {
  const int lane = threadIdx.x & 31;
  const int rows = A.N2 * A.N3;
  for (int r = blockIdx.x * PACK_WARPS + (threadIdx.x >> 5); r < 3 * rows; r += gridDim.x * PACK_WARPS) {
    const int q = r >= 2 * rows ? 2 : (r >= rows ? 1 : 0);
    const int z = (r - q * rows) / A.N2, y = r - q * rows - z * A.N2;
    T* f = (q == 0 ? A.f[0] : (q == 1 ? A.f[1] : A.f[2])) + y * A.sy + z * A.sz;
    T* d = A.dense + (long long)r * A.N1;
    int x_lo = 0, x_hi = A.N1;
    if (UNPACK) {
      const bool in = y >= A.lo[q][1] && y < A.hi[q][1] && z >= A.lo[q][2] && z < A.hi[q][2];
      x_lo = A.lo[q][0];
      x_hi = in ? A.hi[q][0] : 0;
    }
    for (int x0 = lane; x0 < A.N1; x0 += 32 * PACK_UNROLL) {
      T v[PACK_UNROLL];
#pragma unroll
      for (int k = 0; k < PACK_UNROLL; ++k) {
        const int x = x0 + 32 * k;
        v[k] = T(0);
        if (UNPACK ? (x >= x_lo && x < x_hi) : x < A.N1) v[k] = UNPACK ? d[x] : f[x];
      }
#pragma unroll
      for (int k = 0; k < PACK_UNROLL; ++k) {
        const int x = x0 + 32 * k;
        if (x < A.N1) (UNPACK ? f : d)[x] = v[k];
      }
    }
  }
}

template <typename T>
static cudaError_t launch_pack_args(const PackArgs<T>& A, bool unpack, cudaStream_t s) {
  const long long rows = 3LL * A.N2 * A.N3;
  const int blocks = (int)std::min<long long>(152 * 8, (rows + PACK_WARPS - 1) / PACK_WARPS);
  if (unpack) k_pack<T, true><<<blocks, 32 * PACK_WARPS, 0, s>>>(A);
  else k_pack<T, false><<<blocks, 32 * PACK_WARPS, 0, s>>>(A);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_pack(const T* const src[3], T* dense, int N1, int N2, int N3, long long sy, long long sz,
                        cudaStream_t s) {
  PackArgs<T> A = {};
  for (int q = 0; q < 3; ++q) A.f[q] = const_cast<T*>(src[q]);
  A.dense = dense;
  A.N1 = N1; A.N2 = N2; A.N3 = N3;
  A.sy = sy; A.sz = sz;
  return launch_pack_args<T>(A, false, s);
}

template <typename T>
cudaError_t launch_unpack(T* const dst[3], const T* dense, int N1, int N2, int N3, long long sy, long long sz,
                          const int (*lo)[3], const int (*hi)[3], cudaStream_t s) {
  PackArgs<T> A = {};
  const int N[3] = {N1, N2, N3};
  for (int q = 0; q < 3; ++q) {
    A.f[q] = dst[q];
    for (int a = 0; a < 3; ++a) {
      A.lo[q][a] = lo ? lo[q][a] : 0;
      A.hi[q][a] = hi ? hi[q][a] : N[a];
    }
  }
  A.dense = const_cast<T*>(dense);
  A.N1 = N1; A.N2 = N2; A.N3 = N3;
  A.sy = sy; A.sz = sz;
  return launch_pack_args<T>(A, true, s);
}

#define FFTM_INST(T)                                                                                               \
  template cudaError_t launch_copy_fields<T>(T* const[3], const T* const[3], long long, cudaStream_t);            \
  template cudaError_t launch_axpy_fields<T>(T* const[3], const T* const[3], const T* const[3], T, long long,     \
                                             cudaStream_t);                                                        \
  template cudaError_t launch_gram<T>(const T* const[4][3], int, long long, double*, int, cudaStream_t,           \
                                      const int*);                                                                 \
  template cudaError_t launch_combine<T>(T* const[3], T* const[3], T* const[3], const T* const[4][3],             \
                                         const T* const[4][3], const T* const[4][3], int, const double*,          \
                                         long long, cudaStream_t, const int*);                                     \
  template cudaError_t launch_pack<T>(const T* const[3], T*, int, int, int, long long, long long, cudaStream_t);   \
  template cudaError_t launch_unpack<T>(T* const[3], const T*, int, int, int, long long, long long,               \
                                        const int (*)[3], const int (*)[3], cudaStream_t);
FFTM_INST(float)
FFTM_INST(double)

}  // namespace fftm
