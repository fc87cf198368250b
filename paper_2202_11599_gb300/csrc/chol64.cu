// FP64 Cholesky factor of an s x s matrix and the product with its inverse (CholQR2, C = chol(Om^T
// Y_nu), B = Y_nu C^{-1} of App. B, and the start of the eigensolve).
//
// One SM's FP64 pipe (2 FMA per clock) needs 0.33 ms for the s^3 / 6 FMAs of s = 200 and took 0.68
// with one barrier-separated step per column.  Here the columns lie cyclically over the eight
// CTAs of a cluster, in shared memory.  The owner of column j + 1 updates it with column j first,
// scales it and writes it into every CTA's buffer through distributed shared memory before the
// rest of step j's update is done, so a step costs its own latency (the cluster barrier, one
// reciprocal square root) and the updates run behind it: 0.24 ms at s = 200.
#include <cooperative_groups.h>

#include <algorithm>

#include "device_util.cuh"
#include "nys_internal.cuh"

namespace nys {
namespace {
namespace cg = cooperative_groups;

constexpr int kCholCtas = 8;
constexpr int kCholThreads = 256;
constexpr int kCholMax = 448;   // 56 columns of 448 and three buffers: 211 KB of shared memory

struct CholArgs {
  const double* M;   // s x s column-major, symmetrised as (M + M^T) / 2
  int s;
  double rel_tol;    // a pivot not above rel_tol max |M_ii| is refused
  double ridge;      // ridge trace(M) is added to the diagonal
  double* C;         // upper factor, C^T C = M (lower part zeroed), or null; may be M
  float* L;          // N x N FP32 lower factor of M 2^-ex (largest diagonal in [1/2, 2)), rows and
  int N;             // columns from s on: sqrt of the ridge on the diagonal; or null
  int* info;         // 0, or k + 1 when the k-th pivot is not positive, not finite or refused
};

__global__ void __launch_bounds__(kCholThreads) chol_cluster_kernel(const CholArgs a) {
  extern __shared__ __align__(16) double sm[];
  __shared__ double s_diag[2], s_r;
  __shared__ int s_bad[3];
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int s = a.s, nown = (s + kCholCtas - 1) / kCholCtas;
  double* cols = sm;                    // [own column q][row]: global column 8 q + rank
  double* lb = sm + (size_t)nown * s;   // [3][s]: scaled columns j, j - 1, j - 2
  if (warp == 0) {
    double mx = 0.0, tr = 0.0;
    for (int i = lane; i < s; i += 32) {
      const double g = a.M[i + (int64_t)i * s];
      mx = fmax(mx, fabs(g));
      tr += g;
    }
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    tr = warp_sum(tr);
    if (lane == 0) {
      s_diag[0] = mx;
      s_diag[1] = tr;
    }
  }
  if (tid < 3) s_bad[tid] = 0;
  __syncthreads();
  const double thresh = a.rel_tol * s_diag[0], ridge = a.ridge * s_diag[1];
  for (int q = warp; q < nown; q += kCholThreads / 32) {
    const int c = q * kCholCtas + rank;
    if (c < s)
      for (int i = c + lane; i < s; i += 32)
        cols[q * s + i] = i == c ? a.M[c + (int64_t)c * s] + ridge
                                 : 0.5 * (a.M[i + (int64_t)c * s] + a.M[c + (int64_t)i * s]);
  }
  cl.sync();
  // scale own column j and hand it to every CTA (all threads of the owner)
  auto finish = [&](int j) {
    double* col = cols + (size_t)(j / kCholCtas) * s;
    if (warp == 0) {
      const double d = col[j];
      const bool ok = d > 0.0 && d > thresh && isfinite(d);
      const double r = ok ? rsqrt(d) : 0.0;
      if (lane == 0) {
        s_r = r;
        if (!ok)
          for (int t = 0; t < kCholCtas; ++t) cl.map_shared_rank(s_bad, t)[j % 3] = 1;
      }
    }
    __syncthreads();
    const double r = s_r;
    for (int i = j + tid; i < s; i += kCholThreads) {
      const double l = col[i] * r;
      col[i] = l;
#pragma unroll
      for (int t = 0; t < kCholCtas; ++t) cl.map_shared_rank(lb, t)[(j % 3) * s + i] = l;
    }
  };
  auto arrive = [] { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); };
  auto wait = [] { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); };
  if (rank == 0) finish(0);
  __syncthreads();
  arrive();
  wait();
  int bad = 0;
  for (int j = 0; j < s; ++j) {
    if (*(volatile int*)&s_bad[j % 3]) {
      bad = j + 1;
      break;
    }
    if (j + 1 == s) break;
    const double* l = lb + (j % 3) * s;
    const bool next_here = (j + 1) % kCholCtas == rank;
    if (next_here) {
      double* col = cols + (size_t)((j + 1) / kCholCtas) * s;
      const double f = l[j + 1];
      for (int i = j + 1 + tid; i < s; i += kCholThreads) col[i] = fma(-f, l[i], col[i]);
      __syncthreads();
      finish(j + 1);
      __syncthreads();
    }
    // buffer (j + 2) % 3 is next written in step j + 1, after every CTA has arrived here and so
    // has read column j - 1 out of it
    arrive();
    // own columns c > j (c = j + 1 is done): first own index past j (+ 1)
    const int first = j + 1 + (next_here ? 1 : 0);
    const int q0 = (first - rank + kCholCtas - 1) / kCholCtas;
    for (int q = q0 + warp; q < nown; q += kCholThreads / 32) {
      const int c = q * kCholCtas + rank;
      if (c < s) {
        double* col = cols + (size_t)q * s;
        const double f = l[c];
        for (int i = c + lane; i < s; i += 32) col[i] = fma(-f, l[i], col[i]);
      }
    }
    __syncthreads();
    wait();
  }
  if (rank == 0 && tid == 0 && a.info) *a.info = bad;
  if (a.C) {
    for (int q = warp; q < nown; q += kCholThreads / 32) {
      const int c = q * kCholCtas + rank;
      if (c < s)
        for (int i = lane; i < s; i += 32) {
          if (i >= c) a.C[c + (int64_t)i * s] = cols[q * s + i];
          else a.C[c + (int64_t)i * s] = 0.0;
        }
    }
  }
  if (a.L) {
    // 4^k within a factor of four of the largest diagonal: L scales by 2^-k exactly
    int ex = 0;
    const bool plain = bad == 0 && s_diag[0] > 0.0 && isfinite(s_diag[0]) && isfinite(s_diag[1]);
    if (plain) frexp(s_diag[0], &ex);
    const int k = ex >> 1;
    for (int q = warp; q * kCholCtas + rank < a.N; q += kCholThreads / 32) {
      const int c = q * kCholCtas + rank;
      for (int i = lane; i < a.N; i += 32) {
        float v = 0.f;
        if (plain) {
          if (c >= s || i >= s) v = i == c ? (float)scalbn(sqrt(ridge), -k) : 0.f;
          else if (i >= c) v = (float)scalbn(cols[q * s + i], -k);
        }
        a.L[i + (int64_t)c * a.N] = v;
      }
    }
  }
  cl.sync();   // no CTA leaves while another may still write to it
}

cudaError_t launch_chol(const CholArgs& a, cudaStream_t st) {
  const int nown = (a.s + kCholCtas - 1) / kCholCtas;
  const size_t smem = ((size_t)nown * a.s + 3 * (size_t)a.s) * sizeof(double);
  NYS_CUDA_TRY(ensure_max_dyn_smem((const void*)chol_cluster_kernel, 212 * 1024));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kCholCtas);
  cfg.blockDim = dim3(kCholThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kCholCtas;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  count_launch();
  return cudaLaunchKernelEx(&cfg, chol_cluster_kernel, a);
}

// Single CTA, matrix in global memory: the form for s beyond kCholMax.
__global__ void __launch_bounds__(1024) chol_upper_kernel(double* M, int s, int* info, double rel_tol) {
  const int tid = threadIdx.x, T = blockDim.x;
  const int warp = tid >> 5, lane = tid & 31, nwarp = T >> 5;
  __shared__ int bad;
  __shared__ double thresh;
  for (int j = warp; j < s; j += nwarp)
    for (int i = lane; i < j; i += 32) M[i + (int64_t)j * s] = 0.5 * (M[i + (int64_t)j * s] + M[j + (int64_t)i * s]);
  if (tid == 0) {
    bad = 0;
    double mx = 0.0;
    for (int j = 0; j < s; ++j) mx = fmax(mx, fabs(M[j + (int64_t)j * s]));
    thresh = rel_tol * mx;
  }
  __syncthreads();
  for (int j = 0; j < s; ++j) {
    if (tid == 0) {
      const double dj = M[j + (int64_t)j * s];
      if (!(dj > 0.0) || !(dj > thresh) || !isfinite(dj)) {
        bad = j + 1;
      } else {
        M[j + (int64_t)j * s] = sqrt(dj);
      }
    }
    __syncthreads();
    if (bad) break;
    const double piv = M[j + (int64_t)j * s];
    for (int c = j + 1 + tid; c < s; c += T) M[j + (int64_t)c * s] /= piv;
    __syncthreads();
    // trailing update of the upper triangle: M[i][c] -= C[j][i] C[j][c], j < i <= c
    // (warps over columns c, lanes over rows i: no index division in the inner loop)
    for (int c = j + 1 + warp; c < s; c += nwarp) {
      const double rc = M[j + (int64_t)c * s];
      double* col = M + (int64_t)c * s;
      for (int i = j + 1 + lane; i <= c; i += 32) col[i] -= M[j + (int64_t)i * s] * rc;
    }
    __syncthreads();
  }
  if (tid == 0) *info = bad;
  // zero the strict lower triangle
  for (int j = warp; j < s; j += nwarp)
    for (int i = j + 1 + lane; i < s; i += 32) M[i + (int64_t)j * s] = 0.0;
}

__device__ __forceinline__ double pow2(int e) { return __hiloint2double((e + 1023) << 20, 0); }   // |e| < 1023

// X = C^{-1} for an upper triangular C (both s x s column-major): warp c solves C x = e_c from the
// last row up, column by column of C (the next column's entries are loaded a step ahead).
constexpr int kInvAhead = 8;   // entries of a column a lane holds: 256 rows; more are read in place
// Row i of the result is scaled by 2^t_i.
__global__ void __launch_bounds__(32) tri_inverse_kernel(const double* __restrict__ C, int s, const int* __restrict__ t,
                                                         double* __restrict__ X) {
  extern __shared__ double y[];
  const int c = s - 1 - (int)blockIdx.x;   // the longest solves first
  const int lane = threadIdx.x;
  double* ri = y + s;
  for (int i = lane; i < s; i += 32) {
    y[i] = i == c ? 1.0 : 0.0;
    ri[i] = i <= c ? 1.0 / C[i + (int64_t)i * s] : 0.0;
  }
  double nx[kInvAhead];
  auto fetch = [&](int k) {
#pragma unroll
    for (int q = 0; q < kInvAhead; ++q) {
      const int i = lane + 32 * q;
      nx[q] = k >= 0 && i < k ? __ldg(C + i + (int64_t)k * s) : 0.0;
    }
  };
  fetch(c);
  __syncwarp();
  for (int k = c; k >= 0; --k) {
    const double xk = y[k] * ri[k];
    double cur[kInvAhead];
#pragma unroll
    for (int q = 0; q < kInvAhead; ++q) cur[q] = nx[q];
    fetch(k - 1);
#pragma unroll
    for (int q = 0; q < kInvAhead; ++q) {
      const int i = lane + 32 * q;
      if (32 * q < k && i < k) y[i] = fma(-cur[q], xk, y[i]);
    }
    for (int i = lane + 32 * kInvAhead; i < k; i += 32) y[i] = fma(-__ldg(C + i + (int64_t)k * s), xk, y[i]);
    __syncwarp();
    if (lane == 0) y[k] = xk;
    __syncwarp();
  }
  for (int i = lane; i < s; i += 32) X[i + (int64_t)c * s] = i <= c ? y[i] * pow2(t[i]) : 0.0;
}

// T(:, k) = 2^-t_k Y(:, k) (d x s), t_k the exponent of the largest entry of C's column k; block (rows, k).
__global__ void __launch_bounds__(256) scale_columns_kernel(const double* __restrict__ C, int s, const double* __restrict__ Y,
                                                            int64_t d, double* __restrict__ T, int* __restrict__ t) {
  __shared__ unsigned top[8];
  const int k = blockIdx.y;
  unsigned h = 0u;
  for (int i = threadIdx.x; i <= k; i += 256) h = max(h, (unsigned)__double2hiint(__ldg(C + i + (int64_t)k * s)) & 0x7fffffffu);
  h = __reduce_max_sync(0xffffffffu, h);
  if ((threadIdx.x & 31) == 0) top[threadIdx.x >> 5] = h;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < 8; ++w) h = max(h, top[w]);
  const int e = min(max((int)(h >> 20) - 1023, -1000), 1000);
  if (blockIdx.x == 0 && threadIdx.x == 0) t[k] = e;
  const double f = pow2(-e);
  const int64_t base = (int64_t)k * d;
  for (int64_t i = blockIdx.x * 256ll + threadIdx.x; i < d; i += gridDim.x * 256ll) T[base + i] = Y[base + i] * f;
}

size_t up256(size_t b) { return (b + 255) / 256 * 256; }

}  // namespace

cudaError_t chol_upper(double* M, int s, int* info, cudaStream_t st, double rel_tol) {
  if (s <= kCholMax) {
    CholArgs a = {};
    a.M = M;
    a.s = s;
    a.rel_tol = rel_tol;
    a.C = M;
    a.info = info;
    return launch_chol(a, st);
  }
  count_launch();
  chol_upper_kernel<<<1, 1024, 0, st>>>(M, s, info, rel_tol);
  return cudaGetLastError();
}

cudaError_t chol_lower_f32(const double* G, int s, double ridge, float* L, int N, cudaStream_t st) {
  if (s > kCholMax) return cudaErrorInvalidValue;
  CholArgs a = {};
  a.M = G;
  a.s = s;
  a.ridge = ridge;
  a.L = L;
  a.N = N;
  return launch_chol(a, st);
}

// ------------------------------------------------------------------ B = Y C^{-1}
// The inverse of the triangular factor, column by column, then one FP64 product on the tensor
// cores.  (Substitution row by row on the FP64 pipe: 0.75 ms at 10,000 x 200;
// the inverse takes 83 us there and the product 55.)  Each column x of
// the computed inverse satisfies |C x - e| <= eps s |C| |x|, so B = Y X has the error bound of
// substitution, B (I + F) with |F| <= eps s |C| |C^{-1}|.  The product's error is relative to the largest
// entries of Y's rows and X's columns, so the columns of Y are brought to one scale first, by powers of two
// that X's rows take up (test matrices and their images need not have columns of one scale).
size_t trsm_work_bytes(int64_t d, int s) {
  return up256((size_t)d * s * sizeof(double)) + up256((size_t)s * s * sizeof(double)) +
         up256((size_t)(d + 2 * s) * sizeof(unsigned)) + gemm64_work_bytes(d, s, s);
}

cudaError_t trsm_right_upper(const double* C, int s, double* Y, int64_t d, void* work, int* status, cudaStream_t st) {
  unsigned char* b = reinterpret_cast<unsigned char*>(work);
  double* T = reinterpret_cast<double*>(b);
  b += up256((size_t)d * s * sizeof(double));
  double* X = reinterpret_cast<double*>(b);
  b += up256((size_t)s * s * sizeof(double));
  unsigned* ed = reinterpret_cast<unsigned*>(b);
  unsigned* ex = ed + d;
  int* t = reinterpret_cast<int*>(ex + s);
  b += up256((size_t)(d + 2 * s) * sizeof(unsigned));
  count_launch();
  scale_columns_kernel<<<dim3((unsigned)std::min<int64_t>(8, (d + 255) / 256), (unsigned)s), 256, 0, st>>>(C, s, Y, d, T, t);
  NYS_CUDA_TRY(cudaGetLastError());
  count_launch();
  tri_inverse_kernel<<<s, 32, 2 * (size_t)s * sizeof(double), st>>>(C, s, t, X);
  NYS_CUDA_TRY(cudaGetLastError());
  NYS_CUDA_TRY(absmax_f64(X, s, s, s, ex, nullptr, st));
  NYS_CUDA_TRY(absmax_f64(T, s, d, d, nullptr, ed, st));
  return gemm64(T, false, d, ed, d, X, s, ex, s, s, nullptr, Y, d, b, status, st, /*any_scale=*/false);
}

}  // namespace nys
