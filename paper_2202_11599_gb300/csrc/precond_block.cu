// P^{-1} on a block of k vectors (Eq. Nystrom preconditioner):
//   Y = V + U diag(c) U^T V,  c_i = (lam_s + rho) / (lam_i + rho) - 1,
// for nys_precond_apply and the multi-RHS PCG.  Three launches for the whole block:
//   1. partials of G = U^T V over chunks of rows,
//   2. G summed over the chunks in a fixed order in FP64, scaled by c and rounded once,
//   3. y_j = v_j + sum_i U_ji g_i as one fma chain in increasing i (the order of the PCG tail).
// The block is read as a matrix, so U (8 MB at 10,000 x 200 FP32, L2-resident) is read once
// per 64 columns instead of once per column: 10,000 x 200, 64 columns FP32 went from 2,713 us
// (four launches per column) to 120 us a call, host side included.
//
// Blocks of more than kSmallCols columns take 64 x 16 or 64 x 64 output tiles; fewer columns
// take a warp per eight rows of U^T (step 1) and a thread per row (step 3), which do no work
// for padded columns -- the FP64 pipe (2 FMA per clock and SM) has none to spare.
#include "device_util.cuh"
#include "solver.cuh"

#include <algorithm>

namespace nys {
namespace {

constexpr int BT_M = 64, BT_K = 16;
constexpr int kSmallCols = 4;
constexpr int kSmallChunk = 256;   // rows of one partial of the small-block form
constexpr int kPairRows = 256;
constexpr int kRowThreads = 64;    // step 3 of the small-block form: rows per CTA

// part[z][c][i] = sum over the rows j of chunk z of U[j, i] V[j, c]; U and V column-major,
// ld d.  Tile 64 (i) x TN (c), 256 threads, 4 x TN / 16 outputs each.  FP32 sums are formed in
// runs of 64 rows; PAIR adds these up as a pair (two-sum), for chunks of more than kPairRows rows: wide
// blocks have chunks of thousands (rank 200, 4,096 columns: all rows in one), whose rounding must
// not grow with their length.
template <typename T, int TN, bool PAIR>
__global__ void __launch_bounds__(256) utv_tile_kernel(const T* __restrict__ U, const T* __restrict__ V, int64_t d,
                                                       int s, int k, int64_t kc, T* __restrict__ part) {
  constexpr int RN = TN / 16;
  __shared__ T As[BT_K][BT_M + 1];
  __shared__ T Bs[BT_K][TN + 1];
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  const int m0 = blockIdx.x * BT_M, n0 = blockIdx.y * TN;
  const int64_t kb = (int64_t)blockIdx.z * kc, ke = min(d, kb + kc);
  const int lk = threadIdx.x % BT_K, lr = threadIdx.x / BT_K;   // load: row of the slab, first column
  T ra[4], rb[RN];
  auto load = [&](int64_t k0) {
    const int64_t j = k0 + lk;
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      const int i = m0 + lr + 16 * l;
      ra[l] = (j < ke && i < s) ? U[j + (int64_t)i * d] : T(0);
    }
#pragma unroll
    for (int l = 0; l < RN; ++l) {
      const int c = n0 + lr + 16 * l;
      rb[l] = (j < ke && c < k) ? V[j + (int64_t)c * d] : T(0);
    }
  };
  T acc[4][RN] = {}, run[4][RN] = {}, low[4][RN] = {};   // low: what the additions to acc rounded off
  load(kb);
  int in_run = 0;
  for (int64_t k0 = kb; k0 < ke; k0 += BT_K) {
#pragma unroll
    for (int l = 0; l < 4; ++l) As[lk][lr + 16 * l] = ra[l];
#pragma unroll
    for (int l = 0; l < RN; ++l) Bs[lk][lr + 16 * l] = rb[l];
    __syncthreads();
    if (k0 + BT_K < ke) load(k0 + BT_K);
#pragma unroll
    for (int kk = 0; kk < BT_K; ++kk) {
      T a[4], b[RN];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][tx + 16 * i];
#pragma unroll
      for (int j = 0; j < RN; ++j) b[j] = Bs[kk][ty + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < RN; ++j) run[i][j] = fma(a[i], b[j], run[i][j]);
    }
    if (++in_run == 4 || k0 + BT_K >= ke) {
      in_run = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < RN; ++j) {
          if constexpr (PAIR) {
            const T t = acc[i][j] + run[i][j], z = t - acc[i][j];
            low[i][j] += (acc[i][j] - (t - z)) + (run[i][j] - z);
            acc[i][j] = t;
          } else {
            acc[i][j] += run[i][j];
          }
          run[i][j] = T(0);
        }
    }
    __syncthreads();
  }
  T* out = part + (int64_t)blockIdx.z * k * s;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < RN; ++j) {
      const int m = m0 + tx + 16 * i, c = n0 + ty + 16 * j;
      // (a sum that overflowed has no low part)
      if (m < s && c < k) out[(int64_t)c * s + m] = PAIR && isfinite(acc[i][j]) ? acc[i][j] + low[i][j] : acc[i][j];
    }
}

// The same partials for TN <= 4 columns: warp w of CTA (z, y) takes rows i = 64 y + 8 w .. + 7
// of U^T over chunk z, lanes over the chunk's rows.
template <typename T, int TN>
__global__ void __launch_bounds__(256) utv_small_kernel(const T* __restrict__ U, const T* __restrict__ V, int64_t d,
                                                        int s, int k, T* __restrict__ part) {
  constexpr int RW = 8;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t j0 = (int64_t)blockIdx.x * kSmallChunk, j1 = min(d, j0 + kSmallChunk);
  const int i0 = blockIdx.y * 64 + warp * RW;
  if (i0 >= s) return;
  T acc[RW][TN] = {};
  for (int64_t j = j0 + lane; j < j1; j += 32) {
    T v[TN];
#pragma unroll
    for (int c = 0; c < TN; ++c) v[c] = c < k ? V[j + (int64_t)c * d] : T(0);
#pragma unroll
    for (int q = 0; q < RW; ++q) {
      const T u = i0 + q < s ? U[j + (int64_t)(i0 + q) * d] : T(0);
#pragma unroll
      for (int c = 0; c < TN; ++c) acc[q][c] = fma(u, v[c], acc[q][c]);
    }
  }
#pragma unroll
  for (int q = 0; q < RW; ++q)
#pragma unroll
    for (int c = 0; c < TN; ++c) {
      const T t = warp_sum(acc[q][c]);
      if (lane == 0 && i0 + q < s && c < k) part[((int64_t)blockIdx.x * k + c) * s + i0 + q] = t;
    }
}

// G[c][i] = c_i sum_z part[z][c][i] (FP64, increasing z).  The factor c_i comes from `cvec` or,
// without it, from the eigenvalues.
template <typename T>
__global__ void block_g_kernel(const T* __restrict__ part, int nz, int s, int k, const T* __restrict__ cvec,
                               const double* __restrict__ lam, double rho, T* __restrict__ G) {
  const int64_t len = (int64_t)s * k;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < len; e += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(e % s);
    const double ci = cvec ? (double)cvec[i] : (double)(T)((lam[s - 1] + rho) / (lam[i] + rho) - 1.0);
    double t = 0.0;
    for (int z0 = 0; z0 < nz; z0 += 16) {
      T v[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) v[q] = z0 + q < nz ? part[(z0 + q) * len + e] : T(0);
#pragma unroll
      for (int q = 0; q < 16; ++q)
        if (z0 + q < nz) t += (double)v[q];
    }
    G[e] = (T)(ci * t);
  }
}

// Y = V + U G, tile 64 (j) x TN (c); each element's chain runs over i in increasing order.
// Y may be V: a thread reads its elements of V before it writes them.
template <typename T, int TN>
__global__ void __launch_bounds__(256) ug_tile_kernel(const T* __restrict__ U, const T* __restrict__ G, int64_t d,
                                                      int s, int k, const T* V, T* Y) {
  constexpr int RN = TN / 16;
  constexpr int LB = (BT_K * TN + 255) / 256;
  __shared__ T As[BT_K][BT_M + 1];
  __shared__ T Bs[BT_K][TN + 1];
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  const int64_t m0 = (int64_t)blockIdx.x * BT_M;
  const int n0 = blockIdx.y * TN;
  T acc[4][RN];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < RN; ++j) {
      const int64_t m = m0 + tx + 16 * i;
      const int c = n0 + ty + 16 * j;
      acc[i][j] = (m < d && c < k) ? V[m + (int64_t)c * d] : T(0);
    }
  T ra[4], rb[LB];
  auto load = [&](int k0) {
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      const int idx = threadIdx.x + 256 * l, mm = idx % BT_M, kk = idx / BT_M;
      ra[l] = (k0 + kk < s && m0 + mm < d) ? U[m0 + mm + (int64_t)(k0 + kk) * d] : T(0);
    }
#pragma unroll
    for (int l = 0; l < LB; ++l) {
      const int idx = threadIdx.x + 256 * l, kk = idx % BT_K, c = n0 + idx / BT_K;
      rb[l] = (k0 + kk < s && c < k && idx < BT_K * TN) ? G[(int64_t)c * s + k0 + kk] : T(0);
    }
  };
  load(0);
  for (int k0 = 0; k0 < s; k0 += BT_K) {
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      const int idx = threadIdx.x + 256 * l;
      As[idx / BT_M][idx % BT_M] = ra[l];
    }
#pragma unroll
    for (int l = 0; l < LB; ++l) {
      const int idx = threadIdx.x + 256 * l;
      if (idx < BT_K * TN) Bs[idx % BT_K][idx / BT_K] = rb[l];
    }
    __syncthreads();
    if (k0 + BT_K < s) load(k0 + BT_K);
    const int kend = min(BT_K, s - k0);
    auto step = [&](int kk) {
      T a[4], b[RN];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][tx + 16 * i];
#pragma unroll
      for (int j = 0; j < RN; ++j) b[j] = Bs[kk][ty + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < RN; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    };
    if (kend == BT_K) {
#pragma unroll
      for (int kk = 0; kk < BT_K; ++kk) step(kk);
    } else {
      for (int kk = 0; kk < kend; ++kk) step(kk);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < RN; ++j) {
      const int64_t m = m0 + tx + 16 * i;
      const int c = n0 + ty + 16 * j;
      if (m < d && c < k) Y[m + (int64_t)c * d] = acc[i][j];
    }
}

// The same for TN <= 4 columns: a thread per row j.
template <typename T, int TN>
__global__ void __launch_bounds__(kRowThreads) ug_small_kernel(const T* __restrict__ U, const T* __restrict__ G,
                                                               int64_t d, int s, int k, const T* V, T* Y) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  T* g = reinterpret_cast<T*>(sm_raw);   // [s][TN]
  for (int e = threadIdx.x; e < s * TN; e += kRowThreads) {
    const int i = e / TN, c = e % TN;
    g[e] = c < k ? G[(int64_t)c * s + i] : T(0);
  }
  __syncthreads();
  const int64_t j = blockIdx.x * (int64_t)kRowThreads + threadIdx.x;
  if (j >= d) return;
  T acc[TN];
#pragma unroll
  for (int c = 0; c < TN; ++c) acc[c] = c < k ? V[j + (int64_t)c * d] : T(0);
  constexpr int B = TN == 1 ? 32 : 16;   // loads of U in flight (4,000 x 700, one FP32 vector: 97 us a call with 32, 182 with 16)
  for (int i0 = 0; i0 < s; i0 += B) {
    T u[B];
#pragma unroll
    for (int q = 0; q < B; ++q) u[q] = i0 + q < s ? U[j + (int64_t)(i0 + q) * d] : T(0);
#pragma unroll
    for (int q = 0; q < B; ++q)
      if (i0 + q < s) {
#pragma unroll
        for (int c = 0; c < TN; ++c) acc[c] = fma(u[q], g[(i0 + q) * TN + c], acc[c]);
      }
  }
#pragma unroll
  for (int c = 0; c < TN; ++c)
    if (c < k) Y[j + (int64_t)c * d] = acc[c];
}

// Rows per partial of the tiled form: about two CTAs per SM, whole 64-row runs, and at most
// 4 x 10^6 partial values.
int64_t tile_chunk(int64_t d, int s, int k, int tn) {
  const int64_t tiles = (int64_t)((s + BT_M - 1) / BT_M) * ((k + tn - 1) / tn);
  int64_t nz = std::max<int64_t>(1, 2 * (int64_t)sm_count() / tiles);
  nz = std::max<int64_t>(1, std::min<int64_t>(nz, (4ll << 20) / ((int64_t)s * k)));
  const int64_t kc = (d + nz - 1) / nz;
  return (kc + 63) / 64 * 64;
}
int tile_cols(int k) { return k <= 16 ? 16 : 64; }

template <typename T, int TN>
cudaError_t launch_small(const T* U, const T* cvec, const double* lam, double rho, int64_t d, int s, int k, const T* V,
                         T* Y, T* part, T* G, cudaStream_t st) {
  const int nz = (int)((d + kSmallChunk - 1) / kSmallChunk);
  count_launch();
  utv_small_kernel<T, TN><<<dim3((unsigned)nz, (s + 63) / 64), 256, 0, st>>>(U, V, d, s, k, part);
  NYS_CUDA_TRY(cudaGetLastError());
  count_launch();
  block_g_kernel<T><<<(s * k + 127) / 128, 128, 0, st>>>(part, nz, s, k, cvec, lam, rho, G);
  NYS_CUDA_TRY(cudaGetLastError());
  count_launch();
  ug_small_kernel<T, TN><<<(unsigned)((d + kRowThreads - 1) / kRowThreads), kRowThreads, (size_t)s * TN * sizeof(T), st>>>(
      U, G, d, s, k, V, Y);
  return cudaGetLastError();
}

template <typename T, int TN>
cudaError_t launch_tile(const T* U, const T* cvec, const double* lam, double rho, int64_t d, int s, int k, const T* V,
                        T* Y, T* part, T* G, cudaStream_t st) {
  const int64_t kc = tile_chunk(d, s, k, TN);
  const int nz = (int)((d + kc - 1) / kc);
  const unsigned nt = (unsigned)((k + TN - 1) / TN);
  count_launch();
  const dim3 tiles((s + BT_M - 1) / BT_M, nt, (unsigned)nz);
  if (sizeof(T) == 4 && kc > kPairRows) utv_tile_kernel<T, TN, sizeof(T) == 4><<<tiles, 256, 0, st>>>(U, V, d, s, k, kc, part);
  else utv_tile_kernel<T, TN, false><<<tiles, 256, 0, st>>>(U, V, d, s, k, kc, part);
  NYS_CUDA_TRY(cudaGetLastError());
  count_launch();
  block_g_kernel<T><<<(unsigned)std::min<int64_t>(2048, ((int64_t)s * k + 127) / 128), 128, 0, st>>>(
      part, nz, s, k, cvec, lam, rho, G);
  NYS_CUDA_TRY(cudaGetLastError());
  count_launch();
  ug_tile_kernel<T, TN><<<dim3((unsigned)((d + BT_M - 1) / BT_M), nt), 256, 0, st>>>(U, G, d, s, k, V, Y);
  return cudaGetLastError();
}

}  // namespace

template <typename T>
size_t precond_block_work(int64_t d, int s, int k) {
  int64_t nz;
  if (k <= kSmallCols) {
    nz = (d + kSmallChunk - 1) / kSmallChunk;
  } else {
    const int64_t kc = tile_chunk(d, s, k, tile_cols(k));
    nz = (d + kc - 1) / kc;
  }
  return (size_t)(nz + 1) * s * k;
}

template <typename T>
cudaError_t precond_block(const T* U, const T* cvec, const double* lam, double rho, int64_t d, int s, int k,
                          const T* V, T* Y, T* work, cudaStream_t st) {
  if (s < 1 || k < 1) return cudaErrorInvalidValue;
  T* G = work;
  T* part = work + (size_t)s * k;
  if (k == 1) return launch_small<T, 1>(U, cvec, lam, rho, d, s, k, V, Y, part, G, st);
  if (k == 2) return launch_small<T, 2>(U, cvec, lam, rho, d, s, k, V, Y, part, G, st);
  if (k <= kSmallCols) return launch_small<T, 4>(U, cvec, lam, rho, d, s, k, V, Y, part, G, st);
  if (tile_cols(k) == 16) return launch_tile<T, 16>(U, cvec, lam, rho, d, s, k, V, Y, part, G, st);
  return launch_tile<T, 64>(U, cvec, lam, rho, d, s, k, V, Y, part, G, st);
}

template size_t precond_block_work<float>(int64_t, int, int);
template size_t precond_block_work<double>(int64_t, int, int);
template cudaError_t precond_block<float>(const float*, const float*, const double*, double, int64_t, int, int,
                                          const float*, float*, float*, cudaStream_t);
template cudaError_t precond_block<double>(const double*, const double*, const double*, double, int64_t, int, int,
                                           const double*, double*, double*, cudaStream_t);

}  // namespace nys
