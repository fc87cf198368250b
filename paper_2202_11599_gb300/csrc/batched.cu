// Multi-right-hand-side Nystrom PCG for a lasso regularisation path.
//
// k lasso problems that share A, b and rho (and differ in gamma) share the
// x-subproblem matrix H + rho I of Eq. ADMMSubProb and therefore one Nystrom
// preconditioner.  Their k PCG solves (Alg. Nystrom PCG, one per column) are run
// side by side: every matvec reads A ONCE for all k columns as the two dense
// products W = A P (n x k) and V = A^T W + rho P (d x k), and the preconditioner is
// applied to the d x k block with two small GEMMs.  Each column keeps its own
// alpha, beta, residual and stop test; a converged column is frozen (alpha = 0).
// Vectors are d x k column-major in the PCG compute type; reductions are
// fixed-order per column.
#include <algorithm>
#include <vector>

#include "device_util.cuh"
#include "nys_internal.cuh"
#include "solver.cuh"

namespace nys {
namespace {

// Per-column scalars of the k PCG solves.  Every kernel below that changes them reads one copy
// and writes another (its blocks with chunk 0), so that the blocks of a column all see the
// same values.
struct BCol {
  double wy, pv, w2, r2, thresh2;
  float alpha, beta;
  int iters, done, status, pad;
};

// Vector kernels: block (b, c) of kVecThreads threads owns rows [1024 b, 1024 b + 1024) of
// column c, four elements per thread, and leaves one partial sum per block, so a column's dot
// product is nb partials added in increasing b.  (One block per 1,024 rows over all columns
// left four blocks for a 4,000 x 64 panel: 62 us per dot and 206 us per prox step.)
constexpr int kColChunk = 1024;
constexpr int kColPer = kColChunk / kVecThreads;
int col_blocks(int64_t d) { return (int)((d + kColChunk - 1) / kColChunk); }

// V = rho P + (sum of the partials of A^T D A P); with nz = 0 the sum is in V already.
template <typename C>
__global__ void b_matvec_finish_kernel(const C* __restrict__ part, int nz, int64_t len, C rho, const C* __restrict__ P,
                                       C* __restrict__ V) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len; i += (int64_t)gridDim.x * blockDim.x) {
    C s = nz ? C(0) : V[i];
    for (int z = 0; z < nz; ++z) s += part[z * len + i];
    V[i] = fma(rho, P[i], s);
  }
}

// Sum of a column's partials part[b * k + c] (increasing b; nb is small).
__device__ __forceinline__ double col_sum(const double* __restrict__ part, int nb, int k, int c) {
  double s = 0.0;
  for (int b = 0; b < nb; ++b) s += part[(int64_t)b * k + c];
  return s;
}

// part[b][c] = the block's share of x_c . y_c.  With `in` the column's stop test runs first
// (||w||^2 from w2_part, the iteration counted): the dot is w . y of the same iteration.
template <typename C>
__global__ void __launch_bounds__(kVecThreads) b_dot_kernel(const C* __restrict__ X, const C* __restrict__ Y,
                                                            int64_t d, int k, double* part,
                                                            const double* __restrict__ w2_part, int maxit,
                                                            const BCol* __restrict__ in, BCol* __restrict__ out) {
  __shared__ double sh[kVecThreads / 32];
  const int c = blockIdx.y;
  const int64_t j0 = (int64_t)blockIdx.x * kColChunk + threadIdx.x;
  double acc = 0.0;
#pragma unroll
  for (int q = 0; q < kColPer; ++q) {
    const int64_t j = j0 + q * kVecThreads;
    if (j < d) acc += (double)X[(int64_t)c * d + j] * (double)Y[(int64_t)c * d + j];
  }
  const double t = block_sum_t0<kVecThreads>(acc, sh);
  if (threadIdx.x != 0) return;
  part[(int64_t)blockIdx.x * k + c] = t;
  if (in && blockIdx.x == 0) {
    BCol s = in[c];
    if (!s.done) {
      s.w2 = col_sum(w2_part, gridDim.x, k, c);
      s.iters += 1;
      if (!(s.w2 > s.thresh2)) {
        s.done = 1;
      } else if (s.iters >= maxit) {
        s.done = 1;
        s.status = NYS_ENOCONV;
      }
    }
    out[c] = s;
  }
}

// w = r - v (v = (H + rho I) x0, or x0 = 0) with the partials of ||r||^2 and ||w||^2.
template <typename C>
__global__ void __launch_bounds__(kVecThreads) b_init_w_kernel(int64_t d, int k, const C* __restrict__ R,
                                                               const C* __restrict__ V, C* __restrict__ W,
                                                               double* r2_part, double* w2_part) {
  __shared__ double sh[kVecThreads / 32];
  const int c = blockIdx.y;
  const int64_t j0 = (int64_t)blockIdx.x * kColChunk + threadIdx.x;
  double lr = 0.0, lw = 0.0;
#pragma unroll
  for (int q = 0; q < kColPer; ++q) {
    const int64_t j = j0 + q * kVecThreads;
    if (j < d) {
      const int64_t e = (int64_t)c * d + j;
      const C r = R[e], w = V ? r - V[e] : r;
      W[e] = w;
      lr += (double)r * (double)r;
      lw += (double)w * (double)w;
    }
  }
  const double tr = block_sum_t0<kVecThreads>(lr, sh);
  const double tw = block_sum_t0<kVecThreads>(lw, sh);
  if (threadIdx.x == 0) {
    r2_part[(int64_t)blockIdx.x * k + c] = tr;
    w2_part[(int64_t)blockIdx.x * k + c] = tw;
  }
}

// Thresholds and first stop test of every column.
__global__ void b_start_kernel(int k, int nb, const double* r2_part, const double* w2_part, double tol, int tol_abs,
                               BCol* out) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= k) return;
  BCol s = {};
  s.r2 = col_sum(r2_part, nb, k, c);
  s.w2 = col_sum(w2_part, nb, k, c);
  s.thresh2 = tol_abs ? tol * tol : tol * tol * s.r2;
  s.done = !(s.w2 > s.thresh2);
  out[c] = s;
}

// alpha = w . y / p . v of each column (0 for a finished one), x += alpha p, w -= alpha v and
// the partials of ||w||^2.
template <typename C>
__global__ void __launch_bounds__(kVecThreads) b_update_kernel(int64_t d, int k, C* __restrict__ X, C* __restrict__ W,
                                                               const C* __restrict__ P, const C* __restrict__ V,
                                                               const double* __restrict__ pv_part, double* w2_part,
                                                               const BCol* __restrict__ in, BCol* __restrict__ out) {
  __shared__ double sh[kVecThreads / 32];
  __shared__ float s_alpha;
  const int c = blockIdx.y;
  if (threadIdx.x == 0) {
    BCol s = in[c];
    s.pv = col_sum(pv_part, gridDim.x, k, c);
    s.alpha = 0.f;
    if (!s.done) {
      if (!(s.pv > 0.0) || !isfinite(s.pv)) {
        s.done = 1;
        s.status = s.iters == 0 ? NYS_EBREAKDOWN : NYS_ENOCONV;
      } else {
        s.alpha = (float)(s.wy / s.pv);
      }
    }
    s_alpha = s.alpha;
    if (blockIdx.x == 0) out[c] = s;
  }
  __syncthreads();
  const C a = (C)s_alpha;
  const int64_t j0 = (int64_t)blockIdx.x * kColChunk + threadIdx.x;
  double acc = 0.0;
#pragma unroll
  for (int q = 0; q < kColPer; ++q) {
    const int64_t j = j0 + q * kVecThreads;
    if (j < d) {
      const int64_t e = (int64_t)c * d + j;
      X[e] = fma(a, P[e], X[e]);
      const C w = fma(-a, V[e], W[e]);
      W[e] = w;
      acc += (double)w * (double)w;
    }
  }
  const double t = block_sum_t0<kVecThreads>(acc, sh);
  if (threadIdx.x == 0) w2_part[(int64_t)blockIdx.x * k + c] = t;
}

// beta = (w . y)_new / (w . y)_old of each column, p = y + beta p (init: p = y).  Counts the
// finished columns in *ndone (zeroed by the caller).
template <typename C>
__global__ void __launch_bounds__(kVecThreads) b_direction_kernel(int64_t d, int k, const C* __restrict__ Y,
                                                                  C* __restrict__ P,
                                                                  const double* __restrict__ wy_part, int init,
                                                                  const BCol* __restrict__ in, BCol* __restrict__ out,
                                                                  int* ndone) {
  __shared__ float s_beta;
  const int c = blockIdx.y;
  if (threadIdx.x == 0) {
    BCol s = in[c];
    const double wy = col_sum(wy_part, gridDim.x, k, c);
    s.beta = s.wy > 0.0 ? (float)(wy / s.wy) : 0.f;
    s.wy = wy;
    s_beta = s.beta;
    if (blockIdx.x == 0) {
      out[c] = s;
      if (s.done) atomicAdd(ndone, 1);
    }
  }
  __syncthreads();
  const C b = (C)s_beta;
  const int64_t j0 = (int64_t)blockIdx.x * kColChunk + threadIdx.x;
#pragma unroll
  for (int q = 0; q < kColPer; ++q) {
    const int64_t j = j0 + q * kVecThreads;
    if (j < d) {
      const int64_t e = (int64_t)c * d + j;
      P[e] = init ? Y[e] : fma(b, P[e], Y[e]);
    }
  }
}

unsigned grid_for(int64_t len) { return (unsigned)std::max<int64_t>(1, std::min<int64_t>(8192, (len + 255) / 256)); }

}  // namespace

template <typename C>
nys_status batched_pcg_run(const PcgProblem& pb, const TcPrepared* tcp, const PrecondView& P, const C* R, C* X, int k,
                           const PcgParams& prm, cudaStream_t st, std::vector<int>* iters_out) {
  const int64_t d = pb.A->d, n = pb.A->n;
  const int s = P.s;
  const int64_t len = d * k;
  const int nb = col_blocks(d);
  const bool use_tc = tcp != nullptr;
  Pool pool(st);
  C* W = pool.alloc<C>(len);
  C* Y = pool.alloc<C>(len);
  C* Pd = pool.alloc<C>(len);
  C* V = pool.alloc<C>(len);
  constexpr bool f64 = sizeof(C) == 8;
  const bool cuda_cores = !f64 && !use_tc;
  C* Wn = cuda_cores ? pool.alloc<C>((size_t)n * k) : nullptr;
  const size_t atw_bytes = cuda_cores ? sketch_atw_work_bytes(pb.A, k) : 0;
  void* atw = cuda_cores ? pool.alloc<unsigned char>(atw_bytes) : nullptr;
  void* tcw = use_tc ? pool.alloc<unsigned char>(tc_hmm_work_bytes(pb.A, *tcp, k))
                     : (f64 ? pool.alloc<unsigned char>(hmm64_bytes(pb.A, k)) : nullptr);
  C* gwork = s > 0 ? pool.alloc<C>(precond_block_work<C>(d, s, k)) : nullptr;
  double* pv_part = pool.alloc<double>((size_t)nb * k);
  double* w2_part = pool.alloc<double>((size_t)nb * k);
  double* wy_part = pool.alloc<double>((size_t)nb * k);
  BCol* cols = pool.alloc<BCol>(2 * (size_t)k);
  int* ndone = pool.alloc<int>(2);   // finished columns; status of the tensor-core products
  if (!pool.ok()) return NYS_ENOMEM;
  BCol *cin = cols, *cout = cols + k;
  int* tc_status = f64 ? hmm64_status(pb.A, k, tcw) : ndone + 1;
  const C* U = reinterpret_cast<const C*>(P.U);
  const C* cvec = reinterpret_cast<const C*>(P.c);
#define B_OK(x)                             \
  do {                                      \
    if ((x) != cudaSuccess) return NYS_ECUDA; \
  } while (0)
  auto launch_ok = [&]() { return cudaGetLastError() == cudaSuccess; };
  const dim3 cgrid((unsigned)nb, (unsigned)k);
  if (f64) B_OK(hmm64_prepare(pb.A, k, tcw, st));
  // BF16 and FP32 storage: the k-column products run on the tensor cores (the same tcgen05
  // GEMMs as the sketch, FP32 operand as three BF16 terms);
  // FP64 storage on the FP64 products of the sketch.
  // V = A^T (A P) + rho P for the k columns of P (reads A once)
  auto bmatvec = [&](const C* Pin, C* Vout) -> bool {
    if constexpr (sizeof(C) == 4) {
      if (use_tc) return tc_hmm(pb.A, *tcp, pb.D, reinterpret_cast<const float*>(Pin), k, pb.rho,
                                reinterpret_cast<float*>(Vout), tcw, tc_status, st) == cudaSuccess;
    } else {
      if (hmm64(pb.A, pb.D, Pin, k, Vout, tcw, st) != cudaSuccess) return false;
      count_launch();
      b_matvec_finish_kernel<C><<<grid_for(len), 256, 0, st>>>(nullptr, 0, len, (C)pb.rho, Pin, Vout);
      return launch_ok();
    }
    if (sketch_aw(pb.A, Pin, k, pb.D, Wn, st) != cudaSuccess) return false;
    int nz = 0;
    if (sketch_atw_partials(pb.A, Wn, k, atw, atw_bytes, &nz, st) != cudaSuccess) return false;
    count_launch();
    b_matvec_finish_kernel<C><<<grid_for(len), 256, 0, st>>>((const C*)atw, nz, len, (C)pb.rho, Pin, Vout);
    return launch_ok();
  };
  // Y = P^{-1} W = U diag(c) U^T W + W
  auto precond = [&]() -> bool {
    if (s == 0) return cudaMemcpyAsync(Y, W, len * sizeof(C), cudaMemcpyDeviceToDevice, st) == cudaSuccess;
    return precond_block<C>(U, cvec, nullptr, 0.0, d, s, k, W, Y, gwork, st) == cudaSuccess;
  };
  auto direction = [&](int init) -> bool {
    count_launch();
    b_direction_kernel<C><<<cgrid, kVecThreads, 0, st>>>(d, k, Y, Pd, wy_part, init, cin, cout, ndone);
    std::swap(cin, cout);
    return launch_ok();
  };

  // init: W = R - (H + rho I) X0, thresholds, Y = P^{-1} W, P = Y
  B_OK(cudaMemsetAsync(ndone, 0, 2 * sizeof(int), st));
  if (!prm.x0_zero) {
    if (!bmatvec(X, V)) return NYS_ECUDA;
  }
  count_launch();
  b_init_w_kernel<C><<<cgrid, kVecThreads, 0, st>>>(d, k, R, prm.x0_zero ? nullptr : V, W, pv_part, w2_part);
  count_launch();
  b_start_kernel<<<(k + 127) / 128, 128, 0, st>>>(k, nb, pv_part, w2_part, prm.tol, prm.tol_abs, cin);
  if (!launch_ok() || !precond()) return NYS_ECUDA;
  count_launch();
  b_dot_kernel<C><<<cgrid, kVecThreads, 0, st>>>(W, Y, d, k, wy_part, nullptr, 0, nullptr, nullptr);
  if (!launch_ok() || !direction(1)) return NYS_ECUDA;
  std::vector<BCol> hc(k);
  int host2[2] = {0, 0};
  B_OK(cudaMemcpyAsync(host2, ndone, sizeof(host2), cudaMemcpyDeviceToHost, st));
  B_OK(cudaStreamSynchronize(st));
  const int cap = prm.fixed >= 0 ? prm.fixed : prm.maxit;
  for (int it = 0; it < cap && host2[0] < k && !host2[1]; ++it) {
    if (!bmatvec(Pd, V)) return NYS_ECUDA;
    count_launch();
    b_dot_kernel<C><<<cgrid, kVecThreads, 0, st>>>(Pd, V, d, k, pv_part, nullptr, 0, nullptr, nullptr);
    count_launch();
    b_update_kernel<C><<<cgrid, kVecThreads, 0, st>>>(d, k, X, W, Pd, V, pv_part, w2_part, cin, cout);
    std::swap(cin, cout);
    B_OK(cudaMemsetAsync(ndone, 0, sizeof(int), st));
    if (!launch_ok() || !precond()) return NYS_ECUDA;
    count_launch();
    b_dot_kernel<C><<<cgrid, kVecThreads, 0, st>>>(W, Y, d, k, wy_part, w2_part, prm.maxit, cin, cout);
    std::swap(cin, cout);
    if (!launch_ok() || !direction(0)) return NYS_ECUDA;
    B_OK(cudaMemcpyAsync(host2, ndone, sizeof(host2), cudaMemcpyDeviceToHost, st));
    B_OK(cudaStreamSynchronize(st));
  }
  B_OK(cudaMemcpyAsync(hc.data(), cin, k * sizeof(BCol), cudaMemcpyDeviceToHost, st));
  B_OK(cudaMemcpyAsync(host2 + 1, tc_status, sizeof(int), cudaMemcpyDeviceToHost, st));
  B_OK(cudaStreamSynchronize(st));
#undef B_OK
  if (host2[1]) return NYS_ECUDA;   // a bounded wait of a tensor-core product ran out
  nys_status res = NYS_OK;
  if (iters_out) iters_out->assign(k, 0);
  for (int c = 0; c < k; ++c) {
    if (iters_out) (*iters_out)[c] = hc[c].iters;
    if (hc[c].status == NYS_EBREAKDOWN) res = NYS_EBREAKDOWN;
    else if (res == NYS_OK && (hc[c].status == NYS_ENOCONV || (!hc[c].done && prm.fixed < 0))) res = NYS_ENOCONV;
  }
  return res;
}
template nys_status batched_pcg_run<float>(const PcgProblem&, const TcPrepared*, const PrecondView&, const float*,
                                           float*, int, const PcgParams&, cudaStream_t, std::vector<int>*);
template nys_status batched_pcg_run<double>(const PcgProblem&, const TcPrepared*, const PrecondView&, const double*,
                                            double*, int, const PcgParams&, cudaStream_t, std::vector<int>*);

// ------------------------------------------------------------------ ADMM steps on d x k blocks
namespace {
template <typename C>
__global__ void __launch_bounds__(kVecThreads) b_rhs_kernel(int64_t d, const double* __restrict__ q,
                                                            const double* __restrict__ Z,
                                                            const double* __restrict__ Uu, double rho,
                                                            C* __restrict__ R) {
  const int64_t j0 = (int64_t)blockIdx.x * kColChunk + threadIdx.x, base = (int64_t)blockIdx.y * d;
#pragma unroll
  for (int t = 0; t < kColPer; ++t) {
    const int64_t j = j0 + t * kVecThreads;
    if (j < d) R[base + j] = (C)fma(rho, Z[base + j] - Uu[base + j], q[j]);
  }
}

// column c: z = S_{kappa_c}(x + u), u += x - z; partials of ||x - z||^2 and ||z - z_old||^2
template <typename C>
__global__ void __launch_bounds__(kVecThreads) b_zu_kernel(int64_t d, int k, const C* __restrict__ Xc,
                                                           double* __restrict__ X, double* __restrict__ Z,
                                                           double* __restrict__ Uu, const double* __restrict__ kappa,
                                                           double* part) {
  __shared__ double sh[kVecThreads / 32];
  const int c = blockIdx.y;
  const int64_t j0 = (int64_t)blockIdx.x * kColChunk + threadIdx.x;
  const double kap = kappa[c];
  double a0 = 0.0, a1 = 0.0;
#pragma unroll
  for (int t = 0; t < kColPer; ++t) {
    const int64_t j = j0 + t * kVecThreads;
    if (j < d) {
      const int64_t i = (int64_t)c * d + j;
      const double xj = (double)Xc[i];
      const double zo = Z[i];
      const double uo = Uu[i];
      const double vj = xj + uo;
      const double mag = fabs(vj) - kap;
      const double zj = mag > 0.0 ? copysign(mag, vj) : 0.0;
      X[i] = xj;
      Z[i] = zj;
      Uu[i] = uo + (xj - zj);
      a0 += (xj - zj) * (xj - zj);
      a1 += (zj - zo) * (zj - zo);
    }
  }
  const double t0 = block_sum_t0<kVecThreads>(a0, sh);
  const double t1 = block_sum_t0<kVecThreads>(a1, sh);
  if (threadIdx.x == 0) {
    part[((int64_t)blockIdx.x * k + c) * 2] = t0;
    part[((int64_t)blockIdx.x * k + c) * 2 + 1] = t1;
  }
}
}  // namespace

template <typename C>
cudaError_t batched_rhs(int64_t d, int k, const double* q, const double* Z, const double* Uu, double rho, C* R,
                        cudaStream_t st) {
  count_launch();
  b_rhs_kernel<C><<<dim3((unsigned)col_blocks(d), (unsigned)k), kVecThreads, 0, st>>>(d, q, Z, Uu, rho, R);
  return cudaGetLastError();
}
template <typename C>
cudaError_t batched_zu(int64_t d, int k, const C* Xc, double* X, double* Z, double* Uu, const double* kappa,
                       double* part, int* nb_out, cudaStream_t st) {
  const int nb = col_blocks(d);
  count_launch();
  b_zu_kernel<C><<<dim3((unsigned)nb, (unsigned)k), kVecThreads, 0, st>>>(d, k, Xc, X, Z, Uu, kappa, part);
  *nb_out = nb;
  return cudaGetLastError();
}
int batched_zu_blocks(int64_t d) { return col_blocks(d); }
template cudaError_t batched_rhs<float>(int64_t, int, const double*, const double*, const double*, double, float*,
                                        cudaStream_t);
template cudaError_t batched_rhs<double>(int64_t, int, const double*, const double*, const double*, double, double*,
                                         cudaStream_t);
template cudaError_t batched_zu<float>(int64_t, int, const float*, double*, double*, double*, const double*, double*,
                                       int*, cudaStream_t);
template cudaError_t batched_zu<double>(int64_t, int, const double*, double*, double*, double*, const double*,
                                        double*, int*, cudaStream_t);

}  // namespace nys
