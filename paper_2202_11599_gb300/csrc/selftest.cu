// Entry points for the tests only, not part of nysadmm.h: single device functions that the library otherwise
// runs inside a sketch, so that their results can be compared entry by entry.
#include "device_util.cuh"
#include "nys_internal.cuh"
#include "solver.cuh"

namespace {
__global__ void g_entry_kernel(const float* part, int nb, int s, float c, float* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < s) out[i] = nys::g_entry<float>(part, nb, s, i, c);
}
nys_status read_status(const int* status, cudaStream_t st) {
  int h = 0;
  if (cudaMemcpyAsync(&h, status, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return NYS_ECUDA;
  return (nys_status)h;
}
}  // namespace

// gemm64: C (M x N, column-major) = diag(D) A B^T with the exponents taken from A and B here.  k_contiguous: A is
// M x K row-major, else K x M; B is N x K row-major; all arrays on the device.
extern "C" nys_status nys_test_gemm64(const double* A, int32_t k_contiguous, int64_t lda, int64_t M, const double* B,
                                      int64_t ldb, int32_t N, int64_t K, const double* D, double* C, void* stream) {
  using namespace nys;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  Pool pool(st);
  unsigned* ea = pool.alloc<unsigned>(M);
  unsigned* eb = pool.alloc<unsigned>(N);
  void* work = pool.alloc<unsigned char>(gemm64_work_bytes(M, N, K));
  int* status = pool.alloc<int>(1);
  if (!pool.ok()) return NYS_ENOMEM;
  if (cudaMemsetAsync(status, 0, sizeof(int), st) != cudaSuccess) return NYS_ECUDA;
  if ((k_contiguous ? absmax_f64(A, M, K, lda, ea, nullptr, st) : absmax_f64(A, K, M, lda, nullptr, ea, st)) != cudaSuccess ||
      absmax_f64(B, N, K, ldb, eb, nullptr, st) != cudaSuccess ||
      gemm64(A, k_contiguous != 0, lda, ea, M, B, ldb, eb, N, K, D, C, M, work, status, st, /*any_scale=*/true) != cudaSuccess)
    return NYS_ECUDA;
  return read_status(status, st);
}

// chol_upper of M (s x s, column-major, in place: C^T C = M) and, when Y is given, Y <- Y C^{-1} (d x s, column-major).
// *info (host): chol_upper's.
extern "C" nys_status nys_test_triangular(double* M, int32_t s, double* Y, int64_t d, int32_t* info, void* stream) {
  using namespace nys;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  Pool pool(st);
  int* words = pool.alloc<int>(2);   // info, status
  void* work = pool.alloc<unsigned char>(Y ? trsm_work_bytes(d, s) : 1);
  if (!pool.ok()) return NYS_ENOMEM;
  if (cudaMemsetAsync(words, 0, 2 * sizeof(int), st) != cudaSuccess || chol_upper(M, s, words, st) != cudaSuccess ||
      (Y && trsm_right_upper(M, s, Y, d, work, words + 1, st) != cudaSuccess) ||
      cudaMemcpyAsync(info, words, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess)
    return NYS_ECUDA;
  return read_status(words + 1, st);
}

// Rows per step the autotuner would time on A (rows[0 .. return value)) and the one that the plan takes now (*planned; 0: no plan).
extern "C" int32_t nys_test_rows(const nys_matrix* A, int32_t* rows, int32_t* planned) {
  int cand[3] = {0, 0, 0};
  const int n = nys::apass_row_candidates(A, cand);
  for (int i = 0; i < n; ++i) rows[i] = cand[i];
  nys::ApassPlan plan;
  *planned = nys::apass_plan(A, &plan) ? plan.rows_per_step : 0;
  return n;
}

extern "C" nys_status nys_test_step_status(int32_t wait, int32_t usable, int32_t if_not) {
  return nys::step_status(wait, usable != 0, (nys_status)if_not);
}

// out[i] = c sum_b part[b][i] as the fused vector steps form it (part nb x s).
extern "C" nys_status nys_test_g_entry(const float* part, int32_t nb, int32_t s, float c, float* out, void* stream) {
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  g_entry_kernel<<<(s + 127) / 128, 128, 0, st>>>(part, nb, s, c, out);
  return cudaGetLastError() == cudaSuccess && cudaStreamSynchronize(st) == cudaSuccess ? NYS_OK : NYS_ECUDA;
}
