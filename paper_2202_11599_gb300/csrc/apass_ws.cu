// Warp-specialised fused A-pass kernels: one pass y = A^T phi(A p) per launch (Table 1's
// T_mv, the H-matvec of Alg. Nystrom PCG), the same result layout as the kernels of
// apass.cu.  The roles and their per-stage mbarriers are described in apass_ws.cuh.
#include "apass_ws.cuh"

namespace nys {

// ------------------------------------------------------------------ float compute
template <int DT, int VPT, int R, int G>
__global__ void __launch_bounds__((2 * G + 2) * 32, 1) apass_ws_kernel(const ApassKArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) WsFloatSmem<R, G> sm;
  if (a.skip && *a.skip) return;
  if (a.executed && blockIdx.x == 0 && threadIdx.x == 0) *a.executed = 1;
  if (threadIdx.x == 0) {
    ws_init(sm.bars, a.S, G, G);
    sm.abort_flag = 0;
    sm.loss = 0.0;
  }
  __syncthreads();
  (void)ws_pass_float<DT, VPT, R, G>(a, sm, smem, 0, PSrcPlain{reinterpret_cast<const float*>(a.p)});
}

// ------------------------------------------------------------------ host side
namespace {

// Column vectors per thread of a group, from the instantiated set.
int ws_vpt(int64_t nvec, int group_threads, const int* set, int nset) {
  const int64_t need = (nvec + group_threads - 1) / group_threads;
  for (int i = 0; i < nset; ++i)
    if (need <= set[i]) return set[i];
  return -1;
}

constexpr int kVptF32[] = {1, 2, 3, 4, 5, 6, 8, 10};
constexpr int kVptBF16[] = {1, 2, 3, 4, 5, 6, 8};
constexpr int kVptFP8[] = {1, 2, 3, 4};

template <typename K>
cudaError_t ws_launch_kernel(K fn, int threads, const ApassKArgs& k, const ApassPlan& plan, cudaStream_t st,
                             bool prepare_only) {
  NYS_CUDA_TRY(ensure_max_dyn_smem((const void*)fn, kSmemBudget));
  if (prepare_only) return cudaSuccess;
  count_launch();
  fn<<<plan.grid, threads, plan.smem, st>>>(k);
  return cudaGetLastError();
}

template <int DT, int VPT>
cudaError_t ws_float_r(const ApassKArgs& k, const ApassPlan& plan, cudaStream_t st, bool prep) {
  constexpr int G = kWsGroupWarps;
  switch (plan.rows_per_step) {
    case 1: return ws_launch_kernel(apass_ws_kernel<DT, VPT, 1, G>, (2 * G + 2) * 32, k, plan, st, prep);
    case 2: return ws_launch_kernel(apass_ws_kernel<DT, VPT, 2, G>, (2 * G + 2) * 32, k, plan, st, prep);
    case 4: return ws_launch_kernel(apass_ws_kernel<DT, VPT, 4, G>, (2 * G + 2) * 32, k, plan, st, prep);
    default: return cudaErrorInvalidValue;
  }
}

template <int DT>
cudaError_t ws_float(const ApassKArgs& k, const ApassPlan& plan, cudaStream_t st, bool prep) {
  switch (plan.vpt) {
    case 1: return ws_float_r<DT, 1>(k, plan, st, prep);
    case 2: return ws_float_r<DT, 2>(k, plan, st, prep);
    case 3: return ws_float_r<DT, 3>(k, plan, st, prep);
    case 4: return ws_float_r<DT, 4>(k, plan, st, prep);
    case 5:
      if constexpr (DT != NYS_FP8E4M3) return ws_float_r<DT, 5>(k, plan, st, prep);
      break;
    case 6:
      if constexpr (DT != NYS_FP8E4M3) return ws_float_r<DT, 6>(k, plan, st, prep);
      break;
    case 8:
      if constexpr (DT != NYS_FP8E4M3) return ws_float_r<DT, 8>(k, plan, st, prep);
      break;
    case 10:
      if constexpr (DT == NYS_F32) return ws_float_r<DT, 10>(k, plan, st, prep);
      break;
    default: break;
  }
  return cudaErrorInvalidValue;
}

}  // namespace

bool apass_ws_layout(int dtype, int64_t d, int* threads, int* vpt) {
  switch (dtype) {
    case NYS_F32: *vpt = ws_vpt((d + 3) / 4, 32 * kWsGroupWarps, kVptF32, 8); break;
    case NYS_BF16: *vpt = ws_vpt((d + 7) / 8, 32 * kWsGroupWarps, kVptBF16, 7); break;
    case NYS_FP8E4M3: *vpt = ws_vpt((d + 15) / 16, 32 * kWsGroupWarps, kVptFP8, 4); break;
    case NYS_F64: *vpt = apass_wide64_vpt(d); break;
    default: return false;
  }
  if (*vpt < 0) return false;
  *threads = dtype == NYS_F64 ? apass_wide64_threads() : (2 * kWsGroupWarps + 2) * 32;
  return true;
}

cudaError_t apass_ws_launch(const ApassKArgs& k, const ApassPlan& plan, int dtype, cudaStream_t st,
                            bool prepare_only) {
  if (dtype == NYS_F64) return apass_wide64_launch(k, plan, st, prepare_only);
  if (plan.stages > kWsMaxStages || plan.stages < 2) return cudaErrorInvalidValue;
  switch (dtype) {
    case NYS_F32: return ws_float<NYS_F32>(k, plan, st, prepare_only);
    case NYS_BF16: return ws_float<NYS_BF16>(k, plan, st, prepare_only);
    case NYS_FP8E4M3: return ws_float<NYS_FP8E4M3>(k, plan, st, prepare_only);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace nys
