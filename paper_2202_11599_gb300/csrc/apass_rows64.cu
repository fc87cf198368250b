// Fused FP64 A-pass for narrow rows (the pass for FP64 matrices apass_wide64.cu does not take):
// y = A^T phi(A p) with one read of A, the result layout of apass.cu.
//
// The FP64 pipe bounds it: an SM quarter issues one FP64 warp instruction per 64 clocks, so
// the rows' n d products and n d updates set the pace and any FP64 instruction beside them
// costs the same, however few lanes need it.  Per stage of R rows:
//   * warps form the row dots, four rows per warp (p through L1, one reduce-scatter of six
//     additions for the four rows), a row's columns split over WS warps when R < 32;
//   * lanes r < R of one warp add a row's WS partials and apply phi;
//   * every thread applies the rank-R update to the column vectors it owns.
// With every thread adding the 16 warp partials of every row (64 dependent FP64 additions per
// thread and four-row step) the 2,000 x 500 pass, whose products take 3.3 us, took 52 us; it takes 8.6.
#include "apass_common.cuh"
#include "apass_ws.cuh"

namespace nys {

namespace {
constexpr int kR64Threads = 256;
constexpr int kR64Warps = kR64Threads / 32;
}  // namespace

template <int VPT>
__global__ void __launch_bounds__(kR64Threads, 1) apass_rows64_kernel(const ApassKArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t bars[kMaxStages];
  __shared__ double red[kR64Warps][kRows64Max];
  __shared__ double us[kRows64Max];
  __shared__ double lsh;
  if (a.skip && *a.skip) return;
  if (a.executed && blockIdx.x == 0 && threadIdx.x == 0) *a.executed = 1;
  const int ts_slot = timer_begin(a);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nvec = (int)((a.d + 1) / 2);
  const int64_t rowbytes = a.ld * 8;
  const int R = a.R, S = a.S;
  const int64_t stage_bytes = (int64_t)R * rowbytes;
  const int64_t r0 = a.n * (int64_t)blockIdx.x / gridDim.x;
  const int64_t r1 = a.n * (int64_t)(blockIdx.x + 1) / gridDim.x;
  const int nsteps = (int)((r1 - r0 + R - 1) / R);
  const int tail_vec = (a.d & 1) ? (int)(a.d / 2) : -1;   // its second element lies outside the matrix
  const bool nodot = a.mode == MODE_CONST;
  const uint32_t sbase = smem_u32(smem);
  const double* p = reinterpret_cast<const double*>(a.p);
  const bool p16 = (reinterpret_cast<uintptr_t>(p) & 15u) == 0;
  // WS warps share the columns of a group of four rows
  const int ngroups = (R + 3) / 4;
  const int WS = ngroups <= 1 ? 8 : (ngroups <= 2 ? 4 : (ngroups <= 4 ? 2 : 1));
  const int grp = warp / WS, part = warp % WS;

  if (tid == 0) {
    for (int s = 0; s < S; ++s) mbar_init(&bars[s], 1);
    fence_mbar_init();
    lsh = 0.0;
  }
  __syncthreads();
  const uint64_t pol = l2_evict_first_policy();   // A is streamed once per pass
  auto issue = [&](int step) {
    const int stage = step % S;
    const int64_t row = r0 + (int64_t)step * R;
    const uint32_t bytes = (uint32_t)(min((int64_t)R, r1 - row) * rowbytes);
    mbar_arrive_expect_tx(&bars[stage], bytes);
    tma_load_1d_hint(smem + stage * stage_bytes, a.A + row * rowbytes, bytes, &bars[stage], pol);
  };
  int issued = 0;
  if (tid == 0) {
    for (int st = 0; st < S && st < nsteps; ++st) issue(st);
    issued = min(S, nsteps);
  }
  double2 acc[VPT];
#pragma unroll
  for (int kk = 0; kk < VPT; ++kk) acc[kk] = make_double2(0.0, 0.0);
  double loss = 0.0;
  bool aborted = false;
  int k = 0;
  for (; k < nsteps; ++k) {
    const int stage = k % S;
    const uint32_t sb = sbase + (uint32_t)(stage * stage_bytes);
    const int64_t row0 = r0 + (int64_t)k * R;
    const int rows_here = (int)min((int64_t)R, r1 - row0);
    const double rin = tid < rows_here ? row_input(a, row0 + tid) : 0.0;
    const bool ok = mbar_wait_bounded(&bars[stage], (uint32_t)((k / S) & 1));
    if (ok && !nodot && grp < ngroups) {
      const int rb = 4 * grp, nr = min(4, rows_here - rb);   // nr <= 0: nothing
      double dot[4] = {0.0, 0.0, 0.0, 0.0};
      auto body = [&](auto full) {
        for (int v = part * 32 + lane; v < nvec; v += 32 * WS) {
          double p0, p1;
          if (v == tail_vec) {
            p0 = __ldg(p + 2 * (int64_t)v);
            p1 = 0.0;
          } else if (p16) {
            const double2 pv = __ldg(reinterpret_cast<const double2*>(p) + v);
            p0 = pv.x;
            p1 = pv.y;
          } else {
            p0 = __ldg(p + 2 * (int64_t)v);
            p1 = __ldg(p + 2 * (int64_t)v + 1);
          }
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            if (decltype(full)::value || r < nr) {
              uint4 x = lds128(sb + (uint32_t)((rb + r) * rowbytes) + (uint32_t)v * 16u);
              if (v == tail_vec) x.z = x.w = 0u;
              dot[r] = fma(__hiloint2double((int)x.y, (int)x.x), p0, dot[r]);
              dot[r] = fma(__hiloint2double((int)x.w, (int)x.z), p1, dot[r]);
            }
          }
        }
      };
      if (nr == 4) body(std::true_type{});
      else body(std::false_type{});
      const double t = warp_sum_rows<4>(dot, lane);
      if ((lane & 7) == 0) red[part][rb + (lane >> 3)] = t;
    }
    if (__syncthreads_or(!ok)) {
      aborted = true;
      break;
    }
    // every thread is done with stage k - 1: refill it
    if (tid == 0 && k >= 1 && k - 1 + S < nsteps) {
      issue(k - 1 + S);
      ++issued;
    }
    if (tid < R) {
      double u = 0.0;
      if (tid < rows_here) {
        double t = 0.0;
        if (!nodot)
          for (int w = 0; w < WS; ++w) t += red[w][tid];
        u = row_phi_d(a, row0 + tid, t, rin, loss);
        if (!nodot && a.t_out) a.t_out[row0 + tid] = t;
      }
      us[tid] = u;
    }
    __syncthreads();
    auto update = [&](int r, int cnt) {
#pragma unroll
      for (int kk = 0; kk < VPT; ++kk) {
        const int v = tid + kk * kR64Threads;
        if (v < nvec) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if (q < cnt) {
              uint4 x = lds128(sb + (uint32_t)((r + q) * rowbytes) + (uint32_t)v * 16u);
              if (v == tail_vec) x.z = x.w = 0u;
              const double u = us[r + q];
              acc[kk].x = fma(__hiloint2double((int)x.y, (int)x.x), u, acc[kk].x);
              acc[kk].y = fma(__hiloint2double((int)x.w, (int)x.z), u, acc[kk].y);
            }
          }
        }
      }
    };
    int r = 0;
    for (; r + 4 <= rows_here; r += 4) update(r, 4);
    if (r < rows_here) update(r, rows_here - r);
  }
  if (aborted) {
    // drain the copies still in flight into this CTA's shared memory (bounded), then report
    if (tid == 0) {
      for (int st = k; st < issued; ++st) (void)mbar_wait_bounded(&bars[st % S], (uint32_t)((st / S) & 1));
      atomicExch(a.status, (int)NYS_ETIMEOUT);
    }
    return;
  }
  double* part_out = reinterpret_cast<double*>(a.partial) + (int64_t)blockIdx.x * a.dpad;
#pragma unroll
  for (int kk = 0; kk < VPT; ++kk) {
    const int v = tid + kk * kR64Threads;
    if (v < nvec) *reinterpret_cast<double2*>(part_out + 2 * (int64_t)v) = acc[kk];
  }
  if (a.loss_part) {
    // rows are finished by the lanes of warp 0
    if (warp == 0) {
      const double l = warp_sum(loss);
      if (lane == 0) a.loss_part[blockIdx.x] = l;
    }
  }
  timer_end(a, ts_slot, NYS_F64);
}

// Column vectors (two values) per thread of the update; 24 cover 12,288 columns.
int apass_rows64_vpt(int64_t d) {
  const int64_t need = ((d + 1) / 2 + kR64Threads - 1) / kR64Threads;
  for (int v : {1, 2, 4, 8, 16, 24})
    if (need <= v) return v;
  return -1;
}

namespace {
template <int VPT>
cudaError_t rows64_launch(const ApassKArgs& k, const ApassPlan& plan, cudaStream_t st, bool prepare_only) {
  auto fn = apass_rows64_kernel<VPT>;
  NYS_CUDA_TRY(ensure_max_dyn_smem((const void*)fn, kSmemBudget));
  if (prepare_only) return cudaSuccess;
  count_launch();
  fn<<<plan.grid, kR64Threads, plan.smem, st>>>(k);
  return cudaGetLastError();
}
}  // namespace

cudaError_t apass_rows64_launch(const ApassKArgs& k, const ApassPlan& plan, cudaStream_t st, bool prepare_only) {
  if (plan.stages > kMaxStages || plan.rows_per_step > kRows64Max) return cudaErrorInvalidValue;
  switch (plan.vpt) {
    case 1: return rows64_launch<1>(k, plan, st, prepare_only);
    case 2: return rows64_launch<2>(k, plan, st, prepare_only);
    case 4: return rows64_launch<4>(k, plan, st, prepare_only);
    case 8: return rows64_launch<8>(k, plan, st, prepare_only);
    case 16: return rows64_launch<16>(k, plan, st, prepare_only);
    case 24: return rows64_launch<24>(k, plan, st, prepare_only);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace nys
