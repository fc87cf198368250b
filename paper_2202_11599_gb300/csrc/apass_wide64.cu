// Fused FP64 A-pass for wide rows: y = A^T phi(A p) by row blocks, the result layout of apass.cu.
//
// The FP64 pipe bounds it (64 clocks per warp instruction and SM quarter; HBM could deliver A
// 1.4 times over in the time of its 2 n d FMAs), so what counts is how little else goes through
// that pipe and that it never waits.  A CTA takes its rows in blocks of up to 16 R: its sixteen warps
// form R rows' dots each (p in shared memory, two FMA chains a row), the lanes of one warp apply phi
// to the whole block at once, then every thread adds the block to the columns it owns,
// reading the rows again, through L2 or HBM.  Beside the FMAs a block of 32 rows costs one
// reduction per warp and one evaluation of phi.
//
// 39,999 x 4,001: 567 us (FMAs alone 527), 200,000 x 5,000 in logistic mode 3.42 ms (3.3).  With dot, finishing
// and update warps side by side over a ring of stages it was 684 us and 5.55 ms: each FP64 instruction of the
// finisher's chain queues for the pipe behind every other warp's.
#include "apass_common.cuh"
#include "apass_ws.cuh"

namespace nys {

namespace {
constexpr int kW64Threads = 512;
constexpr int kW64Warps = kW64Threads / 32;

// 16 bytes of A: read once per phase by one SM, so kept out of L1.
__device__ __forceinline__ double2 load_a(const double2* p) {
  double2 v;
  asm volatile("ld.global.nc.L1::no_allocate.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
  return v;
}
}  // namespace

template <int VPT>
__global__ void __launch_bounds__(kW64Threads, 1) apass_wide64_kernel(const ApassKArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ double ts[2 * kW64Warps], us[2 * kW64Warps];
  if (a.skip && *a.skip) return;
  if (a.executed && blockIdx.x == 0 && threadIdx.x == 0) *a.executed = 1;
  const int ts_slot = timer_begin(a);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nvec = (int)((a.d + 1) / 2);
  const int tail_vec = (a.d & 1) ? nvec - 1 : -1;   // its second element lies outside the matrix
  const int64_t ldv = a.ld / 2;
  const double2* A = reinterpret_cast<const double2*>(a.A);
  const int64_t r0 = a.n * (int64_t)blockIdx.x / gridDim.x;
  const int64_t r1 = a.n * (int64_t)(blockIdx.x + 1) / gridDim.x;
  const int64_t cap = (int64_t)kW64Warps * a.R, rows = r1 - r0, nblk = (rows + cap - 1) / cap;
  const int B = (int)((rows + nblk - 1) / max((int64_t)1, nblk));   // blocks evened out over the slab
  const bool nodot = a.mode == MODE_CONST;
  double2* psh = reinterpret_cast<double2*>(smem);
  if (!nodot) {
    const double* p = reinterpret_cast<const double*>(a.p);
    for (int v = tid; v < nvec; v += kW64Threads)
      psh[v] = make_double2(__ldg(p + 2 * (int64_t)v), v == tail_vec ? 0.0 : __ldg(p + 2 * (int64_t)v + 1));
    __syncthreads();
  }
  double2 acc[VPT];
#pragma unroll
  for (int kk = 0; kk < VPT; ++kk) acc[kk] = make_double2(0.0, 0.0);
  double loss = 0.0;

  // dots of NR rows, kW64Warps apart, from Ar on (lanes over the column vectors); of `share` warps on the same
  // rows, this is number `part` and takes every share-th batch of columns
  auto dots = [&](auto nr, const double2* Ar, int part, int share) -> double {
    constexpr int NR = decltype(nr)::value, U = (VPT <= 6 ? 8 : 4) / NR;
    double sx[NR], sy[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) sx[r] = sy[r] = 0.0;
    auto batch = [&](int v0, auto full) {
      double2 x[NR][U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int v = v0 + 32 * u;
        if (decltype(full)::value || v < nvec) {
#pragma unroll
          for (int r = 0; r < NR; ++r) x[r][u] = load_a(Ar + (int64_t)r * kW64Warps * ldv + v);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int v = v0 + 32 * u;
        if (decltype(full)::value || v < nvec) {
          const double2 pv = psh[v];
#pragma unroll
          for (int r = 0; r < NR; ++r) {
            if (!decltype(full)::value && v == tail_vec) x[r][u].y = 0.0;
            sx[r] = fma(x[r][u].x, pv.x, sx[r]);
            sy[r] = fma(x[r][u].y, pv.y, sy[r]);
          }
        }
      }
    };
    int v0 = lane + 32 * U * part;
    const int step = 32 * U * share;
    const int whole = (nvec - 1) / (32 * U) * (32 * U);   // batches that end before the last vector
    for (; v0 < whole; v0 += step) batch(v0, std::true_type{});
    for (; v0 < nvec; v0 += step) batch(v0, std::false_type{});
#pragma unroll
    for (int r = 0; r < NR; ++r) sx[r] += sy[r];
    __syncwarp();
    return warp_sum_rows<NR>(sx, lane);
  };
  // acc += sum_r u_r a_r over the block, the first NV of this thread's vectors (the last one may lie
  // beyond the row: it reads the row's last vector and is not stored)
  auto update = [&](auto nv, const double2* Ab, int nr) {
    constexpr int NV = decltype(nv)::value;
    constexpr int RB = NV <= 1 ? 8 : (NV <= 2 ? 4 : (NV <= 6 ? 2 : 1));   // rows in flight
    if constexpr (NV > 0) {
      auto step = [&](int r, auto cnt) {
        constexpr int CNT = decltype(cnt)::value;
        double2 x[CNT][NV];
#pragma unroll
        for (int q = 0; q < CNT; ++q)
#pragma unroll
          for (int kk = 0; kk < NV; ++kk)
            x[q][kk] = load_a(Ab + (int64_t)(r + q) * ldv + (kk < VPT - 1 ? tid + kk * kW64Threads : min(tid + kk * kW64Threads, nvec - 1)));
#pragma unroll
        for (int q = 0; q < CNT; ++q) {
          const double u = us[r + q];
#pragma unroll
          for (int kk = 0; kk < NV; ++kk) {
            acc[kk].x = fma(x[q][kk].x, u, acc[kk].x);
            acc[kk].y = fma(x[q][kk].y, u, acc[kk].y);
          }
        }
      };
      int r = 0;
      for (; r + RB <= nr; r += RB) step(r, std::integral_constant<int, RB>{});
      for (; r < nr; ++r) step(r, std::integral_constant<int, 1>{});
    }
  };
  const bool last = warp * 32 + (VPT - 1) * kW64Threads < nvec;   // this warp owns vectors of the last group

  for (int64_t base = r0; base < r1; base += B) {
    const int nr = (int)min((int64_t)B, r1 - base);
    const double2* Ab = A + base * ldv;
    const double rin = warp == 0 && lane < nr ? row_input(a, base + lane) : 0.0;
    // Few rows: 2, 4, 8 or all warps share one (152 x 10,000, a row per CTA: 13.1 us a pass, 23.2 with a warp a row)
    const int share = nr > 8 ? 1 : (nr > 4 ? 2 : (nr > 2 ? 4 : (nr > 1 ? 8 : 16)));
    if (!nodot && warp < nr * share) {
      if (warp + kW64Warps < nr) {
        const double t = dots(std::integral_constant<int, 2>{}, Ab + warp * ldv, 0, 1);
        if ((lane & 15) == 0) ts[warp + (lane >> 4) * kW64Warps] = t;
      } else {
        const double t = dots(std::integral_constant<int, 1>{}, Ab + warp / share * ldv, warp % share, share);
        if (lane == 0) ts[warp] = t;
      }
    }
    __syncthreads();
    if (warp == 0 && lane < nr) {
      double t = nodot ? 0.0 : ts[lane * share];
      if (!nodot)
        for (int w = 1; w < share; ++w) t += ts[lane * share + w];
      us[lane] = row_phi_d(a, base + lane, t, rin, loss);
      if (!nodot && a.t_out) a.t_out[base + lane] = t;
    }
    __syncthreads();
    if (last) update(std::integral_constant<int, VPT>{}, Ab, nr);
    else update(std::integral_constant<int, VPT - 1>{}, Ab, nr);
  }
  double* part_out = reinterpret_cast<double*>(a.partial) + (int64_t)blockIdx.x * a.dpad;
#pragma unroll
  for (int kk = 0; kk < VPT; ++kk) {
    const int v = tid + kk * kW64Threads;
    if (v < nvec) {
      if (v == tail_vec) acc[kk].y = 0.0;
      *reinterpret_cast<double2*>(part_out + 2 * (int64_t)v) = acc[kk];
    }
  }
  if (a.loss_part && warp == 0) {
    const double l = warp_sum(loss);
    if (lane == 0) a.loss_part[blockIdx.x] = l;
  }
  timer_end(a, ts_slot, NYS_F64);
}

// Column vectors (two values) per thread: up to twelve, 12,288 columns (-1: wider).
int apass_wide64_vpt(int64_t d) {
  const int64_t v = ((d + 1) / 2 + kW64Threads - 1) / kW64Threads;
  return v <= 12 ? (int)v : -1;
}
int apass_wide64_threads() { return kW64Threads; }

namespace {
template <int VPT>
cudaError_t wide64_launch(const ApassKArgs& k, const ApassPlan& plan, cudaStream_t st, bool prepare_only) {
  auto fn = apass_wide64_kernel<VPT>;
  NYS_CUDA_TRY(ensure_max_dyn_smem((const void*)fn, kSmemBudget));
  if (prepare_only) return cudaSuccess;
  count_launch();
  fn<<<plan.grid, kW64Threads, plan.smem, st>>>(k);
  return cudaGetLastError();
}
}  // namespace

cudaError_t apass_wide64_launch(const ApassKArgs& k, const ApassPlan& plan, cudaStream_t st, bool prepare_only) {
  if (plan.rows_per_step < 1 || plan.rows_per_step > 2) return cudaErrorInvalidValue;
  switch (plan.vpt) {
    case 1: return wide64_launch<1>(k, plan, st, prepare_only);
    case 2: return wide64_launch<2>(k, plan, st, prepare_only);
    case 3: return wide64_launch<3>(k, plan, st, prepare_only);
    case 4: return wide64_launch<4>(k, plan, st, prepare_only);
    case 5: return wide64_launch<5>(k, plan, st, prepare_only);
    case 6: return wide64_launch<6>(k, plan, st, prepare_only);
    case 7: return wide64_launch<7>(k, plan, st, prepare_only);
    case 8: return wide64_launch<8>(k, plan, st, prepare_only);
    case 9: return wide64_launch<9>(k, plan, st, prepare_only);
    case 10: return wide64_launch<10>(k, plan, st, prepare_only);
    case 11: return wide64_launch<11>(k, plan, st, prepare_only);
    case 12: return wide64_launch<12>(k, plan, st, prepare_only);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace nys
