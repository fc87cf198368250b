// FP32 start of the symmetric eigensolve of the Nystrom core: an orthogonal V0 that makes
// V0^T G V0 diagonal to FP32 accuracy, from which the FP64 Jacobi sweeps (core.cu) need one or two
// sweeps instead of six to eleven.
//
// A round of the FP64 sweeps costs ~4.3 us whatever the size (grid barrier, L2 loads, the FP64
// square root of the rotation), so a 200 x 200 eigensolve took 9 x 199 of them, 8.1 ms.  Here
// everything stays on chip in FP32: one-sided Jacobi (Hestenes) on the columns of the Cholesky
// factor L of G + eps I in one thread-block cluster, one warp per pair of columns, the columns in
// registers.  A round is three dot products, a rotation and the systolic exchange of the
// round-robin order: each warp passes one column to each neighbour through the neighbour's shared
// memory.  Inside a CTA a round ends with __syncthreads; across CTAs the edge warps send their
// column by st.async, whose arrival an mbarrier at the receiver counts (a cluster barrier per
// round made 200 x 200 1.84 ms and 50 x 50, in one CTA, 0.31; now 1.19 and 0.13).  The left
// singular vectors of L -- the normalised columns at the end -- are the eigenvectors of G, so no
// V is carried, and starting from the Cholesky factor saves a third of the sweeps (Drmac and
// Veselic, SIAM J. Matrix Anal. Appl. 29, 2008).  L is factored in FP64 and rounded, and the
// rotation test is relative, so small eigenpairs are as accurate as large ones; eps = 1e-7
// trace(G) leaves the eigenvectors as they are and keeps a singular G's columns above rounding.
// V0 is then orthonormalised in FP64 (two Newton-Schulz steps: the columns leave the FP32 stage
// orthogonal to 1e-6 .. 1e-4) and checked on the device: if V0^T V0 is off the identity by more
// than 1e-13 the sweeps start from the identity instead, as they do without this stage.
//
// So they do for a steep spectrum (kJacSteep).  Orthonormalising and A = V^T G V are accurate
// relative to lam_1, so what is left of eigenvalue i's row carries eps lam_1 / lam_i, while sweeps from the
// identity keep the relative accuracy of a graded G.  With columns decaying like j^-p, FP64, ranks 100 to 300,
// U^T U - I is 1e-15 .. 3e-13 with this start down to lam_s / lam_1 = 3e-9 (4e-14 .. 2e-7 from the identity),
// but 3e-4 at 2e-10 (1e-6); on rows or columns scaled by 10^+-6, where the ratio is 1e-14 and below, PCG with the
// result no longer converged.  An FP32-class sketch's shift keeps the ratio above 1e-6.
#include <cooperative_groups.h>

#include <algorithm>

#include "device_util.cuh"
#include "nys_internal.cuh"

namespace nys {
namespace {
namespace cg = cooperative_groups;

constexpr double kJacRidge = 1e-7;     // eps / trace(G)
constexpr double kJacSteep = 0x1p-24;  // lam_s / lam_1 below which the sweeps start from the identity
constexpr float kJacSkip2 = 1e-14f;    // squared cosine below which two columns are orthogonal to rounding
constexpr float kJacAgain2 = 1e-6f;    // a sweep that met none above this was the last (quadratic)

// Warp sums of three values, in every lane: a reduce-scatter over the first two lane bits, one
// value per lane after that, and a broadcast of each (9 exchanges for 15).
__device__ __forceinline__ void sum3(float& a, float& b, float& c, int lane) {
  constexpr unsigned F = 0xffffffffu;
  const bool h4 = (lane & 16) != 0, h3 = (lane & 8) != 0;
  // lanes 0-15 go on with (a, b), lanes 16-31 with (c, -)
  float x = (h4 ? c : a) + __shfl_xor_sync(F, h4 ? a : c, 16);
  float y = b + __shfl_xor_sync(F, b, 16);
  // then lanes with bit 3 clear keep x (a or c), the others y (b)
  float v = (h3 ? y : x) + __shfl_xor_sync(F, h3 ? x : y, 8);
  v += __shfl_xor_sync(F, v, 4);
  v += __shfl_xor_sync(F, v, 2);
  v += __shfl_xor_sync(F, v, 1);
  a = __shfl_sync(F, v, 0);
  b = __shfl_sync(F, v, 8);
  c = __shfl_sync(F, v, 16);
}

// A column in a buffer: elements l of the lanes as 16-byte, then 8-byte, then 4-byte words.
template <int NL>
__device__ __forceinline__ void put_column(float* d, const float (&v)[NL], int lane) {
#pragma unroll
  for (int q = 0; q < NL / 4; ++q)
    reinterpret_cast<float4*>(d)[q * 32 + lane] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
  constexpr int R = NL / 4 * 4;
  if constexpr (NL % 4 >= 2) reinterpret_cast<float2*>(d + 32 * R)[lane] = make_float2(v[R], v[R + 1]);
  if constexpr (NL % 2 == 1) d[32 * (NL - 1) + lane] = v[NL - 1];
}
template <int NL>
__device__ __forceinline__ void get_column(const float* d, float (&v)[NL], int lane) {
#pragma unroll
  for (int q = 0; q < NL / 4; ++q) {
    const float4 x = reinterpret_cast<const float4*>(d)[q * 32 + lane];
    v[4 * q] = x.x;
    v[4 * q + 1] = x.y;
    v[4 * q + 2] = x.z;
    v[4 * q + 3] = x.w;
  }
  constexpr int R = NL / 4 * 4;
  if constexpr (NL % 4 >= 2) {
    const float2 x = reinterpret_cast<const float2*>(d + 32 * R)[lane];
    v[R] = x.x;
    v[R + 1] = x.y;
  }
  if constexpr (NL % 2 == 1) v[NL - 1] = d[32 * (NL - 1) + lane];
}
// put_column into another CTA of the cluster: `d` and the mbarrier `bar` there count the bytes.
template <int NL>
__device__ __forceinline__ void send_column(uint32_t d, uint32_t bar, const float (&v)[NL], int lane) {
#pragma unroll
  for (int q = 0; q < NL / 4; ++q)
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(
                     d + (uint32_t)(q * 32 + lane) * 16u),
                 "f"(v[4 * q]), "f"(v[4 * q + 1]), "f"(v[4 * q + 2]), "f"(v[4 * q + 3]), "r"(bar)
                 : "memory");
  constexpr int R = NL / 4 * 4;
  if constexpr (NL % 4 >= 2)
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(
                     d + (uint32_t)(128 * R + 8 * lane)),
                 "f"(v[R]), "f"(v[R + 1]), "r"(bar)
                 : "memory");
  if constexpr (NL % 2 == 1)
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(
                     d + (uint32_t)(128 * (NL - 1) + 4 * lane)),
                 "f"(v[NL - 1]), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ uint32_t cluster_address(uint32_t addr, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// Bounded wait for what other CTAs of the cluster sent.
__device__ __forceinline__ bool cluster_wait(uint64_t* bar, uint32_t parity) {
  const long long t0 = clock64();
  for (;;) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
    if (clock64() - t0 > kWaitCycles) return false;
  }
}

// One-sided Jacobi on the columns of L.  N even; warp m of the cluster holds pair m of H = N / 2;
// NL elements per lane (32 NL >= N).  Shared memory: [2][warps][2][32 NL] exchange buffers
// (t, b).  V (N x N FP64 out, column-major): the normalised columns.  ONE: a single CTA.
//
// Two buffers are enough, inside a CTA and across: round n + 2 overwrites what round n brought, and
// by then the receiver has passed its round n + 1 on (__syncthreads, or the column that comes back
// from it: neighbours always exchange both ways).
template <int NL, bool ONE>
__global__ void jacobi32_kernel(const float* __restrict__ L, int N, double* __restrict__ V, int max_sweeps) {
  extern __shared__ __align__(16) float xbuf[];
  __shared__ int flag[3];
  __shared__ __align__(8) uint64_t in_bar[2][2];   // [from the CTA before / after][buffer]
  cg::cluster_group cl = cg::this_cluster();
  const int wpc = blockDim.x >> 5;
  const int rank = ONE ? 0 : (int)cl.block_rank();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int H = N / 2, m = rank * wpc + warp;
  const bool on = m < H;
  constexpr int LEN = 32 * NL;
  const bool before = !ONE && on && warp == 0 && m >= 1;             // neighbour m - 1 in another CTA
  const bool after = !ONE && on && warp == wpc - 1 && m < H - 1;     // neighbour m + 1
  if (threadIdx.x < 3) flag[threadIdx.x] = 0;
  if (threadIdx.x == 0) {
    for (int q = 0; q < 4; ++q) mbar_init(&in_bar[q >> 1][q & 1], 1);
    fence_mbar_init();
  }
  // pair m starts with columns m and N - 1 - m
  float t[NL], b[NL];
#pragma unroll
  for (int l = 0; l < NL; ++l) {
    const int i = l * 32 + lane;
    t[l] = on && i < N ? L[i + (int64_t)m * N] : 0.f;
    b[l] = on && i < N ? L[i + (int64_t)(N - 1 - m) * N] : 0.f;
  }
  // where this warp's columns go after a round: t to pair m + 1's t (pair 0 keeps it; the last
  // pair's becomes its own b), b to pair m - 1's b (pair 0's becomes pair 1's t)
  auto slot = [&](int w, int buf, int part) -> float* { return xbuf + ((buf * wpc + w) * 2 + part) * LEN; };
  int* flags0 = flag;
  if constexpr (ONE) {
    __syncthreads();
  } else {
    flags0 = cl.map_shared_rank(flag, 0);
    cl.sync();
  }
  int round = 0;
  bool lost = false;   // a wait gave up: the result will not pass its check
  for (int sweep = 0; sweep < max_sweeps && H > 1; ++sweep) {
    if (rank == 0 && threadIdx.x == 0) flag[(sweep + 1) % 3] = 0;
    bool again = false;
    for (int r = 0; r < N - 1; ++r, ++round) {
      const int buf = round & 1;
      if (on) {
        float a = 0.f, c2 = 0.f, g = 0.f;
#pragma unroll
        for (int l = 0; l < NL; ++l) {
          a = fmaf(t[l], t[l], a);
          c2 = fmaf(b[l], b[l], c2);
          g = fmaf(t[l], b[l], g);
        }
        sum3(a, c2, g, lane);
        const float ab = a * c2, gg = g * g;
        if (gg > kJacSkip2 * ab) {
          if (gg > kJacAgain2 * ab) again = true;
          // the smaller root, by h = |b|^2 - |t|^2, r = sqrt(h^2 + 4 g^2): c^2 = (1 + |h| / r) / 2,
          // s = sign(h g) |g| / (r c): two reciprocal square roots and a reciprocal
          const float h = c2 - a, g2 = 2.f * g;
          const float ir = rsqrtf(fmaf(h, h, g2 * g2));
          const float cc = fmaf(0.5f * fabsf(h), ir, 0.5f);
          const float ic = rsqrtf(cc);
          const float sn = 0.5f * ic * ir * (h < 0.f ? -g2 : g2);
          // Rutishauser's form: the rounding of a rotation shrinks with its angle, so the
          // columns' lengths do not drift over the two thousand rounds
          const float tau = __fdividef(sn, fmaf(cc, ic, 1.f));
#pragma unroll
          for (int l = 0; l < NL; ++l) {
            const float x = t[l], y = b[l];
            t[l] = fmaf(-sn, fmaf(tau, x, y), x);
            b[l] = fmaf(sn, fmaf(-tau, y, x), y);
          }
        }
        if (before)
          send_column<NL>(cluster_address(smem_u32(slot(wpc - 1, buf, 1)), rank - 1),
                          cluster_address(smem_u32(&in_bar[1][buf]), rank - 1), b, lane);
        else if (m >= 1)
          put_column<NL>(slot(warp - 1, buf, 1), b, lane);
        if (after)
          send_column<NL>(cluster_address(smem_u32(slot(0, buf, 0)), rank + 1),
                          cluster_address(smem_u32(&in_bar[0][buf]), rank + 1), t, lane);
        else if (m == 0)
          put_column<NL>(slot(1, buf, 0), b, lane);
        else if (m < H - 1)
          put_column<NL>(slot(warp + 1, buf, 0), t, lane);
        if (lane == 0) {
          if (before) mbar_arrive_expect_tx(&in_bar[0][buf], LEN * 4);
          if (after) mbar_arrive_expect_tx(&in_bar[1][buf], LEN * 4);
        }
      }
      if (r == N - 2 && again && lane == 0) flags0[sweep % 3] = 1;
      __syncthreads();
      if (!ONE && on && !lost) {
        const uint32_t ph = (uint32_t)((round >> 1) & 1);
        if (before && !cluster_wait(&in_bar[0][buf], ph)) lost = true;
        if (after && !cluster_wait(&in_bar[1][buf], ph)) lost = true;
        lost = __any_sync(0xffffffffu, lost);
      }
      if (on) {
        if (m == H - 1) {
#pragma unroll
          for (int l = 0; l < NL; ++l) b[l] = t[l];
        } else {
          get_column<NL>(slot(warp, buf, 1), b, lane);
        }
        if (m >= 1) get_column<NL>(slot(warp, buf, 0), t, lane);
      }
    }
    if constexpr (!ONE) cl.sync();   // every CTA's flag
    if (*(volatile int*)(flags0 + sweep % 3) == 0) break;
  }
  if (on) {
    float a = 0.f, c2 = 0.f;
#pragma unroll
    for (int l = 0; l < NL; ++l) {
      a = fmaf(t[l], t[l], a);
      c2 = fmaf(b[l], b[l], c2);
    }
    a = warp_sum(a);
    c2 = warp_sum(c2);
    const float ia = a > 0.f ? rsqrtf(a) : 0.f, ib = c2 > 0.f ? rsqrtf(c2) : 0.f;
#pragma unroll
    for (int l = 0; l < NL; ++l) {
      const int i = l * 32 + lane;
      if (i < N) {
        V[i + (int64_t)(2 * m) * N] = (double)(t[l] * ia);
        V[i + (int64_t)(2 * m + 1) * N] = (double)(b[l] * ib);
      }
    }
  }
  if constexpr (!ONE) cl.sync();   // no CTA leaves while another may still read its flag
}

// S <- 1.5 I - 0.5 S (the factor of the Newton-Schulz step V <- V (1.5 I - 0.5 V^T V))
__global__ void schulz_kernel(double* __restrict__ S, int N) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < (int64_t)N * N; e += (int64_t)gridDim.x * blockDim.x)
    S[e] = (e % N == e / N ? 1.5 : 0.0) - 0.5 * S[e];
}
// *bad |= any |S - I| > tol (or NaN)
__global__ void gap_kernel(const double* __restrict__ S, int N, double tol, int* bad) {
  int b = 0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < (int64_t)N * N; e += (int64_t)gridDim.x * blockDim.x)
    b |= !(fabs(S[e] - (e % N == e / N ? 1.0 : 0.0)) <= tol);
  if (__syncthreads_or(b) && threadIdx.x == 0) atomicOr(bad, 1);
}
// bad[1] = the spectrum on the diagonal of T = V^T G V is steep.  The padding row's own eigenvector (N > s), if
// any, is left out.
__global__ void __launch_bounds__(512) steep_kernel(const double* __restrict__ T, const double* __restrict__ V, int N, int s,
                                                    int* bad) {
  __shared__ double lo[16], hi[16];
  double mn = INFINITY, mx = 0.0;
  for (int i = threadIdx.x; i < N; i += 512)
    if (N == s || fabs(V[(N - 1) + (int64_t)i * N]) < 0.5) {
      const double t = T[i + (int64_t)i * N];
      mn = fmin(mn, t);
      mx = fmax(mx, t);
    }
  for (int o = 16; o > 0; o >>= 1) {
    mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, o));
    mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  if ((threadIdx.x & 31) == 0) {
    lo[threadIdx.x >> 5] = mn;
    hi[threadIdx.x >> 5] = mx;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 16; ++w) {
      mn = fmin(mn, lo[w]);
      mx = fmax(mx, hi[w]);
    }
    bad[1] = !(mn >= kJacSteep * mx);
  }
}
// A <- (T + T^T) / 2, V <- Vn; when Vn failed its check (bad[0]) or the spectrum is steep (bad[1]) A stays, and V too
// (V = I with `reset`).  Vn may be V.
__global__ void accept_kernel(const double* __restrict__ T, int N, const int* __restrict__ bad, int reset,
                              double* __restrict__ A, const double* Vn, double* V) {
  const bool no = (bad[0] | bad[1]) != 0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < (int64_t)N * N; e += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(e % N), j = (int)(e / N);
    if (no) {
      if (reset) V[e] = i == j ? 1.0 : 0.0;
    } else {
      A[e] = 0.5 * (T[i + (int64_t)j * N] + T[j + (int64_t)i * N]);
      if (Vn != V) V[e] = Vn[e];
    }
  }
}
__global__ void fill_kernel(unsigned* x, int n, unsigned v) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) x[i] = v;
}

// E <- E_ij = A_ij / (A_jj - A_ii), antisymmetric, zero where it is not small (a near-degenerate pair)
__global__ void first_order_kernel(const double* __restrict__ A, int N, double* __restrict__ E) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < (int64_t)N * N; e += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(e % N), j = (int)(e / N);
    const double h = A[j + (int64_t)j * N] - A[i + (int64_t)i * N];
    const double g = 0.5 * (A[e] + A[j + (int64_t)i * N]);
    E[e] = i != j && fabs(g) <= 2e-3 * fabs(h) && h != 0.0 ? g / h : 0.0;
  }
}
// U = I + E + E2 / 2
__global__ void exp2_kernel(const double* __restrict__ E, const double* __restrict__ E2, int N, double* __restrict__ U) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < (int64_t)N * N; e += (int64_t)gridDim.x * blockDim.x)
    U[e] = (e % N == e / N ? 1.0 : 0.0) + E[e] + 0.5 * E2[e];
}
// Z = op(X) Y for N x N column-major matrices, op the transpose with kc.  Up to kSmallProduct on the FP64
// pipe, a 16 x 16 tile per CTA (100 x 100: 49 CTAs, 6 us; the tensor-core product's stages and
// split take ~17 us there), beyond as the FP64 product on the tensor cores (200 x 200: ~20 us
// either way, 320: 30 for 60).  ex, ey: exponents of op(X)'s rows and Y's columns (tensor cores).
constexpr int kSmallProduct = 128;
__global__ void __launch_bounds__(256) small_product_kernel(const double* __restrict__ X, int kc,
                                                            const double* __restrict__ Y, double* __restrict__ Z, int N) {
  __shared__ double As[16][17], Bs[16][17];   // [k][m], [k][n]
  const int lo = threadIdx.x & 15, hi = threadIdx.x >> 4;
  const int m0 = blockIdx.x * 16, n0 = blockIdx.y * 16;
  auto load = [&](int k0, double& a, double& b) {
    // kc: K runs along X's columns' storage
    const int am = m0 + (kc ? hi : lo), ak = k0 + (kc ? lo : hi), bn = n0 + hi, bk = k0 + lo;
    a = am < N && ak < N ? X[kc ? (int64_t)am * N + ak : (int64_t)ak * N + am] : 0.0;
    b = bn < N && bk < N ? Y[(int64_t)bn * N + bk] : 0.0;
  };
  double a, b, acc = 0.0;
  load(0, a, b);
  for (int k0 = 0; k0 < N; k0 += 16) {
    if (kc) As[lo][hi] = a;
    else As[hi][lo] = a;
    Bs[lo][hi] = b;
    __syncthreads();
    if (k0 + 16 < N) load(k0 + 16, a, b);
#pragma unroll
    for (int k = 0; k < 16; ++k) acc = fma(As[k][lo], Bs[k][hi], acc);
    __syncthreads();
  }
  if (m0 + lo < N && n0 + hi < N) Z[(int64_t)(n0 + hi) * N + m0 + lo] = acc;
}
cudaError_t square_product(const double* X, bool kc, const unsigned* ex, const double* Y, const unsigned* ey, double* Z,
                           int N, void* gw, int* status, cudaStream_t st) {
  if (N > kSmallProduct) return gemm64(X, kc, N, ex, N, Y, N, ey, N, N, nullptr, Z, N, gw, status, st, false);
  count_launch();
  small_product_kernel<<<dim3((N + 15) / 16, (N + 15) / 16), 256, 0, st>>>(X, kc ? 1 : 0, Y, Z, N);
  return cudaGetLastError();
}

// Cluster shape: one CTA while its 32 warps hold every pair, else eight CTAs.
int jac_ctas(int H) { return H <= 32 ? 1 : 8; }

template <int NL, bool ONE>
cudaError_t launch_jacobi32_ctas(const float* L, int N, double* V, cudaStream_t st, bool* ran) {
  const int H = N / 2, C = jac_ctas(H), wpc = (H + C - 1) / C;
  const size_t smem = (size_t)2 * wpc * 2 * 32 * NL * sizeof(float);
  NYS_CUDA_TRY(ensure_max_dyn_smem((const void*)jacobi32_kernel<NL, ONE>, 200 * 1024));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)C);
  cfg.blockDim = dim3((unsigned)(32 * wpc));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = ONE ? 0 : 1;
  int n_clusters = 0;
  if (!ONE && (cudaOccupancyMaxActiveClusters(&n_clusters, jacobi32_kernel<NL, ONE>, &cfg) != cudaSuccess || n_clusters < 1)) {
    (void)cudaGetLastError();
    *ran = false;   // the cluster does not fit this device: the FP64 sweeps start from the identity
    return cudaSuccess;
  }
  count_launch();
  *ran = true;
  return cudaLaunchKernelEx(&cfg, jacobi32_kernel<NL, ONE>, L, N, V, 12);
}
template <int NL>
cudaError_t launch_jacobi32(const float* L, int N, double* V, cudaStream_t st, bool* ran) {
  if constexpr (NL <= 2)   // 32 pairs at most
    return launch_jacobi32_ctas<NL, true>(L, N, V, st, ran);
  else
    return launch_jacobi32_ctas<NL, false>(L, N, V, st, ran);
}

size_t up256(size_t b) { return (b + 255) / 256 * 256; }

}  // namespace

// Ranks the start covers: 10 elements per lane, the warps of 320 columns in eight CTAs.
bool jacobi_start_supported(int s) { return s >= 8 && s <= 320; }

// Scratch of the start and of the correction: two N x N matrices, exponents, the products' own.
namespace {
struct StartWork {
  double *S, *P;
  unsigned *e1, *eg, *et;   // exponents: of entries below 4, of G's rows, of a product's columns
  int* bad;                 // the check of V; a steep spectrum (of the start, kept through the corrections)
  void* gw;
  StartWork(void* work, int N) {
    unsigned char* b = reinterpret_cast<unsigned char*>(work);
    const size_t m = up256((size_t)N * N * sizeof(double));
    S = reinterpret_cast<double*>(b);
    P = reinterpret_cast<double*>(b + m);
    e1 = reinterpret_cast<unsigned*>(b + 2 * m);
    eg = e1 + N;
    et = eg + N;
    bad = reinterpret_cast<int*>(et + N);
    gw = b + 2 * m + up256(3 * (size_t)N * sizeof(unsigned) + 2 * sizeof(int));
  }
};
}  // namespace

size_t jacobi_start_work_bytes(int s) {
  const size_t N = s + (s & 1);
  return 2 * up256(N * N * sizeof(double)) + up256(3 * N * sizeof(unsigned) + 2 * sizeof(int)) +
         gemm64_work_bytes(N, (int)N, N);
}

cudaError_t jacobi_start(const double* G, int s, double* A, double* V, void* work, int* status, cudaStream_t st,
                         bool* ran) {
  const int N = s + (s & 1);
  const int64_t nn = (int64_t)N * N;
  const StartWork w(work, N);
  float* L = reinterpret_cast<float*>(w.S);
  NYS_CUDA_TRY(chol_lower_f32(G, s, kJacRidge, L, N, st));
  // two orthonormalisation steps, V -> P -> V
  if (N <= 64) NYS_CUDA_TRY(launch_jacobi32<2>(L, N, V, st, ran));
  else if (N <= 128) NYS_CUDA_TRY(launch_jacobi32<4>(L, N, V, st, ran));
  else if (N <= 224) NYS_CUDA_TRY(launch_jacobi32<7>(L, N, V, st, ran));
  else NYS_CUDA_TRY(launch_jacobi32<10>(L, N, V, st, ran));
  if (!*ran) return cudaSuccess;
  const unsigned grid = (unsigned)std::min<int64_t>(1024, (nn + 255) / 256);
  count_launch();
  fill_kernel<<<(N + 127) / 128, 128, 0, st>>>(w.e1, N, 0x40000000u);
  NYS_CUDA_TRY(cudaMemsetAsync(w.bad, 0, sizeof(int), st));
  auto mul = [&](const double* X, bool kc, const unsigned* ex, const double* Y, const unsigned* ey, double* Z) {
    return square_product(X, kc, ex, Y, ey, Z, N, w.gw, status, st);
  };
  double *cur = V, *nxt = w.P;
  for (int k = 0; k < 2; ++k) {
    NYS_CUDA_TRY(mul(cur, true, w.e1, cur, w.e1, w.S));
    count_launch();
    schulz_kernel<<<grid, 256, 0, st>>>(w.S, N);
    NYS_CUDA_TRY(cudaGetLastError());
    NYS_CUDA_TRY(mul(cur, false, w.e1, w.S, w.e1, nxt));
    std::swap(cur, nxt);
  }
  NYS_CUDA_TRY(mul(V, true, w.e1, V, w.e1, w.S));
  count_launch();
  gap_kernel<<<grid, 256, 0, st>>>(w.S, N, 1e-13, w.bad);
  NYS_CUDA_TRY(cudaGetLastError());
  // A <- V^T A V
  if (N > kSmallProduct) NYS_CUDA_TRY(absmax_f64(A, N, N, N, w.eg, nullptr, st));
  NYS_CUDA_TRY(mul(A, true, w.eg, V, w.e1, w.S));
  if (N > kSmallProduct) NYS_CUDA_TRY(absmax_f64(w.S, N, N, N, w.et, nullptr, st));
  NYS_CUDA_TRY(mul(V, true, w.e1, w.S, w.et, w.P));
  count_launch();
  steep_kernel<<<1, 512, 0, st>>>(w.P, V, N, s, w.bad);
  NYS_CUDA_TRY(cudaGetLastError());
  count_launch();
  accept_kernel<<<grid, 256, 0, st>>>(w.P, N, w.bad, 1, A, V, V);
  return cudaGetLastError();
}

cudaError_t jacobi_polish(const double* G, int N, double* A, double* T, double* V, void* work, int* status,
                          cudaStream_t st) {
  const int64_t nn = (int64_t)N * N;
  const StartWork w(work, N);   // e1 and eg as jacobi_start left them
  const unsigned grid = (unsigned)std::min<int64_t>(1024, (nn + 255) / 256);
  auto mul = [&](const double* X, bool kc, const unsigned* ex, const double* Y, const unsigned* ey, double* Z) {
    return square_product(X, kc, ex, Y, ey, Z, N, w.gw, status, st);
  };
  // exp(E) to second order, its departure from orthogonality (E^4 / 4) squared away by one
  // Newton-Schulz step; checked like the start's V, and left out when it fails
  NYS_CUDA_TRY(cudaMemsetAsync(w.bad, 0, sizeof(int), st));
  count_launch();
  first_order_kernel<<<grid, 256, 0, st>>>(A, N, w.S);
  NYS_CUDA_TRY(mul(w.S, false, w.e1, w.S, w.e1, w.P));
  count_launch();
  exp2_kernel<<<grid, 256, 0, st>>>(w.S, w.P, N, w.S);
  NYS_CUDA_TRY(mul(V, false, w.e1, w.S, w.e1, w.P));
  NYS_CUDA_TRY(mul(w.P, true, w.e1, w.P, w.e1, w.S));
  count_launch();
  schulz_kernel<<<grid, 256, 0, st>>>(w.S, N);
  NYS_CUDA_TRY(cudaGetLastError());
  NYS_CUDA_TRY(mul(w.P, false, w.e1, w.S, w.e1, T));
  NYS_CUDA_TRY(mul(T, true, w.e1, T, w.e1, w.S));
  count_launch();
  gap_kernel<<<grid, 256, 0, st>>>(w.S, N, 1e-13, w.bad);
  NYS_CUDA_TRY(cudaGetLastError());
  NYS_CUDA_TRY(mul(G, true, w.eg, T, w.e1, w.S));
  if (N > kSmallProduct) NYS_CUDA_TRY(absmax_f64(w.S, N, N, N, w.et, nullptr, st));
  NYS_CUDA_TRY(mul(T, true, w.e1, w.S, w.et, w.P));
  count_launch();
  accept_kernel<<<grid, 256, 0, st>>>(w.P, N, w.bad, 0, A, T, V);
  return cudaGetLastError();
}

}  // namespace nys
