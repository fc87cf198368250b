// FP64 matrix products on the FP16 tensor cores.
//
//   C (M x N) = diag(D) A B^T,   A(m, k), B(n, k) FP64
//
// GB300's FP64 pipe retires about 2 FMA per clock and SM; its tensor cores ~3,400 MAC.
// Each operand row is written in fixed point relative to its own largest exponent, as eight
// signed 8-bit digits (62 bits below the row's maximum):
//   A(m, k) = 2^(ea_m - 1084) sum_i a_i 256^(7 - i),  a_i in [-128, 127] (exact in FP16),
// so a product of digits is an integer of at most 2^14, and the tensor core's FP32
// accumulators add them exactly while |sum| < 2^24.  The digit products of equal weight
// (order o = i + j = 0 .. 7, o + 1 pairs) share one TMEM accumulator: 36 MMAs per K step for
// 64 output columns x 8 orders = all 512 TMEM columns.  Every 256 K the accumulators are read
// out as integers and added to a 96-bit integer sum per output.  In 256 K orders 0-4 cannot leave 2^24 for
// any input; orders 5-7 can in the last MMAs of a group whose digits are nearly all at their largest and of
// one sign (sum |a||b| is above 2^-4 2^ea 2^eb then), and round by at most 2^-47 2^ea 2^eb, less than
// a chain of FMAs there.  The final integer is rounded to FP64 once.
// (Fixed-point splitting of a product into exact low-precision ones: Ozaki, Ogita, Oishi, Rump,
// Numer. Algorithms 59, 2012.)
//
// Error: with |a| < 2 x 2^ea and |b| < 2 x 2^eb over the rows, cutting the digits off (toward zero, below
// 2^-61) and dropping the orders from 8 on (order 8: 7 x 2^-60) leaves at most
//   9.1 K 2^-60 2^ea 2^eb + 2^-53 |C|,
// which is relative to the rows' largest entries, not to the entries that meet: where large ones of A only
// meet small ones of B a chain of FMAs, K 2^-53 sum |a||b|, is better, by any factor.  So for products
// with a caller's matrix (hmm64) gemm64_check_kernel first finds the outputs with sum |a||b| <
// 9.1/128 2^ea 2^eb, where the FMAs' bound is the smaller, and this kernel forms those (in columns of 32 rows)
// by FMAs.  Of A Omega and A^T W with columns decaying like 1/j there are none, with 1/j^2 5 % of the
// columns; rows scaled against their weights have all.  (Sketch of 40,000 x 4,000, rank 100: 6.6 ms, 0.1 of it the
// check; 13 with columns like 1/j^2, 44 with the rows so scaled; 83 on the FP64 pipe alone.)
//
// Measured (FP64 pipe before, this kernel after): the two products of a 40,000 x 4,000 sketch of
// rank 100, 36.1 + 40.4 ms -> 1.7 + 1.7 ms; X^T Y at 10,000 x 200, 0.52 (symmetric) and 0.90 ms
// -> 0.1 ms; U = B V at 10,000 x 200, 1.09 -> 0.05 ms.
//
// What bounds it: per 32 K a tile makes the digits of 6,144 elements (~40 integer operations each at
// 64 lanes per clock: 3,900 clocks) and issues 72 MMAs (multiplying takes 2,300, reading A and B
// from shared memory 3,500); together it takes 6,100.  So sixteen warps convert, one thread
// issues the MMAs, and they meet only through mbarriers; the read-out of a 256-K group runs after
// the next stage's digits are written; MMAs that share an A tile follow each other and keep it
// in the collector; a digit is one byte in the significand of an FP16 number and one
// subtraction (in BF16 pairs: three integer operations more per two digits, 8 % of the kernel).
// (One warp doing both and a barrier per stage: 9,200 clocks, tensor pipe 26 % active.)  Both
// operands are converted in the kernel: the digits are never written to memory, and an operand
// stored along M (A^T) is transposed on the way into shared memory.
#include <cooperative_groups.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "solver.cuh"
#include "tc_ptx.cuh"

namespace nys {
namespace {

constexpr int EM = 128, EN = 64, EK = 32;     // tile and K of one stage
constexpr int ECW = 16;                       // converting warps
constexpr int ET = 32 * (ECW + 4);            // and a warpgroup of which one thread issues the MMAs
constexpr int ESL = 8;                        // digits per operand = orders kept
constexpr int EFLUSH = 8;                     // stages between read-outs (256 K)
constexpr uint32_t EA_SLICE = EM * EK * 2, EB_SLICE = EN * EK * 2;
constexpr uint32_t E_STAGE = ESL * (EA_SLICE + EB_SLICE);   // 96 KB
constexpr int E_MINSTEPS = 2;                 // K steps a split slice has at least
constexpr int ESPREAD = (EM / 32) * (EN / 8); // bytes of a tile in EmuArgs::spread

struct EmuArgs {
  const double* A;
  int64_t lda;
  const unsigned* ea;   // per row m: top word of its largest magnitude (exponent in bits 20-30)
  const double* B;
  int64_t ldb;
  const unsigned* eb;
  int64_t M, K, kslice;
  int N;
  const double* D;      // row factors, applied when the K range is not split
  double* C;            // slice z at C + z * cslice, column n at + n * ldc
  int64_t ldc, cslice;
  // which outputs the FMAs form: per tile 4 x 8 bytes, bit n % 8 of byte (m / 32, n / 8) for column n of the
  // 32 rows; or null (none)
  unsigned char* spread;
  int* status;
};

// Fixed-point value of x at the scale of its row (largest exponent field emax), each byte the
// digit + 128: (lo, hi) words.
__device__ __forceinline__ void digits(double x, int emax, uint32_t& lo, uint32_t& hi) {
  const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
  const int e = (int)((h >> 20) & 0x7ffu);
  // significand at bits 9 .. 61 (its leading one, implicit unless e = 0, at 61)
  uint32_t mh = (__funnelshift_l(l, h, 9) & 0x1fffffffu) | 0x20000000u;
  int sh = min(emax - e, 63);   // 62 bits shifted by 62 or more are zero: no test for e = 0, unless
  if (emax < 64) {              // the row's maximum is itself within 2^64 of the denormals
    if (e == 0) mh &= 0x1fffffffu;
    sh = emax - max(e, 1);
  }
  if (sh < 0) sh = 63;          // a value above its row's bound: only where the caller discards the result
  const uint64_t q = (((uint64_t)mh << 32) | (uint64_t)(l << 9)) >> sh;
  const uint32_t sg = (uint32_t)((int)h >> 31);
  const uint32_t a = (uint32_t)q ^ sg, c = (uint32_t)(q >> 32) ^ sg;
  asm("add.cc.u32 %0, %2, %3;\n addc.u32 %1, %4, 0x80808080;" : "=r"(lo), "=r"(hi) : "r"(a), "r"(0x80808080u - sg), "r"(c));
}

// The four digits of a word of two biased values as FP16 pairs, lowest byte first: 1,024 + (d + 128)
// is the FP16 number 0x6400 | byte, so a byte needs no more than its place and one subtraction.
__device__ __forceinline__ void digit_pairs(uint32_t x0, uint32_t x1, uint32_t (&d)[4]) {
  const uint32_t lo = __byte_perm(x0, x1, 0x5140), hi = __byte_perm(x0, x1, 0x7362);   // bytes 0 0' 1 1', 2 2' 3 3'
  const uint32_t m = 0x64646464u, off = 0x64806480u;                                   // off: 1,152 twice
  const uint32_t p[4] = {__byte_perm(lo, m, 0x4140), __byte_perm(lo, m, 0x4342), __byte_perm(hi, m, 0x4140),
                         __byte_perm(hi, m, 0x4342)};
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const __half2 r = __hsub2(*reinterpret_cast<const __half2*>(&p[b]), *reinterpret_cast<const __half2*>(&off));
    d[b] = *reinterpret_cast<const uint32_t*>(&r);
  }
}

// v 2^sh rounded once to FP64 (to nearest, ties to even).
__device__ __forceinline__ double fixed_to_double(__int128 v, int sh) {
  if (v == 0) return 0.0;
  const bool neg = v < 0;
  unsigned __int128 u = neg ? (unsigned __int128)(-v) : (unsigned __int128)v;
  const uint64_t uh = (uint64_t)(u >> 64);
  const int lz = uh ? __clzll((long long)uh) : 64 + __clzll((long long)(uint64_t)u);
  u <<= lz;
  const uint64_t top = (uint64_t)(u >> 64);
  const bool sticky = (uint64_t)u != 0;
  uint64_t m = top >> 11;
  const uint32_t r = (uint32_t)(top & 0x7ffu);
  if (r > 0x400u || (r == 0x400u && (sticky || (m & 1)))) ++m;
  int e = 127 + sh - lz;
  if (m >> 53) {
    m >>= 1;
    ++e;
  }
  double x;
  if (e > 1023) x = __longlong_as_double(0x7ff0000000000000ll);
  else if (e < -1022) x = scalbn((double)m, e - 52);
  else x = __longlong_as_double((long long)(((uint64_t)(e + 1023) << 52) | (m & 0xfffffffffffffull)));
  return neg ? -x : x;
}

// C(m, n) over [kb, ke) by FMAs in increasing k for m = mb + lane and the columns n = nb + (bits of `cols`);
// of two warps, `part` takes every other column.  Four columns at a time; A(m, k) from each lane's own row or column,
// eight K ahead of their use, B(n, k) by lanes over k.  Bound by the FP64 pipe where all columns are formed here, by
// latency where a few are.  Zeros in B (triangular factors) are passed over while A is finite.
template <bool KC>
__device__ __forceinline__ void fma_columns(const EmuArgs& a, int64_t mb, int nb, uint32_t cols, int part, int64_t kb, int64_t ke) {
  constexpr int AHEAD = 8;
  const int lane = threadIdx.x & 31;
  const int64_t m = mb + lane;
  const bool mok = m < a.M;
  const double* Ap = KC ? a.A + (mok ? m : 0) * a.lda : a.A + (mok ? m : 0);
  const int64_t step = KC ? 1 : a.lda;
  const bool finite = !__any_sync(0xffffffffu, mok && (a.ea[m] >> 20) == 0x7ffu);
  const double dm = a.D && mok ? a.D[m] : 1.0;
  double* out = a.C + (int64_t)blockIdx.z * a.cslice + m;
  if (part && cols) cols &= cols - 1;
  while (cols) {
    int n[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      n[j] = cols ? nb + __ffs(cols) - 1 : -1;
      cols &= cols - 1;   // this one
      cols &= cols - 1;   // the other warp's
    }
    double acc[4] = {0.0, 0.0, 0.0, 0.0}, bn[4];
    auto load_b = [&](int64_t k0) {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        bn[j] = n[j] >= 0 && k0 + lane < ke ? __ldg(a.B + (int64_t)n[j] * a.ldb + k0 + lane) : 0.0;
    };
    load_b(kb);
    for (int64_t k0 = kb; k0 < ke; k0 += 32) {
      double bv[4];
      uint32_t some = 0u;   // the K that count
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        bv[j] = bn[j];
        some |= __ballot_sync(0xffffffffu, bv[j] != 0.0);
      }
      if (k0 + 32 < ke) load_b(k0 + 32);
      if (!finite) some = ke - k0 >= 32 ? 0xffffffffu : (1u << (ke - k0)) - 1u;
      const double* Ak = Ap + k0 * step;
      uint32_t ahead = some;
      double an[AHEAD];
      auto load_a = [&]() {
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) {
          an[u] = ahead && mok ? __ldg(Ak + (__ffs(ahead) - 1) * step) : 0.0;
          ahead &= ahead - 1;
        }
      };
      load_a();
      while (some) {
        double av[AHEAD];
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) av[u] = an[u];
        if (ahead) load_a();
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) {
          if (some) {
            const int k = __ffs(some) - 1;
            some &= some - 1;
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[j] = fma(av[u], __shfl_sync(0xffffffffu, bv[j], k), acc[j]);
          }
        }
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (mok && n[j] >= 0) out[(int64_t)n[j] * a.ldc] = a.D ? dm * acc[j] : acc[j];
  }
}

// KC: A(m, k) = A[m lda + k]; else A(m, k) = A[k lda + m].  B(n, k) = B[n ldb + k].
template <bool KC>
__global__ void __launch_bounds__(ET, 1) gemm64_tc_kernel(const EmuArgs a) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t full_bar[2], empty_bar[2], drained, done;
  __shared__ volatile int s_fail;
  __shared__ uint32_t tmem_slot;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t m0 = (int64_t)blockIdx.y * EM;
  const int n0 = blockIdx.x * EN;
  const int64_t kb = (int64_t)blockIdx.z * a.kslice, ke = min(a.K, kb + a.kslice);
  const uint32_t* spread =
      a.spread ? reinterpret_cast<const uint32_t*>(a.spread) + ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * (ESPREAD / 4)
               : nullptr;
  int nt = (int)((ke - kb + EK - 1) / EK);
  if (spread) {   // a tile all of FMAs needs no digits
    bool all = true;
    for (int w = 0; w < ESPREAD / 4; ++w) {
      const int nv = min(32, max(0, a.N - n0 - 32 * (w & 1)));
      if (m0 + 32 * (w >> 1) < a.M && nv > 0) all = all && spread[w] == 0xffffffffu >> (32 - nv);
    }
    if (all) nt = 0;
  }
  const uint32_t sbase = smem_u32(smem);
  if (warp == 0) {
    tmem_alloc(&tmem_slot, 512);
    tmem_relinquish();
  }
  if (tid == 0) {
    for (int q = 0; q < 2; ++q) {
      mbar_init(&full_bar[q], ECW);
      mbar_init(&empty_bar[q], 1);
    }
    mbar_init(&drained, ECW);
    mbar_init(&done, 1);
    s_fail = 0;
    fence_mbar_init();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  // Conversion: this thread's chunk of A is row ar, K 8 ac .. + 7 of a stage; its half chunk of
  // B is row br, K 4 bc .. + 3.  Lanes run over the rows of a core matrix (8 rows x 16 bytes),
  // so the 16-byte stores of eight lanes fill one.
  int ar, ac;
  if (KC) {
    ar = (8 * warp + (lane & 7)) % EM;
    ac = lane >> 3;
  } else {
    ar = 32 * (warp & 3) + lane;
    ac = warp >> 2;
  }
  // (B: 16 lanes fill the two halves of eight rows; the issuing warpgroup converts nothing)
  const int br = (8 * (warp >> 1) + ((lane >> 1) & 7)) % EN, bc = 2 * (2 * (warp & 1) + (lane >> 4)) + (lane & 1);
  const int64_t am = m0 + ar;
  const bool aok = am < a.M, bok = n0 + br < a.N;
  const int emA = aok ? max(1, (int)(a.ea[am] >> 20)) : 1;
  const int emB = bok ? max(1, (int)(a.eb[n0 + br] >> 20)) : 1;
  const double* Ap = KC ? a.A + (aok ? am : 0) * a.lda : a.A + (aok ? am : 0);
  const double* Bp = a.B + (int64_t)(bok ? n0 + br : 0) * a.ldb;
  const bool avec = KC && (a.lda & 1) == 0 && (reinterpret_cast<uintptr_t>(a.A) & 15u) == 0 && (kb & 1) == 0;
  const bool bvec = (a.ldb & 1) == 0 && (reinterpret_cast<uintptr_t>(a.B) & 15u) == 0 && (kb & 1) == 0;
  double ra[8], rb[4];
  auto load = [&](int t) {
    const int64_t ka = kb + (int64_t)t * EK + 8 * ac, kk = kb + (int64_t)t * EK + 4 * bc;
    if (KC && avec && aok && ka + 8 <= ke) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const double2 v = __ldg(reinterpret_cast<const double2*>(Ap + ka) + e);
        ra[2 * e] = v.x;
        ra[2 * e + 1] = v.y;
      }
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e)
        ra[e] = (aok && ka + e < ke) ? __ldg(KC ? Ap + ka + e : Ap + (ka + e) * a.lda) : 0.0;
    }
    if (bvec && bok && kk + 4 <= ke) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const double2 v = __ldg(reinterpret_cast<const double2*>(Bp + kk) + e);
        rb[2 * e] = v.x;
        rb[2 * e + 1] = v.y;
      }
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) rb[e] = (bok && kk + e < ke) ? __ldg(Bp + kk + e) : 0.0;
    }
  };
  // byte offsets of the chunks in a slice: core matrix (row / 8, K chunk) at 512 (row / 8) + 128 chunk
  const uint32_t aoff = (uint32_t)((ar >> 3) * 512 + ac * 128 + (ar & 7) * 16);
  const uint32_t boff = (uint32_t)((br >> 3) * 512 + (bc >> 1) * 128 + (br & 7) * 16 + (bc & 1) * 8);
  auto store = [&](uint32_t st) {
    {
      uint32_t lo[8], hi[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        digits(ra[e], emA, lo[e], hi[e]);
      }
      auto put = [&](int slice, uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3) {
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(st + slice * EA_SLICE + aoff), "r"(w0), "r"(w1),
                     "r"(w2), "r"(w3)
                     : "memory");
      };
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const uint32_t* w = half == 0 ? hi : lo;
        uint32_t dg[4][4];   // [pair of elements][byte]
#pragma unroll
        for (int q = 0; q < 4; ++q) digit_pairs(w[2 * q], w[2 * q + 1], dg[q]);
#pragma unroll
        for (int b = 3; b >= 0; --b) put(4 * half + 3 - b, dg[0][b], dg[1][b], dg[2][b], dg[3][b]);
      }
    }
    {
      uint32_t lo[4], hi[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        digits(rb[e], emB, lo[e], hi[e]);
      }
      auto put = [&](int slice, uint32_t w0, uint32_t w1) {
        asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(st + ESL * EA_SLICE + slice * EB_SLICE + boff), "r"(w0),
                     "r"(w1)
                     : "memory");
      };
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const uint32_t* w = half == 0 ? hi : lo;
        uint32_t dg[2][4];
        digit_pairs(w[0], w[1], dg[0]);
        digit_pairs(w[2], w[3], dg[1]);
#pragma unroll
        for (int b = 3; b >= 0; --b) put(4 * half + 3 - b, dg[0][b], dg[1][b]);
      }
    }
  };

  // Read-out: warp w holds rows 32 (w % 4) + lane, columns 16 (w / 4) .. + 15, each as a 96-bit
  // integer in units of order 7: orders 0-3 times 2^32 plus orders 4-7.
  const int quad = warp & 3, cg = (warp >> 2) * 16;
  uint32_t w0[16], w1[16], w2[16];
#pragma unroll
  for (int e = 0; e < 16; ++e) w0[e] = w1[e] = w2[e] = 0u;
  const uint32_t trow = tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)cg;
  auto flush = [&]() {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        int64_t s[8];
#pragma unroll
        for (int o = 0; o < 4; ++o) {
          uint32_t v[8];
          tmem_ld8(trow + (uint32_t)((4 * half + o) * EN + 8 * h), v);
          tmem_ld_wait(v);
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const int64_t t = (int64_t)__float2int_rn(__uint_as_float(v[e]));
            s[e] = o == 0 ? t : (s[e] << 8) + t;
          }
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const int x = 8 * h + e;
          const uint32_t s0 = (uint32_t)s[e], s1 = (uint32_t)((uint64_t)s[e] >> 32);
          if (half == 0)
            asm("add.cc.u32 %0, %0, %2;\n addc.u32 %1, %1, %3;" : "+r"(w1[x]), "+r"(w2[x]) : "r"(s0), "r"(s1));
          else
            asm("add.cc.u32 %0, %0, %3;\n addc.cc.u32 %1, %1, %4;\n addc.u32 %2, %2, %5;"
                : "+r"(w0[x]), "+r"(w1[x]), "+r"(w2[x])
                : "r"(s0), "r"(s1), "r"((uint32_t)((int)s1 >> 31)));
        }
      }
    }
  };

  constexpr uint32_t idesc = mma_idesc_f16(EM, EN);
  // 20 warps of 96 registers; the issuing warpgroup gives up what the converting ones take
  // (512 x 112 + 128 x 24 = 60,416 of 640 x 96 = 61,440)
  if (warp < ECW) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
    // step t's accumulators are complete once the commit of step t has arrived
    auto drain = [&](int t) -> bool {
      if (!__all_sync(0xffffffffu, mbar_wait_bounded(&empty_bar[t & 1], (uint32_t)((t >> 1) & 1)))) return false;
      tc_fence_after();
      flush();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&drained);
      return true;
    };
    if (nt > 0) load(0);
    for (int t = 0; t < nt; ++t) {
      const int s = t & 1;
      // the MMAs of this stage's previous use must be done reading it
      const bool bad = s_fail || (t >= 2 && !mbar_wait_bounded(&empty_bar[s], (uint32_t)(((t >> 1) - 1) & 1)));
      if (__any_sync(0xffffffffu, bad)) {
        s_fail = 1;
        break;
      }
      store(sbase + (uint32_t)s * E_STAGE);
      const bool group = t > 0 && t % EFLUSH == 0;
      if (t + 1 < nt && !group) load(t + 1);   // (not across a read-out: registers)
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&full_bar[s]);
      // the group that ended with step t - 1 (the MMAs of step t wait for its read-out)
      if (group) {
        if (!drain(t - 1)) {
          s_fail = 1;
          break;
        }
        if (t + 1 < nt) load(t + 1);
      }
    }
    const bool whole = !__any_sync(0xffffffffu, s_fail != 0) && (nt == 0 || drain(nt - 1));
    if (!whole) s_fail = 1;
    const int64_t m = m0 + 32 * quad + lane;
    const uint32_t fma_cols = spread && whole ? spread[2 * quad + (cg >> 5)] >> (cg & 31) : 0u;
    if (m < a.M) {
      const unsigned wa = a.ea[m];
      const double dm = a.D ? a.D[m] : 1.0;
      double* out = a.C + (int64_t)blockIdx.z * a.cslice + m;
  #pragma unroll
      for (int e = 0; e < 16; ++e) {
        const int n = n0 + cg + e;
        if (n < a.N && !(fma_cols >> e & 1)) {
          const unsigned wb = a.eb[n];
          const uint64_t low = ((uint64_t)w1[e] << 32) | w0[e];
          double x = fixed_to_double((((__int128)(int)w2[e]) << 64) | (__int128)(unsigned __int128)low,
                                     56 - 2168 + max(1, (int)(wa >> 20)) + max(1, (int)(wb >> 20)));
          if (!whole || (wa >> 20) == 0x7ffu || (wb >> 20) == 0x7ffu) x = __longlong_as_double(0x7ff8000000000000ll);
          out[(int64_t)n * a.ldc] = a.D ? dm * x : x;
        }
      }
    }
    // two warps per 32 x 32 part of the tile share its columns of FMAs
    if (spread && whole) fma_columns<KC>(a, m0 + 32 * (warp >> 2), n0 + 32 * ((warp >> 1) & 1), spread[warp >> 1], warp & 1, kb, ke);
  } else {
   asm volatile("setmaxnreg.dec.sync.aligned.u32 24;");
   if (tid == 32 * ECW) {
    for (int t = 0; t < nt && !s_fail; ++t) {
      const int s = t & 1;
      if (!mbar_wait_bounded(&full_bar[s], (uint32_t)((t >> 1) & 1)) ||
          (t > 0 && t % EFLUSH == 0 && !mbar_wait_bounded(&drained, (uint32_t)((t / EFLUSH - 1) & 1)))) {
        s_fail = 1;
        break;
      }
      tc_fence_after();
      const uint32_t st = sbase + (uint32_t)s * E_STAGE;
      const bool first = t % EFLUSH == 0;
      const uint64_t ad0 = smem_desc(st, 128u, 512u), bd0 = smem_desc(st + ESL * EA_SLICE, 128u, 512u);
#pragma unroll 1
      for (int kk = 0; kk < EK / 16; ++kk) {
        // digit i of A against digits 0 .. 7 - i of B, each onto another order's accumulator: A stays
        // in the collector, and no MMA waits for the one before (the sums are exact in any order)
#pragma unroll
        for (int i = 0; i < ESL; ++i) {
          const uint64_t ad = ad0 + (uint64_t)((i * EA_SLICE + kk * 256u) >> 4);
          const uint32_t acc = (first && kk == 0 && i == 0) ? 0u : 1u;
          mma_same_a<true>(tmem + (uint32_t)(i * EN), ad, bd0 + (uint64_t)((kk * 256u) >> 4), idesc, acc);
#pragma unroll
          for (int o = i + 1; o < ESL; ++o)
            mma_same_a<false>(tmem + (uint32_t)(o * EN), ad, bd0 + (uint64_t)(((o - i) * EB_SLICE + kk * 256u) >> 4),
                                   idesc, acc);
        }
      }
      mma_commit(&empty_bar[s]);
    }
   }
  }
  tc_fence_before();
  __syncthreads();
  if (s_fail) {   // whoever gave up: MMAs still queued finish before their operands and TMEM are given back
    if (tid == 32 * ECW && nt > 0) {
      mma_commit(&done);
      (void)mbar_wait_bounded(&done, 0u);
    }
    if (tid == 0) atomicExch(a.status, (int)NYS_ETIMEOUT);
    __syncthreads();
  }
  if (warp == 0) tmem_dealloc(tmem, 512);
}

// Fills EmuArgs::spread: the outputs of a tile with sum_k |a||b| < kSpread 2^ea 2^eb.  The sum is taken over the
// entries' magnitudes in FP16 at the scale of their rows, cut to 11 bits (2^-14 of the row's scale and
// smaller count as zero), so it is a lower bound, on mma.sync with FP32 sums.
//
// What bounds it is latency: the sums of ordinary rows pass within the first 64 K, so the CTAs of a tile's
// cluster (one to eight, a slice of K each, so that few tiles fill the chip too) look at 64 K
// each, add their sums up in one order and stop when every output has passed; only else they go on to
// the end of their slices.  Only the top words of the FP64 values are used.
constexpr float kSpread = 9.1f / 128.f;
constexpr int CK = 64, CPITCH = CK + 8;   // K of a step; halves from one row to the next
template <bool KC>
__global__ void __launch_bounds__(256, 2) gemm64_check_kernel(const EmuArgs a) {
  namespace cg = cooperative_groups;
  __shared__ __align__(16) unsigned char sm[EM * EN * sizeof(float)];
  static_assert((EM + EN) * CPITCH * sizeof(__half) <= sizeof(sm), "stage and sums share shared memory");
  __shared__ unsigned s_ea[EM], s_eb[EN];
  __shared__ unsigned s_fail[EM / 32][EN / 8];   // as EmuArgs::spread
  __shared__ int s_pass[8];
  unsigned short* As = reinterpret_cast<unsigned short*>(sm);
  unsigned short* Bs = As + EM * CPITCH;
  float* S = reinterpret_cast<float*>(sm);
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), nrank = (int)cl.num_blocks();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t m0 = (int64_t)blockIdx.y * EM;
  const int n0 = blockIdx.x * EN;
  const int64_t steps = (a.K + CK - 1) / CK, per = (steps + nrank - 1) / nrank;
  const int64_t s0 = min(steps, rank * per), s1 = min(steps, s0 + per);
  if (tid < EM) s_ea[tid] = m0 + tid < a.M ? a.ea[m0 + tid] : 0u;
  if (tid < EN) s_eb[tid] = n0 + tid < a.N ? a.eb[n0 + tid] : 0u;
  __syncthreads();
  // This thread's entries of a step: of A rows warp + 8 i at K lane and lane + 32 (KC), else columns lane + 32 j at K
  // warp + 8 i; of B rows warp + 8 i at K lane and lane + 32.
  unsigned ra[32], rb[16];
  auto top = [](const double* p) { return __ldg(reinterpret_cast<const unsigned*>(p) + 1) & 0x7fffffffu; };
  const double* pa = KC ? a.A + (m0 + warp) * a.lda + lane : a.A + (int64_t)warp * a.lda + m0 + lane;
  const double* pb = a.B + (int64_t)(n0 + warp) * a.ldb + lane;
  const int mv = (int)min((int64_t)EM, a.M - m0), nv = min(EN, a.N - n0);
  auto load = [&](int64_t st) {
    const int64_t k0 = st * CK;
    const int kv = (int)min((int64_t)CK, a.K - k0);
    const double* q = KC ? pa + k0 : pa + k0 * a.lda;
#pragma unroll
    for (int i = 0; i < (KC ? 16 : 8); ++i, q += 8 * a.lda) {
      if (KC) {
#pragma unroll
        for (int j = 0; j < 2; ++j) ra[2 * i + j] = warp + 8 * i < mv && lane + 32 * j < kv ? top(q + 32 * j) : 0u;
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) ra[4 * i + j] = warp + 8 * i < kv && lane + 32 * j < mv ? top(q + 32 * j) : 0u;
      }
    }
    q = pb + k0;
#pragma unroll
    for (int i = 0; i < 8; ++i, q += 8 * a.ldb)
#pragma unroll
      for (int j = 0; j < 2; ++j) rb[2 * i + j] = warp + 8 * i < nv && lane + 32 * j < kv ? top(q + 32 * j) : 0u;
  };
  // FP16 bits of a magnitude at the scale of its row (largest entries in [1, 2)); rows below 2^-959 and
  // rows that are not finite are decided without their sums
  auto scale_of = [](unsigned e) { return (max((int)(e >> 20), 64) - 15) << 20; };
  auto half_bits = [](unsigned h, int base) {
    const int v = (int)h - base;
    return (unsigned short)(v >= 1 << 20 ? min(v >> 10, 0x7bff) : 0);
  };
  auto store = [&]() {
#pragma unroll
    for (int i = 0; i < (KC ? 16 : 4); ++i) {
      const int r = KC ? warp + 8 * i : lane + 32 * i, base = scale_of(s_ea[r]);
#pragma unroll
      for (int j = 0; j < (KC ? 2 : 8); ++j) {
        const int k = KC ? lane + 32 * j : warp + 8 * j;
        As[r * CPITCH + k] = half_bits(ra[KC ? 2 * i + j : 4 * j + i], base);
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int r = warp + 8 * i, base = scale_of(s_eb[r]);
#pragma unroll
      for (int j = 0; j < 2; ++j) Bs[r * CPITCH + lane + 32 * j] = half_bits(rb[2 * i + j], base);
    }
  };
  // warp w: rows 16 w .. + 15, all columns; the fragments of mma.m16n8k16
  float acc[EN / 8][4] = {};
  const int g = lane >> 2, t = lane & 3;
  auto multiply = [&]() {
#pragma unroll
    for (int kk = 0; kk < CK; kk += 16) {
      auto frag = [&](const unsigned short* X, int r, int k) {
        return *reinterpret_cast<const uint32_t*>(X + r * CPITCH + kk + k + 2 * t);
      };
      const uint32_t x0 = frag(As, 16 * warp + g, 0), x1 = frag(As, 16 * warp + g + 8, 0);
      const uint32_t x2 = frag(As, 16 * warp + g, 8), x3 = frag(As, 16 * warp + g + 8, 8);
#pragma unroll
      for (int j = 0; j < EN / 8; ++j) {
        const uint32_t y0 = frag(Bs, 8 * j + g, 0), y1 = frag(Bs, 8 * j + g, 8);
        asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                     : "+f"(acc[j][0]), "+f"(acc[j][1]), "+f"(acc[j][2]), "+f"(acc[j][3])
                     : "r"(x0), "r"(x1), "r"(x2), "r"(x3), "r"(y0), "r"(y1));
      }
    }
  };
  auto run = [&](int64_t from, int64_t to) {
    if (from < to) load(from);
    for (int64_t st = from; st < to; ++st) {
      __syncthreads();
      store();
      __syncthreads();
      if (st + 1 < to) load(st + 1);
      multiply();
    }
  };
  // Whether every output of the tile has passed.  The columns 8 j .. 8 j + 7 are decided by CTA j / (8 / nrank),
  // from the sums of all CTAs in rank order.
  const int jper = (EN / 8) / nrank;
  auto decide = [&]() -> bool {
    __syncthreads();
    if (tid < EM / 32 * (EN / 8)) s_fail[tid >> 3][tid & 7] = 0u;
    if (nrank > 1) {
#pragma unroll
      for (int j = 0; j < EN / 8; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) S[(4 * j + q) * 256 + tid] = acc[j][q];
      cl.sync();
    } else {
      __syncthreads();
    }
    unsigned any = 0u;
    auto columns = [&](int j, const float (&sum)[4]) {
      unsigned lanes[2] = {0u, 0u};   // of columns 8 j + 2 t and 8 j + 2 t + 1
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int m = 16 * warp + g + 8 * (q >> 1), n = 8 * j + 2 * t + (q & 1);
        const unsigned ea = s_ea[m], eb = s_eb[n], wa = ea >> 20, wb = eb >> 20;
        const bool pass = wa != 0x7ffu && wb != 0x7ffu && (ea == 0u || eb == 0u || (wa >= 64u && wb >= 64u && sum[q] >= kSpread));
        lanes[q & 1] |= __ballot_sync(0xffffffffu, m < mv && n < nv && !pass);
      }
      unsigned byte = 0u;
#pragma unroll
      for (int c = 0; c < 8; ++c) byte |= (unsigned)((lanes[c & 1] & (0x11111111u << (c >> 1))) != 0u) << c;
      if (byte && lane == 0) atomicOr(&s_fail[warp >> 1][j], byte);
      any |= byte;
    };
    if (nrank == 1) {
#pragma unroll
      for (int j = 0; j < EN / 8; ++j) columns(j, acc[j]);
    } else {
      for (int j = rank * jper; j < (rank + 1) * jper; ++j) {
        float sum[4] = {0.f, 0.f, 0.f, 0.f}, part[8][4];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const float* Sr = cl.map_shared_rank(S, r < nrank ? r : rank);
#pragma unroll
          for (int q = 0; q < 4; ++q) part[r][q] = r < nrank ? Sr[(4 * j + q) * 256 + tid] : 0.f;
        }
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
          for (int q = 0; q < 4; ++q) sum[q] += part[r][q];
        columns(j, sum);
      }
    }
    const int fail = __syncthreads_or((int)any);
    if (nrank == 1) return !fail;
    if (tid < nrank) cl.map_shared_rank(s_pass, tid)[rank] = !fail;
    cl.sync();
    bool all = true;
    for (int r = 0; r < nrank; ++r) all = all && s_pass[r];
    return all;
  };
  run(s0, min(s0 + 1, s1));
  if (!decide() && per > 1) {
    run(min(s0 + 1, s1), s1);
    (void)decide();
  }
  if (tid < EM / 32 * (EN / 8) && (tid & 7) / jper == rank)
    a.spread[((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * ESPREAD + tid] = (unsigned char)s_fail[tid >> 3][tid & 7];
}

// Largest magnitude (top word: order and exponent; a NaN or an infinity is above every finite
// value; zero only for zeros) of each row and / or column of the row-major rows x cols matrix X.  Block (bx, by):
// columns 512 bx .. + 511 (two per thread), `slab` rows from by * slab; rowmax and colmax are
// zeroed by the caller.  Bound by the one read of X.
__device__ __forceinline__ unsigned top_word(double x) {
  return ((unsigned)__double2hiint(x) & 0x7fffffffu) | (__double2loint(x) != 0 ? 1u : 0u);
}
constexpr int kAbsCols = 512;
constexpr int kAbsMaxSlab = 256;
__global__ void __launch_bounds__(256) absmax_kernel(const double* __restrict__ X, int64_t rows, int64_t cols,
                                                     int64_t ld, int slab, unsigned* rowmax, unsigned* colmax) {
  __shared__ unsigned rm[kAbsMaxSlab][8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t c = (int64_t)blockIdx.x * kAbsCols + 2 * threadIdx.x;
  const int64_t r0 = (int64_t)blockIdx.y * slab;
  const int nr = (int)min((int64_t)slab, rows - r0);
  const bool vec = (ld & 1) == 0 && (reinterpret_cast<uintptr_t>(X) & 15u) == 0 && c + 1 < cols;
  unsigned m0 = 0u, m1 = 0u;
  for (int b = 0; b < nr; b += 8) {
    unsigned h0[8], h1[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      h0[q] = h1[q] = 0u;
      if (b + q < nr) {
        const double* p = X + (r0 + b + q) * ld + c;
        if (vec) {
          const double2 v = __ldg(reinterpret_cast<const double2*>(p));
          h0[q] = top_word(v.x);
          h1[q] = top_word(v.y);
        } else {
          if (c < cols) h0[q] = top_word(__ldg(p));
          if (c + 1 < cols) h1[q] = top_word(__ldg(p + 1));
        }
      }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      m0 = max(m0, h0[q]);
      m1 = max(m1, h1[q]);
      if (rowmax) {
        const unsigned r = __reduce_max_sync(0xffffffffu, max(h0[q], h1[q]));
        if (lane == 0 && b + q < nr) rm[b + q][warp] = r;
      }
    }
  }
  if (colmax) {
    if (c < cols && m0) atomicMax(colmax + c, m0);
    if (c + 1 < cols && m1) atomicMax(colmax + c + 1, m1);
  }
  if (rowmax) {
    __syncthreads();
    for (int r = threadIdx.x; r < nr; r += 256) {
      unsigned v = 0u;
#pragma unroll
      for (int w = 0; w < 8; ++w) v = max(v, rm[r][w]);
      if (v) atomicMax(rowmax + r0 + r, v);
    }
  }
}

// C (column-major, ldc) = diag(D) sum_z part[z] (column-major, ld M), increasing z.
__global__ void emu_sum_kernel(const double* __restrict__ part, int nz, int64_t M, int64_t len,
                               const double* __restrict__ D, double* __restrict__ C, int64_t ldc) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len; i += (int64_t)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int z0 = 0; z0 < nz; z0 += 8) {
      double v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = z0 + q < nz ? part[(z0 + q) * len + i] : 0.0;
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (z0 + q < nz) s += v[q];
    }
    const int64_t n = i / M, m = i - n * M;
    C[m + n * ldc] = D ? D[m] * s : s;
  }
}

// Split of K: the slice count (at most 64, each of at least E_MINSTEPS stages) whose CTAs take
// the fewest stages in all, counting three stages for a CTA's read-out and start-up.  For 152
// SMs whatever the device, so that the summation order does not depend on it.
int emu_slices(int64_t tiles, int64_t steps) {
  int best = 1;
  int64_t best_cost = INT64_MAX;
  for (int z = 1; z <= 64; ++z) {
    if (z > 1 && steps / z < E_MINSTEPS) break;
    const int64_t waves = (tiles * z + 151) / 152;
    const int64_t cost = waves * ((steps + z - 1) / z + 3);
    if (cost < best_cost) {
      best_cost = cost;
      best = z;
    }
  }
  return best;
}
struct EmuPlan {
  int64_t mt, steps, kslice;
  int ntl, nz;
};
EmuPlan emu_plan(int64_t M, int N, int64_t K) {
  EmuPlan p;
  p.mt = (M + EM - 1) / EM;
  p.ntl = (N + EN - 1) / EN;
  p.steps = std::max<int64_t>(1, (K + EK - 1) / EK);
  const int z = emu_slices(p.mt * p.ntl, p.steps);
  const int64_t per = (p.steps + z - 1) / z;
  p.kslice = per * EK;
  p.nz = (int)((p.steps + per - 1) / per);
  return p;
}

}  // namespace

cudaError_t absmax_f64(const double* X, int64_t rows, int64_t cols, int64_t ld, unsigned* rowmax, unsigned* colmax,
                       cudaStream_t st) {
  if (rowmax) NYS_CUDA_TRY(cudaMemsetAsync(rowmax, 0, rows * sizeof(unsigned), st));
  if (colmax) NYS_CUDA_TRY(cudaMemsetAsync(colmax, 0, cols * sizeof(unsigned), st));
  // slabs of 8 .. 256 rows, a multiple of 8: at least ~600 blocks where the matrix allows
  const int64_t cb = (cols + kAbsCols - 1) / kAbsCols;
  int64_t slab = (rows * cb + 607) / 608;
  slab = std::min<int64_t>(kAbsMaxSlab, std::max<int64_t>(8, (slab + 7) / 8 * 8));
  while ((rows + slab - 1) / slab > 65535 && slab < kAbsMaxSlab) slab += 8;
  for (int64_t r0 = 0; r0 < rows; r0 += 65535 * slab) {
    const int64_t nr = std::min<int64_t>(65535 * slab, rows - r0);
    count_launch();
    absmax_kernel<<<dim3((unsigned)cb, (unsigned)((nr + slab - 1) / slab)), 256, 0, st>>>(
        X + r0 * ld, nr, cols, ld, (int)slab, rowmax ? rowmax + r0 : nullptr, colmax);
    NYS_CUDA_TRY(cudaGetLastError());
  }
  return cudaSuccess;
}

static size_t spread_bytes(const EmuPlan& p) { return ((size_t)p.mt * p.ntl * ESPREAD + 255) / 256 * 256; }

size_t gemm64_work_bytes(int64_t M, int N, int64_t K) {
  const EmuPlan p = emu_plan(M, N, K);
  return spread_bytes(p) + (p.nz > 1 ? (size_t)p.nz * M * N * sizeof(double) : 0);
}

// The check over one launch's tiles, in clusters of up to eight CTAs that split K: about one CTA per SM or more.
template <bool KC>
static cudaError_t launch_check(const EmuArgs& a, dim3 tiles, cudaStream_t st) {
  int c = 1;
  while (c < 8 && (int64_t)tiles.x * tiles.y * c < 152 && (int64_t)2 * c * CK <= a.K) c *= 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(tiles.x, tiles.y, (unsigned)c);
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = (unsigned)c;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  count_launch();
  return cudaLaunchKernelEx(&cfg, gemm64_check_kernel<KC>, a);
}

cudaError_t gemm64(const double* A, bool k_contiguous, int64_t lda, const unsigned* ea, int64_t M, const double* B,
                   int64_t ldb, const unsigned* eb, int N, int64_t K, const double* D, double* C, int64_t ldc,
                   void* work, int* status, cudaStream_t st, bool any_scale) {
  if (M <= 0 || N <= 0 || K <= 0) return cudaErrorInvalidValue;
  const EmuPlan p = emu_plan(M, N, K);
  unsigned char* spread = reinterpret_cast<unsigned char*>(work);
  double* part = reinterpret_cast<double*>(spread + spread_bytes(p));
  if (p.ntl > INT32_MAX) return cudaErrorInvalidValue;
  EmuArgs a;
  a.A = A;
  a.lda = lda;
  a.B = B;
  a.ldb = ldb;
  a.K = K;
  a.kslice = p.kslice;
  a.N = N;
  a.eb = eb;
  a.status = status;
  a.D = p.nz == 1 ? D : nullptr;
  a.ldc = p.nz == 1 ? ldc : M;
  a.cslice = M * (int64_t)N;
  const void* fn = k_contiguous ? (const void*)gemm64_tc_kernel<true> : (const void*)gemm64_tc_kernel<false>;
  NYS_CUDA_TRY(ensure_max_dyn_smem(fn, 2 * E_STAGE));
  // row tiles in launches of at most 65,535
  for (int64_t t0 = 0; t0 < p.mt; t0 += 65535) {
    const int64_t nt = std::min<int64_t>(65535, p.mt - t0), m0 = t0 * EM;
    a.A = A + (k_contiguous ? m0 * lda : m0);
    a.ea = ea + m0;
    a.M = std::min<int64_t>(M - m0, nt * EM);
    a.C = (p.nz == 1 ? C : part) + m0;
    a.D = p.nz == 1 && D ? D + m0 : nullptr;
    const dim3 grid((unsigned)p.ntl, (unsigned)nt, (unsigned)p.nz);
    a.spread = any_scale ? spread + t0 * p.ntl * ESPREAD : nullptr;
    if (any_scale) NYS_CUDA_TRY(k_contiguous ? launch_check<true>(a, grid, st) : launch_check<false>(a, grid, st));
    count_launch();
    if (k_contiguous) gemm64_tc_kernel<true><<<grid, ET, 2 * E_STAGE, st>>>(a);
    else gemm64_tc_kernel<false><<<grid, ET, 2 * E_STAGE, st>>>(a);
    NYS_CUDA_TRY(cudaGetLastError());
  }
  if (p.nz > 1) {
    const int64_t len = M * (int64_t)N;
    count_launch();
    emu_sum_kernel<<<(unsigned)std::min<int64_t>(4096, (len + 127) / 128), 128, 0, st>>>(
        part, p.nz, M, len, D, C, ldc);
    NYS_CUDA_TRY(cudaGetLastError());
  }
  return cudaSuccess;
}

}  // namespace nys

namespace nys {

// ------------------------------------------------------------------ Y = A^T diag(D) A X
namespace {
struct HmmShape {
  size_t row, col, ex, ew, w, status, total;   // byte offsets in the scratch; the products' work last
};
HmmShape hmm_shape(const nys_matrix* A, int m) {
  auto up = [](size_t b) { return (b + 255) / 256 * 256; };
  HmmShape h;
  h.row = 0;
  h.col = h.row + up((size_t)A->n * sizeof(unsigned));
  h.ex = h.col + up((size_t)A->d * sizeof(unsigned));
  h.ew = h.ex + up((size_t)m * sizeof(unsigned));
  h.status = h.ew + up((size_t)m * sizeof(unsigned));
  h.w = h.status + 256;
  h.total = h.w + up((size_t)A->n * m * sizeof(double)) +
            std::max(gemm64_work_bytes(A->n, m, A->d), gemm64_work_bytes(A->d, m, A->n));
  return h;
}
}  // namespace

size_t hmm64_bytes(const nys_matrix* A, int m) { return hmm_shape(A, m).total; }

cudaError_t hmm64_prepare(const nys_matrix* A, int m, void* scratch, cudaStream_t st) {
  const HmmShape h = hmm_shape(A, m);
  unsigned char* b = reinterpret_cast<unsigned char*>(scratch);
  NYS_CUDA_TRY(cudaMemsetAsync(b + h.status, 0, sizeof(int), st));
  return absmax_f64(reinterpret_cast<const double*>(A->data), A->n, A->d, A->ld, reinterpret_cast<unsigned*>(b + h.row),
                    reinterpret_cast<unsigned*>(b + h.col), st);
}

int* hmm64_status(const nys_matrix* A, int m, void* scratch) {
  return reinterpret_cast<int*>(reinterpret_cast<unsigned char*>(scratch) + hmm_shape(A, m).status);
}

cudaError_t hmm64(const nys_matrix* A, const double* D, const double* X, int m, double* Y, void* scratch,
                  cudaStream_t st) {
  const HmmShape h = hmm_shape(A, m);
  unsigned char* b = reinterpret_cast<unsigned char*>(scratch);
  const double* Ad = reinterpret_cast<const double*>(A->data);
  unsigned* row = reinterpret_cast<unsigned*>(b + h.row);
  unsigned* col = reinterpret_cast<unsigned*>(b + h.col);
  unsigned* ex = reinterpret_cast<unsigned*>(b + h.ex);
  unsigned* ew = reinterpret_cast<unsigned*>(b + h.ew);
  double* W = reinterpret_cast<double*>(b + h.w);
  int* status = reinterpret_cast<int*>(b + h.status);
  void* work = b + h.w + ((size_t)A->n * m * sizeof(double) + 255) / 256 * 256;
  const int64_t n = A->n, d = A->d;
  NYS_CUDA_TRY(absmax_f64(X, m, d, d, ex, nullptr, st));
  NYS_CUDA_TRY(gemm64(Ad, true, A->ld, row, n, X, d, ex, m, d, D, W, n, work, status, st, /*any_scale=*/true));
  NYS_CUDA_TRY(absmax_f64(W, m, n, n, ew, nullptr, st));
  return gemm64(Ad, false, A->ld, col, d, W, n, ew, m, n, nullptr, Y, d, work, status, st, /*any_scale=*/true);
}

}  // namespace nys
