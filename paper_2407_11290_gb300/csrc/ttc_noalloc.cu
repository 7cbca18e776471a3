// ttc_noalloc.cu -- sampled relative error of a TT without any allocation.
//
// Callers that must not allocate device memory (code running inside a custom
// allocator or memory-pool callback, a pre-sized real-time or embedded
// process whose whole GPU memory budget is fixed at start-up, a plugin whose
// host forbids cudaMalloc after initialisation) can still check a TT
// against its function with ttcross_sampled_error_noalloc.  It is a variant
// of the error evaluation that ttcross_run performs: the per-chunk partial
// sums it needs live in the file-scope array below, not in memory from
// cudaMalloc.
//
// The arrays are a fixed 66 KiB per GPU: every device that loads the library
// holds them until the process exits.  All calls share them, and each call
// overwrites every slot it later reads, so nothing has to be cleared; but two
// calls whose kernels overlap on the GPU (different streams, or different
// host threads on one device) race on them and must be ordered by the caller.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdio>
#include <mutex>

#include "ttc_split.cuh"
#include "ttcross.h"

namespace ttc {
void set_last_error(const char *msg);  // ttc_api.cu: shared with ttcross_last_error_string
}

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int64_t kChunk = 4096;          // samples per partial-sum slot (at most)
constexpr int kMaxChunks = 4096;          // slots -> at most 16,777,216 samples
constexpr int kMaxRank = 256;             // core sizes s_m: 8 register slots per lane
constexpr int kMaxD = 16;
constexpr int kMaxDevices = 64;

// (sum (X - X~)^2, sum X^2) of every chunk of samples
static __device__ __align__(256) double g_chunk_sums[2 * kMaxChunks];
// largest exponent of row k of middle core m (the tensor-core form)
static __device__ int32_t g_row_exp[kMaxD][32];

struct ErrArgs {
  int32_t d;
  int32_t gen;
  int64_t n[kMaxD];
  const double *core[kMaxD];  // core m: [s_m][n_m][s_{m+1}] row-major (device)
  int32_t s[kMaxD + 1];
  int32_t dx, dv;
  double a_rho, a_u, a_T, vmin, vmax;
  int64_t nsamples;
  int32_t exhaustive;
  uint64_t seed;
};

__device__ __forceinline__ uint64_t mix_at(uint64_t seed, uint64_t k) {
  uint64_t z = seed + (k + 1) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// index of mode m of sample k (SplitMix64 counter form, sample-major,
// mode-minor, index = floor(x n / 2^64); entry k in column-major order when
// every entry is used); computed alone, so no index array lives in memory
__device__ __forceinline__ int32_t coord(const ErrArgs &a, int64_t k, int m) {
  if (a.exhaustive) {
    int64_t l = k;
    for (int j = 0; j < m; ++j) l /= a.n[j];
    return (int32_t)(l % a.n[m]);
  }
  return (int32_t)__umul64hi(mix_at(a.seed, (uint64_t)(k * a.d + m)), (uint64_t)a.n[m]);
}

__device__ __forceinline__ double x_at(const ErrArgs &a, int64_t k, int m) {
  const double two_pi = 6.283185307179586476925286766559;
  return __dmul_rn(two_pi, (double)coord(a, k, m)) / (double)a.n[m];
}

// X at sample k: the Hilbert tensor or the Maxwellian of the generator
__device__ double entry(const ErrArgs &a, int64_t k) {
  if (a.gen == TTC_GEN_HILBERT) {
    int64_t s = 1;
    for (int m = 0; m < a.d; ++m) s += coord(a, k, m);
    return 1.0 / (double)s;
  }
  const double two_pi = 6.283185307179586476925286766559;
  double prod_sin = 1.0, sum_x = 0.0;
  for (int m = 0; m < a.dx; ++m) {
    const double x = x_at(a, k, m);
    prod_sin = __dmul_rn(prod_sin, sin(x));
    sum_x = __dadd_rn(sum_x, x);
  }
  const double rho = __dadd_rn(1.0, __dmul_rn(a.a_rho, prod_sin));
  const double T = __dadd_rn(1.0, __dmul_rn(a.a_T, cos(sum_x)));
  double q = 0.0;
  for (int j = 0; j < a.dv; ++j) {
    const int m = a.dx + j;
    const double v = __dadd_rn(
        a.vmin, __dmul_rn(__dsub_rn(a.vmax, a.vmin), (double)coord(a, k, m)) / (double)(a.n[m] - 1));
    const double u = __dmul_rn(a.a_u, cos(x_at(a, k, (j + 1) % a.dx)));
    const double dvu = __dsub_rn(v, u);
    q = __dadd_rn(q, __dmul_rn(dvu, dvu));
  }
  return __dmul_rn(rho / pow(__dmul_rn(two_pi, T), 0.5 * (double)a.dv), exp(-q / __dmul_rn(2.0, T)));
}

// X~ at sample k by one warp: X~ = G_1(i_1) ... G_d(i_d), left to right.
// Lane l keeps v[32 j + l] (j < K) in registers; each output w[u] of a core
// is the serial FMA chain over p = 0, 1, ... of v[p] G(p, i, u), v[p]
// broadcast from its lane, so the order of the operations is that of a plain
// per-sample loop and no vector lives in local memory.  Every lane returns
// the value.
template <int K>
__device__ double tt_value_warp(const ErrArgs &a, int64_t k) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  double v[K], w[K];
  int rl = a.s[1];
  {
    const double *G = a.core[0] + (int64_t)coord(a, k, 0) * rl;
#pragma unroll
    for (int j = 0; j < K; ++j) v[j] = 32 * j + lane < rl ? G[32 * j + lane] : 0.0;
  }
  for (int m = 1; m < a.d; ++m) {
    const int rr = a.s[m + 1];
    const int64_t ld = a.n[m] * rr;
    const double *G = a.core[m] + (int64_t)coord(a, k, m) * rr;
#pragma unroll
    for (int j = 0; j < K; ++j) w[j] = 0.0;
#pragma unroll
    for (int jp = 0; jp < K; ++jp) {
      if (32 * jp >= rl) break;
      const int lim = min(32, rl - 32 * jp);
      for (int l = 0; l < lim; ++l) {
        const int p = 32 * jp + l;
        const double vp = __shfl_sync(FULL, v[jp], l);
#pragma unroll
        for (int j = 0; j < K; ++j) {
          const int u = 32 * j + lane;
          if (u < rr) w[j] = __fma_rn(vp, G[p * ld + u], w[j]);
        }
      }
    }
#pragma unroll
    for (int j = 0; j < K; ++j) v[j] = w[j];
    rl = rr;
  }
  return __shfl_sync(FULL, v[0], 0);
}

__device__ double block_sum(double v, double *red) {
  for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < kWarps; ++i) s += red[i];
  __syncthreads();
  return s;
}

// one slot per chunk of kChunk samples (a warp per sample, warp w of the
// CTA taking samples w, w + 8, ... of the chunk): the result does not depend
// on the grid, so it is the same on any GPU
template <int K>
__global__ void __launch_bounds__(kThreads) k_chunk_sums(ErrArgs a, int64_t nchunks, double *sums) {
  __shared__ double red[kWarps];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int64_t c = blockIdx.x; c < nchunks; c += gridDim.x) {
    const int64_t k0 = c * kChunk, k1 = min(a.nsamples, k0 + kChunk);
    double num = 0.0, den = 0.0;
    for (int64_t k = k0 + warp; k < k1; k += kWarps) {
      const double xt = tt_value_warp<K>(a, k);
      if (lane == 0) {
        const double x = entry(a, k);
        const double e = __dsub_rn(x, xt);
        num = __fma_rn(e, e, num);
        den = __fma_rn(x, x, den);
      }
    }
    const double sn = block_sum(num, red);
    const double sd = block_sum(den, red);
    if (threadIdx.x == 0) {
      sums[2 * c] = sn;
      sums[2 * c + 1] = sd;
    }
  }
}

// ---------------------------------------------------------------------------
// Cores of sizes up to 32 and middle modes of up to kTcN indices: the middle
// cores on the tensor cores, as exact split-integer products (ttc_error.cuh
// describes the scheme), with everything a CTA needs in its shared memory.
// A CTA takes S = 16384 / KP samples at a time (KP: the core sizes rounded up
// to 16 or 32), keeps their vectors there as fixed-point rows (128 KB), sorts
// the samples by each middle index in turn and multiplies every run of up to
// 16 samples of one index by that index's core slice, whose columns a warp
// brings to fixed point itself.
// Fixed point is as fine as its largest term, and a TT's bonds may be scaled at
// will (a column of one core up, the row of the next down by as much).  So the
// rows of a middle core are taken at their largest exponent, k_row_exp, and the
// columns before them grow by it: both are exponents, no product is rounded.
// That balances a dense bond only.  Where terms have scales of their own (sums of
// TTs, CP forms, a peak beside a smooth part) the term that sets the unit need not
// be one that counts, so every sample carries a bound of its error along:
//   D_k = e_k 2^53 / (KP (d - 2)) - a_k   for entry k of its vector,
// e_k a bound on the entry's error in fixed point and a_k the chain of absolute
// values |G_1| ... |G_m|, of which an FP64 chain loses up to KP (d - 2) 2^-53.
// Both go through a core as its absolute values do, so D does (one bf16 mma.sync
// beside 36 f16 ones), and a core adds the error of its products: dropped digits of
// up to 7 2^-62 a term, the operands' rounding, the sum's to 2^-57 (KP = 32; 2^-58),
// relative to the largest entry of the row and of the column.  Where the sum of D
// times the last core's |entries| is above zero the sample is computed again by
// its FP64 chain, as are samples that met subnormal or non-finite entries or left
// the range of doubles.  (None of the samples of exponential sums in a random
// basis, 0.6 % of those of a 6D n = 64 Hilbert cross, 8 % of a 2+2D Maxwellian's.)
// A warp per sample in FP64 issued one FMA per core row with half its lanes
// idle at size 16: 6.57 ms for 1e6 samples of a 6D n = 64 TT of ranks 16 (its
// 1.04e9 FMAs take 1.7 ms at the FP64 pipe's rate); this form takes 1.33 ms, 0.09 ms
// of them for the rows' exponents and 0.21 ms for D (ranks 32: 5.70 ms, 4.50 without D).
constexpr int kTcThreads = 512, kTcN = 256;

template <int KP>
struct TcSmem {
  static constexpr int S = 16384 / KP;
  uint64_t vec[S][KP];       // fixed-point rows (interleaved pairs)
  uint16_t dif[S][KP];       // D of the rows' entries, bf16, largest entry 1
  int32_t unit[S];           // exponents of their units; after the last core: whether
                             // the sample goes to its FP64 chain
  double res[S];             // X~
  uint16_t key[S], order[S];
  uint32_t tile[S / 16 + kTcN];
  int32_t cnt[kTcN];
  int32_t ntiles, nagain;
  double red[kTcThreads / 32];
};

// the samples' order by index of mode m, and their tiles: index (bits 16..),
// first place (bits 4..15), rows - 1 (bits 0..3)
template <int KP>
__device__ void tc_sort(const ErrArgs &a, int64_t k0, int ns, int m, TcSmem<KP> &sm) {
  constexpr unsigned FULL = 0xffffffffu;
  const int tid = threadIdx.x, n = (int)a.n[m];
  if (tid < kTcN) sm.cnt[tid] = 0;
  __syncthreads();
  for (int s = tid; s < ns; s += kTcThreads) {
    const int i = coord(a, k0 + s, m);
    sm.key[s] = (uint16_t)i;
    atomicAdd(&sm.cnt[i], 1);
  }
  __syncthreads();
  if (tid < 32) {
    // eight indices a lane: exclusive scans of the samples and of the tiles
    int c[8], sum = 0, nt = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      c[q] = tid * 8 + q < n ? sm.cnt[tid * 8 + q] : 0;
      sum += c[q];
      nt += (c[q] + 15) / 16;
    }
    int is = sum, it = nt;
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(FULL, is, o), v = __shfl_up_sync(FULL, it, o);
      if (tid >= o) {
        is += u;
        it += v;
      }
    }
    if (tid == 31) sm.ntiles = it;
    int at = is - sum, ta = it - nt;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      if (tid * 8 + q < n) sm.cnt[tid * 8 + q] = at;
      for (int o = 0; o < c[q]; o += 16)
        sm.tile[ta++] = ((uint32_t)(tid * 8 + q) << 16) | ((uint32_t)(at + o) << 4) |
                        (uint32_t)(min(16, c[q] - o) - 1);
      at += c[q];
    }
  }
  __syncthreads();
  // (the order within a group is free: every row's result is its own)
  for (int s = tid; s < ns; s += kTcThreads) sm.order[atomicAdd(&sm.cnt[sm.key[s]], 1)] = (uint16_t)s;
  __syncthreads();
}

// no exponent: of a row or column of zeros
constexpr int32_t kNone = -(1 << 20);

// g_row_exp: a CTA per row of a middle core.  A row of zeros has none: the
// column that meets it contributes nothing, so it must not set a unit.
__global__ void __launch_bounds__(kThreads) k_row_exp(ErrArgs a) {
  const int m = (int)blockIdx.y + 1, k = (int)blockIdx.x;
  if (k >= a.s[m]) return;
  const int64_t len = a.n[m] * a.s[m + 1];
  const double *G = a.core[m] + (int64_t)k * len;
  int e = 0;
  for (int64_t x = threadIdx.x; x < len; x += kThreads) {
    const int v = ttc::tc_expo(G[x]);
    if (v != 0x7ff) e = max(e, v);  // (the products find what is not finite)
  }
  e = __reduce_max_sync(0xffffffffu, e);
  __shared__ int red[kWarps];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = e;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < kWarps; ++i) e = max(e, red[i]);
    g_row_exp[m][k] = e ? e - 1023 : kNone;
  }
}

// the unit's exponent of a row or column from its largest exponent (kNone: it
// is zero) and whether an entry was not finite
__device__ __forceinline__ int32_t tc_unit_of(int emax, bool bad) {
  return bad ? ttc::TC_BAD : emax - 1084;
}
// (the tests of doubles here are on their bits: a comparison would take the FP64 pipe)
__device__ __forceinline__ bool tc_zero(double x) {
  return ((uint32_t)__double2hiint(x) << 1 | (uint32_t)__double2loint(x)) == 0;
}
// entries that fixed point does not take: not finite, or subnormal
__device__ __forceinline__ bool tc_odd(double x) {
  return (uint32_t)(ttc::tc_expo(x) - 1) >= 0x7fe && !tc_zero(x);
}

// D in bf16 pairs, and its scale: |x| / 2^emax (emax in units of tc_expo, so below
// 1) cut to bf16, a nonzero one to 2^-126 at least
__device__ __forceinline__ uint32_t bf_pair(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
__device__ __forceinline__ float bf_lo(uint32_t p) { return __uint_as_float(p << 16); }
__device__ __forceinline__ float bf_hi(uint32_t p) { return __uint_as_float(p & 0xffff0000u); }
__device__ __forceinline__ uint32_t bf_abs(double x, int emax) {
  const int b = (__double2hiint(x) >> 13) & 0x3ffff;  // exponent field, seven bits of the mantissa
  return b >= 0x80 ? (uint32_t)max(b - ((emax - 126) << 7), 0x80) : 0u;
}
__device__ __forceinline__ float exp2_clamped(int n) {
  return __int_as_float((min(max(n, -126), 127) + 127) << 23);
}
// D 2^n of a float D as a double: next to zero below the range of doubles, NaN or
// Inf above it and for those
__device__ __forceinline__ double dif_real(float x, int n) {
  const uint32_t b = __float_as_uint(x);
  const int e = (int)(b >> 23 & 0xff);
  const int f = e == 0xff ? 0x7ff : min(max(e + 896 + n, 0), 0x7ff);
  const uint32_t hi = (b & 0x80000000u) | (uint32_t)f << 20 | (b & 0x7fffff) >> 3;
  return x == 0.f ? 0.0 : __hiloint2double((int)hi, (int)(b << 29));
}
// bounds of the errors that D counts, in units of KP 2^-53 of one core
constexpr float kDifVec = 0x1p-14f;   // an entry of the first vector: 2^-63, KP >= 16
constexpr float kDifCore = 0.02f;     // 7 2^-62 + 2^-62 a term and 2^-58 (KP = 16) in all

__device__ __forceinline__ void dif_mma(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// one middle core: rows of the vectors times G_m(i), in place; the last one
// meets the last core and leaves X~ and which samples need their FP64 chain
template <int KP>
__device__ void tc_core(const ErrArgs &a, int64_t k0, int m, TcSmem<KP> &sm) {
  using namespace ttc;
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int KS = KP / 16, CT = KP / 8;
  constexpr int sh = 25 - (KP == 16 ? 4 : 5);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const int K = a.s[m], N = a.s[m + 1];
  const bool last = m == a.d - 2;
  const int64_t ld = a.n[m] * N;
  int32_t rx[KS][4];  // of the rows that the lane reads
#pragma unroll
  for (int ks = 0; ks < KS; ++ks)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int k = ks * 16 + 2 * t + (q & 1) + 8 * (q >> 1);
      rx[ks][q] = k < K ? g_row_exp[m][k] : 0;
    }
  for (int x = warp; x < sm.ntiles; x += kTcThreads / 32) {
    const uint32_t tl = sm.tile[x];
    const int i = (int)(tl >> 16), at = (int)(tl >> 4) & 0xfff, rows = (int)(tl & 15) + 1;
    const int sg = sm.order[at + min(g, rows - 1)], sg8 = sm.order[at + min(g + 8, rows - 1)];
    const int32_t e0 = sm.unit[sg], e1 = sm.unit[sg8];
    const double *G = a.core[m] + (int64_t)i * N;
    const double *Y = a.core[a.d - 1];
    const int64_t yn = a.n[a.d - 1];
    int j0 = 0, j1 = 0;
    if (last) {
      j0 = coord(a, k0 + sg, a.d - 1);
      j1 = coord(a, k0 + sg8, a.d - 1);
    }
    int64_t out[CT][4];
    uint32_t dif[CT][2];  // D of the outputs, bf16 (columns 2t, 2t + 1 of rows g, g + 8)
    int32_t ea[CT], eb[CT];
    int top0 = INT_MIN, top1 = INT_MIN;
    bool bad = e0 == TC_BAD || e1 == TC_BAD;
    double v0 = 0.0, v1 = 0.0, d0 = 0.0, d1 = 0.0;
    const float core = kDifCore / (float)(a.d - 2);
#pragma unroll
    for (int c = 0; c < CT; ++c) {
      if (8 * c >= N) break;
      // the lane's entries of column u, their largest exponent over the column
      const int u = 8 * c + g;
      double w[KS][4];
      int emax = kNone;
      bool odd = false;
#pragma unroll
      for (int ks = 0; ks < KS; ++ks)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int k = ks * 16 + 2 * t + (q & 1) + 8 * (q >> 1);
          w[ks][q] = k < K && u < N ? G[k * ld + u] : 0.0;
        }
#pragma unroll
      for (int ks = 0; ks < KS; ++ks)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int e = tc_expo(w[ks][q]);
          odd |= tc_odd(w[ks][q]);
          if (e) emax = max(emax, e - rx[ks][q]);
        }
      emax = max(emax, __shfl_xor_sync(FULL, emax, 1));
      emax = max(emax, __shfl_xor_sync(FULL, emax, 2));
      float dp[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) {
        const uint16_t *x = &sm.dif[sg][ks * 16 + 2 * t], *y = &sm.dif[sg8][ks * 16 + 2 * t];
        const uint32_t da[4] = {
            *reinterpret_cast<const uint32_t *>(x), *reinterpret_cast<const uint32_t *>(y),
            *reinterpret_cast<const uint32_t *>(x + 8), *reinterpret_cast<const uint32_t *>(y + 8)};
        dif_mma(dp, da, bf_abs(w[ks][0], emax + rx[ks][0]) | bf_abs(w[ks][1], emax + rx[ks][1]) << 16,
                bf_abs(w[ks][2], emax + rx[ks][2]) | bf_abs(w[ks][3], emax + rx[ks][3]) << 16);
      }
      const int32_t ge = tc_unit_of(emax, odd);
      ea[c] = __shfl_sync(FULL, ge, 8 * t);      // columns 2t, 2t + 1: lanes 4 (2t), 4 (2t + 1)
      eb[c] = __shfl_sync(FULL, ge, 8 * t + 4);
      bad |= ge == TC_BAD;
      float acc[8][4];
#pragma unroll
      for (int l = 0; l < 8; ++l)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[l][q] = TC_MAGIC;
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) {
        const uint4 z0 = tc_pack(tc_fix(w[ks][0], emax + rx[ks][0]), tc_fix(w[ks][1], emax + rx[ks][1]));
        const uint4 z1 = tc_pack(tc_fix(w[ks][2], emax + rx[ks][2]), tc_fix(w[ks][3], emax + rx[ks][3]));
        const uint64_t *x = &sm.vec[sg][ks * 16 + 2 * t], *y = &sm.vec[sg8][ks * 16 + 2 * t];
        const uint4 x0 = *reinterpret_cast<const uint4 *>(x), x1 = *reinterpret_cast<const uint4 *>(x + 8);
        const uint4 y0 = *reinterpret_cast<const uint4 *>(y), y1 = *reinterpret_cast<const uint4 *>(y + 8);
        uint32_t db[8][2];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          db[j][0] = tc_digits(z0, j);
          db[j][1] = tc_digits(z1, j);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const uint32_t da[4] = {tc_digits(x0, k), tc_digits(y0, k), tc_digits(x1, k), tc_digits(y1, k)};
#pragma unroll
          for (int j = 0; k + j < 8; ++j) tc_mma(acc[k + j], da, db[j][0], db[j][1]);
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int64_t hi = tc_join(tc_int(acc[0][q], true), tc_int(acc[1][q], true),
                                   tc_int(acc[2][q], true), tc_int(acc[3][q], true));
        const int64_t lo = tc_join(tc_int(acc[4][q], true), tc_int(acc[5][q], true),
                                   tc_int(acc[6][q], true), tc_int(acc[7][q], true));
        out[c][q] = (hi << sh) + ((lo + (1ll << (31 - sh))) >> (32 - sh));
        // (an output without a term, padding too, has no error)
        if (dp[q] != 0.f) dp[q] += core;
      }
      if (last) {
        const int ua = 8 * c + 2 * t;
        const double ya0 = ua < N ? Y[ua * yn + j0] : 0.0, yb0 = ua + 1 < N ? Y[(ua + 1) * yn + j0] : 0.0;
        const double ya1 = ua < N ? Y[ua * yn + j1] : 0.0, yb1 = ua + 1 < N ? Y[(ua + 1) * yn + j1] : 0.0;
        const double r0 = tc_real(out[c][0], e0 + ea[c] + 88 - sh), r1 = tc_real(out[c][1], e0 + eb[c] + 88 - sh);
        const double r2 = tc_real(out[c][2], e1 + ea[c] + 88 - sh), r3 = tc_real(out[c][3], e1 + eb[c] + 88 - sh);
        v0 = __fma_rn(r0, ya0, v0);
        v0 = __fma_rn(r1, yb0, v0);
        v1 = __fma_rn(r2, ya1, v1);
        v1 = __fma_rn(r3, yb1, v1);
        d0 = __fma_rn(dif_real(dp[0], e0 + ea[c] + 124), fabs(ya0), d0);
        d0 = __fma_rn(dif_real(dp[1], e0 + eb[c] + 124), fabs(yb0), d0);
        d1 = __fma_rn(dif_real(dp[2], e1 + ea[c] + 124), fabs(ya1), d1);
        d1 = __fma_rn(dif_real(dp[3], e1 + eb[c] + 124), fabs(yb1), d1);
        // (below the range of doubles)
        bad |= (out[c][0] && tc_zero(r0)) || (out[c][1] && tc_zero(r1)) || (out[c][2] && tc_zero(r2)) ||
               (out[c][3] && tc_zero(r3));
      } else {
        // from here on at the scale of the next core's rows
        const int ua = 8 * c + 2 * t;
        const int32_t xa = ua < N ? g_row_exp[m + 1][ua] : 0, xb = ua + 1 < N ? g_row_exp[m + 1][ua + 1] : 0;
        if (xa == kNone) {
          out[c][0] = out[c][2] = 0;
          dp[0] = dp[2] = 0.f;
        }
        if (xb == kNone) {
          out[c][1] = out[c][3] = 0;
          dp[1] = dp[3] = 0.f;
        }
        dif[c][0] = bf_pair(dp[0], dp[1]);
        dif[c][1] = bf_pair(dp[2], dp[3]);
        if (ea[c] != TC_BAD) ea[c] += xa;
        if (eb[c] != TC_BAD) eb[c] += xb;
        if (out[c][0]) top0 = max(top0, ea[c] + 64 - __clzll(llabs(out[c][0])));
        if (out[c][1]) top0 = max(top0, eb[c] + 64 - __clzll(llabs(out[c][1])));
        if (out[c][2]) top1 = max(top1, ea[c] + 64 - __clzll(llabs(out[c][2])));
        if (out[c][3]) top1 = max(top1, eb[c] + 64 - __clzll(llabs(out[c][3])));
      }
    }
    bad = __any_sync(FULL, bad);
    __syncwarp();  // the rows are read
    if (last) {
      for (int o = 1; o < 4; o <<= 1) {
        v0 = __dadd_rn(v0, __shfl_xor_sync(FULL, v0, o));
        v1 = __dadd_rn(v1, __shfl_xor_sync(FULL, v1, o));
        d0 = __dadd_rn(d0, __shfl_xor_sync(FULL, d0, o));
        d1 = __dadd_rn(d1, __shfl_xor_sync(FULL, d1, o));
      }
      // (a D that is Inf - Inf fails the comparison too)
      const bool again = bad || !((t ? d1 : d0) <= 0.0) || tc_expo(t ? v1 : v0) == 0x7ff;
      if (t < 2 && g + 8 * t < rows) {
        sm.res[t ? sg8 : sg] = t ? v1 : v0;
        sm.unit[t ? sg8 : sg] = again;
      }
    } else {
      for (int o = 1; o < 4; o <<= 1) {
        top0 = max(top0, __shfl_xor_sync(FULL, top0, o));
        top1 = max(top1, __shfl_xor_sync(FULL, top1, o));
      }
      // rescale to 62 bits below each row's largest
#pragma unroll
      for (int c = 0; c < CT; ++c)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (g + 8 * h >= rows) continue;
          const int top = h ? top1 : top0;
          int64_t x0 = 0, x1 = 0;
          uint32_t dd = 0;
          if (8 * c < N) {
            // (a row of zeros that may not be one: D is whatever is above zero)
            float da = bf_lo(dif[c][h]), db = bf_hi(dif[c][h]);
            if (top != INT_MIN) {
              x0 = tc_shift(out[c][2 * h], 62 - (top - ea[c]));
              x1 = tc_shift(out[c][2 * h + 1], 62 - (top - eb[c]));
              da *= exp2_clamped(36 + sh + ea[c] - top);
              db *= exp2_clamped(36 + sh + eb[c] - top);
            } else {
              da = da != 0.f ? 0x1p100f : 0.f;
              db = db != 0.f ? 0x1p100f : 0.f;
            }
            dd = bf_pair(da, db);
          }
          *reinterpret_cast<uint32_t *>(&sm.dif[h ? sg8 : sg][8 * c + 2 * t]) = dd;
          *reinterpret_cast<uint4 *>(&sm.vec[h ? sg8 : sg][8 * c + 2 * t]) =
              tc_pack((uint64_t)x0 + TC_BIAS, (uint64_t)x1 + TC_BIAS);
        }
      if (t == 0) {
        if (g < rows) sm.unit[sg] = bad ? TC_BAD : top0 == INT_MIN ? 0 : e0 + 88 - sh + top0 - 62;
        if (g + 8 < rows) sm.unit[sg8] = bad ? TC_BAD : top1 == INT_MIN ? 0 : e1 + 88 - sh + top1 - 62;
      }
    }
  }
  __syncthreads();
}

// one slot per chunk of `chunk` samples (a multiple of S); the chunk depends on
// the sample count alone, and a sample's residual is its own, so the result is
// the same on any GPU
template <int KP>
__global__ void __launch_bounds__(kTcThreads, 1) k_tc_sums(ErrArgs a, int64_t chunk, int64_t nchunks,
                                                           double *sums) {
  using namespace ttc;
  extern __shared__ __align__(16) unsigned char tc_smem_raw[];
  TcSmem<KP> &sm = *reinterpret_cast<TcSmem<KP> *>(tc_smem_raw);
  constexpr int S = TcSmem<KP>::S;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int64_t c = blockIdx.x; c < nchunks; c += gridDim.x) {
    double num = 0.0, den = 0.0;
    for (int64_t k0 = c * chunk; k0 < min(a.nsamples, (c + 1) * chunk); k0 += S) {
      const int ns = (int)min((int64_t)S, a.nsamples - k0);
      // the first core's rows
      for (int s = tid; s < ns; s += kTcThreads) {
        const int K = a.s[1];
        const double *G = a.core[0] + (int64_t)coord(a, k0 + s, 0) * K;
        int emax = kNone;
        bool odd = false;
        for (int k = 0; k < K; ++k) {
          const int e = tc_expo(G[k]);
          odd |= tc_odd(G[k]);
          if (e && g_row_exp[1][k] != kNone) emax = max(emax, e + g_row_exp[1][k]);
        }
        auto fix = [&](int k) {
          return k < K && g_row_exp[1][k] != kNone ? tc_fix(G[k], emax - g_row_exp[1][k]) : TC_BIAS;
        };
        const float vec = kDifVec / (float)(a.d - 2);
        auto dif = [&](int k) {
          if (k >= K || g_row_exp[1][k] == kNone || tc_zero(G[k])) return 0.f;
          return vec - __uint_as_float(bf_abs(G[k], emax - g_row_exp[1][k]) << 16);
        };
        for (int k = 0; k < KP; k += 2) {
          *reinterpret_cast<uint4 *>(&sm.vec[s][k]) = tc_pack(fix(k), fix(k + 1));
          *reinterpret_cast<uint32_t *>(&sm.dif[s][k]) = bf_pair(dif(k), dif(k + 1));
        }
        sm.unit[s] = tc_unit_of(emax, odd);
      }
      if (tid == 0) sm.nagain = 0;
      for (int m = 1; m < a.d - 1; ++m) {
        tc_sort<KP>(a, k0, ns, m, sm);
        tc_core<KP>(a, k0, m, sm);
      }
      // the samples that fixed point is not exact enough for
      for (int s = tid; s < ns; s += kTcThreads)
        if (sm.unit[s]) sm.order[atomicAdd(&sm.nagain, 1)] = (uint16_t)s;
      __syncthreads();
      for (int x = warp; x < sm.nagain; x += kTcThreads / 32) {
        const int s = sm.order[x];
        const double xt = tt_value_warp<1>(a, k0 + s);
        if (lane == 0) sm.res[s] = xt;
      }
      __syncthreads();
      for (int s = tid; s < ns; s += kTcThreads) {
        const double x = entry(a, k0 + s), e = __dsub_rn(x, sm.res[s]);
        num = __fma_rn(e, e, num);
        den = __fma_rn(x, x, den);
      }
      __syncthreads();
    }
    for (int pass = 0; pass < 2; ++pass) {
      double v = pass ? den : num;
      for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
      if (lane == 0) sm.red[warp] = v;
      __syncthreads();
      if (tid == 0) {
        double s = 0.0;
        for (int i = 0; i < kTcThreads / 32; ++i) s += sm.red[i];
        sums[2 * c + pass] = s;
      }
      __syncthreads();
    }
  }
}

template <int KP>
cudaError_t launch_tc(const ErrArgs &a, int64_t chunk, int64_t nchunks, int nsm, double *sums,
                      cudaStream_t cs) {
  const void *f = (const void *)k_tc_sums<KP>;
  cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(TcSmem<KP>));
  if (e != cudaSuccess) return e;
  k_row_exp<<<dim3(32, (unsigned)(a.d - 2)), kThreads, 0, cs>>>(a);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int64_t grid = std::min<int64_t>(nchunks, nsm);
  k_tc_sums<KP><<<(unsigned)grid, kTcThreads, sizeof(TcSmem<KP>), cs>>>(a, chunk, nchunks, sums);
  return cudaGetLastError();
}

__global__ void __launch_bounds__(kThreads) k_finish(const double *sums, int64_t nchunks, double *out) {
  __shared__ double red[kWarps];
  double num = 0.0, den = 0.0;
  for (int64_t c = threadIdx.x; c < nchunks; c += kThreads) {
    num += sums[2 * c];
    den += sums[2 * c + 1];
  }
  const double sn = block_sum(num, red);
  const double sd = block_sum(den, red);
  if (threadIdx.x == 0) *out = sqrt(sn / sd);
}

ttc_status bad(ttc_status s, const char *msg) {
  ttc::set_last_error(msg);
  return s;
}

std::mutex g_mu;
double *g_sums[kMaxDevices] = {};

// Every kernel of this file on the current device: a kernel is loaded, which takes
// device memory, when it is first asked for
cudaError_t load_kernels() {
  const void *all[] = {(const void *)k_chunk_sums<1>, (const void *)k_chunk_sums<2>,
                       (const void *)k_chunk_sums<4>, (const void *)k_chunk_sums<8>,
                       (const void *)k_row_exp,       (const void *)k_tc_sums<16>,
                       (const void *)k_tc_sums<32>,   (const void *)k_finish};
  for (const void *f : all) {
    cudaFuncAttributes fa;
    const cudaError_t e = cudaFuncGetAttributes(&fa, f);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Device address of g_chunk_sums on device dev (the current device).  The
// first call on a device looks it up and keeps it, so that a later call made
// while the stream is being captured needs no lookup, and loads the kernels of
// all sizes, so that no later call does.  Calls outside a
// capture look it up again: after cudaDeviceReset the module is loaded anew
// and the array may sit elsewhere.
ttc_status scratch_on(int dev, bool capturing, double **out) {
  std::lock_guard<std::mutex> lk(g_mu);
  if (!g_sums[dev] || !capturing) {
    void *p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_chunk_sums);
    if (e != cudaSuccess || !p) {
      if (capturing) return bad(TTC_ERR_CUDA, "scratch address unknown: make a first call before capture");
      return bad(TTC_ERR_CUDA, "cudaGetSymbolAddress of the scratch failed");
    }
    if (!g_sums[dev] && load_kernels() != cudaSuccess) return bad(TTC_ERR_CUDA, "loading the kernels failed");
    g_sums[dev] = static_cast<double *>(p);
  }
  *out = g_sums[dev];
  return TTC_OK;
}

template <int K>
cudaError_t launch_sums(const ErrArgs &a, int64_t nchunks, int64_t grid, double *sums,
                        cudaStream_t cs) {
  k_chunk_sums<K><<<(unsigned)grid, kThreads, 0, cs>>>(a, nchunks, sums);
  return cudaGetLastError();
}

}  // namespace

extern "C" ttc_status ttcross_sampled_error_noalloc(int d, const int64_t *n, const ttc_generator *gen,
                                                    const double *const *cores, const int64_t *s,
                                                    int64_t nsamples, uint64_t seed, double *err,
                                                    void *stream) {
  ttc::set_last_error("");
  if (d < 2 || d > kMaxD) return bad(TTC_ERR_INVALID_ARG, "d outside [2,16]");
  if (!n || !gen || !cores || !s || !err) return bad(TTC_ERR_INVALID_ARG, "null argument");
  if (gen->kind != TTC_GEN_HILBERT && gen->kind != TTC_GEN_MAXWELLIAN)
    return bad(TTC_ERR_INVALID_ARG,
               "this entry point evaluates the Hilbert and Maxwellian generators only");
  ErrArgs a{};
  a.d = d;
  a.gen = gen->kind;
  int64_t total = 1;
  bool big = false;
  for (int m = 0; m < d; ++m) {
    if (n[m] < 1 || n[m] > (1 << 24)) return bad(TTC_ERR_INVALID_ARG, "mode size outside [1,2^24]");
    a.n[m] = n[m];
    if (total > ((int64_t)1 << 62) / n[m]) big = true; else total *= n[m];
    if (!cores[m]) return bad(TTC_ERR_INVALID_ARG, "null core pointer");
    a.core[m] = cores[m];
  }
  if (s[0] != 1 || s[d] != 1) return bad(TTC_ERR_INVALID_ARG, "core sizes must start and end with 1");
  for (int m = 0; m <= d; ++m) {
    if (s[m] < 1 || s[m] > kMaxRank) return bad(TTC_ERR_INVALID_ARG, "core size outside [1,256]");
    a.s[m] = (int32_t)s[m];
  }
  int smax = 1;
  for (int m = 0; m <= d; ++m) smax = std::max(smax, a.s[m]);
  if (gen->kind == TTC_GEN_MAXWELLIAN) {
    if (gen->dx < 1 || gen->dv < 1 || gen->dx + gen->dv != d)
      return bad(TTC_ERR_INVALID_ARG, "Maxwellian needs dx, dv >= 1 and dx + dv = d");
    for (int m = gen->dx; m < d; ++m)
      if (n[m] < 2) return bad(TTC_ERR_INVALID_ARG, "velocity modes need n >= 2");
    a.dx = gen->dx;
    a.dv = gen->dv;
    a.a_rho = gen->a_rho;
    a.a_u = gen->a_u;
    a.a_T = gen->a_T;
    a.vmin = gen->vmin;
    a.vmax = gen->vmax;
  }
  a.exhaustive = (nsamples <= 0 || (!big && nsamples >= total)) ? 1 : 0;
  a.nsamples = a.exhaustive ? total : nsamples;
  if (a.exhaustive && big) return bad(TTC_ERR_INVALID_ARG, "every-entry error on more than 2^62 entries");
  const int64_t nchunks = (a.nsamples + kChunk - 1) / kChunk;
  if (nchunks > kMaxChunks) {
    char msg[160];
    snprintf(msg, sizeof msg,
             "%lld samples exceed the static scratch of this entry point (at most %lld)",
             (long long)a.nsamples, (long long)kChunk * kMaxChunks);
    return bad(TTC_ERR_INVALID_ARG, msg);
  }
  a.seed = seed;
  int dev = 0, nsm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices)
    return bad(TTC_ERR_CUDA, "no usable current device");
  if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return bad(TTC_ERR_CUDA, "device query failed");
  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(cs, &cap) != cudaSuccess) return bad(TTC_ERR_CUDA, "stream query failed");
  double *sums = nullptr;
  ttc_status st = scratch_on(dev, cap != cudaStreamCaptureStatusNone, &sums);
  if (st != TTC_OK) return st;
  const int64_t grid = std::min<int64_t>(nchunks, (int64_t)nsm * 4);
  // the tensor-core form: sizes that fit its shared memory, samples enough to
  // fill the GPU's CTAs, and middle modes small enough that a CTA's 512 or 1024
  // samples share indices
  int64_t nmid = 0;
  for (int m = 1; m < d - 1; ++m) nmid = std::max(nmid, n[m]);
  const bool tc = d >= 3 && smax <= 32 && nmid <= kTcN && a.nsamples >= 16384;
  int64_t slots = nchunks;
  cudaError_t e;
  if (tc) {
    int64_t chunk = smax <= 16 ? TcSmem<16>::S : TcSmem<32>::S;
    while ((a.nsamples + chunk - 1) / chunk > kMaxChunks) chunk *= 2;
    slots = (a.nsamples + chunk - 1) / chunk;
    e = smax <= 16 ? launch_tc<16>(a, chunk, slots, nsm, sums, cs)
                   : launch_tc<32>(a, chunk, slots, nsm, sums, cs);
  } else if (smax <= 32)
    e = launch_sums<1>(a, nchunks, grid, sums, cs);
  else if (smax <= 64)
    e = launch_sums<2>(a, nchunks, grid, sums, cs);
  else if (smax <= 128)
    e = launch_sums<4>(a, nchunks, grid, sums, cs);
  else
    e = launch_sums<8>(a, nchunks, grid, sums, cs);
  if (e == cudaSuccess) {
    k_finish<<<1, kThreads, 0, cs>>>(sums, slots, err);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return bad(TTC_ERR_CUDA, cudaGetErrorString(e));
  return TTC_OK;
}
