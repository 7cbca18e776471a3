// ttc_split.cuh -- FP64 products as exact integer products on the tensor cores:
// the fixed-point rows, their digits and the sums of the digit products (the
// scheme and its bounds are described in ttc_error.cuh).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace ttc {

constexpr uint64_t TC_BIAS = 0x8080808080808080ull;
constexpr int32_t TC_BAD = 0x7fffffff;  // exponent of a row / column with an Inf or NaN

__host__ __device__ __forceinline__ int64_t tc_up(int64_t x, int64_t to) {
  return (x + to - 1) / to * to;
}

// the exponent field of x (0: zero or subnormal, taken as zero; 0x7ff: not finite)
__device__ __forceinline__ int tc_expo(double x) {
  return (__double2hiint(x) >> 20) & 0x7ff;
}
// x as a biased integer in units of 2^(emax - 1084), |x| < 2^(emax - 1022)
__device__ __forceinline__ uint64_t tc_fix(double x, int emax) {
  const int e = tc_expo(x);
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  const int s = 9 - (emax - e);
  uint64_t m = (b & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull;
  if (e == 0 || s < -54)
    m = 0;
  else if (s >= 0)
    m <<= s;
  else
    m = (m + (1ull << (-s - 1))) >> -s;
  return ((b >> 63) ? 0ull - m : m) + TC_BIAS;
}
// exponent of the units for a row whose largest exponent field is emax
__device__ __forceinline__ int32_t tc_unit(int emax) { return emax == 0x7ff ? TC_BAD : emax - 1084; }

// the bytes of two biased integers interleaved
__device__ __forceinline__ uint4 tc_pack(uint64_t x, uint64_t y) {
  const uint32_t xh = (uint32_t)(x >> 32), yh = (uint32_t)(y >> 32), xl = (uint32_t)x, yl = (uint32_t)y;
  return make_uint4(__byte_perm(xh, yh, 0x6273), __byte_perm(xh, yh, 0x4051),
                    __byte_perm(xl, yl, 0x6273), __byte_perm(xl, yl, 0x4051));
}

// v 2^s, to nearest (the result fits by the caller's choice of s)
__device__ __forceinline__ int64_t tc_shift(int64_t v, int s) {
  if (s >= 0) return (int64_t)((uint64_t)v << s);
  return s < -62 ? 0 : (v + (1ll << (-s - 1))) >> -s;
}

// v 2^n as a double, to nearest, |v| < 2^62, on the integer pipe (a conversion
// from int64 takes the FP64 pipe, which the tail of a check needs for its dots)
__device__ __forceinline__ double tc_real(int64_t v, int n) {
  const uint64_t a = (uint64_t)(v < 0 ? -v : v);
  const int z = __clzll((long long)a);
  const uint64_t frac = ((a << (z - 1)) + 0x200u) >> 10;  // in [2^52, 2^53]
  const int e = 1085 - z + n;                             // exponent field less one
  if (a == 0 || e < 0) return 0.0;
  const uint64_t s = v < 0 ? 0x8000000000000000ull : 0ull;
  if (e >= 0x7fe) return __longlong_as_double((long long)(s | 0x7FF0000000000000ull));
  return __longlong_as_double((long long)(s | (((uint64_t)e << 52) + frac)));
}

// digit k (0: most significant) of a pair as f16s: 1024 + byte, minus 1152
__device__ __forceinline__ uint32_t tc_digits(const uint4 &q, int k) {
  const uint32_t w = k < 2 ? q.x : k < 4 ? q.y : k < 6 ? q.z : q.w;
  const uint32_t y = __byte_perm(w, 0x64646464u, k & 1 ? 0x4342 : 0x4140);
  uint32_t h;
  asm("sub.f16x2 %0, %1, %2;" : "=r"(h) : "r"(y), "r"(0x64806480u));
  return h;
}

__device__ __forceinline__ void tc_mma(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The sums' FP32 values to integers.  Up to kp = 32 they stay below 2^22, and
// the accumulators start at 1.5 2^23 (TC_MAGIC), whose last bit is one: the
// integer is the difference of the bits.  (A conversion runs at 16 lanes a
// clock and SM; 32 of them per column tile would cost as much as half the
// products of a kp = 32 tile.)
constexpr float TC_MAGIC = 12582912.f;
__device__ __forceinline__ int32_t tc_int(float s, bool magic) {
  return magic ? __float_as_int(s) - __float_as_int(TC_MAGIC) : __float2int_rn(s);
}
// four levels, most significant first, as one integer
__device__ __forceinline__ int64_t tc_join(int32_t s0, int32_t s1, int32_t s2, int32_t s3) {
  const int64_t a = (int64_t)s0 * 256 + s1;
  return (a << 16) + ((int64_t)s2 * 256 + s3);
}

}  // namespace ttc
