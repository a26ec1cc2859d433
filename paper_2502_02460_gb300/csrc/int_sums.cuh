// Sums of FP64 values formed in integer arithmetic (GB300 has about 1.7 FP64 operations per SM per cycle, conversions
// and comparisons included; integer instructions cost a small part of that).
#pragma once
#include "common.cuh"

namespace gev {

// The sum of N <= 63 FP64 values in integer arithmetic: each is taken to 57 bits below the largest exponent and added
// as a 64-bit integer, the total is rounded once.  An FP64 addition occupies a scheduler's pipe for 64 to 72 cycles, the
// dozen integer instructions here for about 24.  The error is below N 2^-56 of the largest value (N 2^-53 of the partial
// sums for additions), and the result does not depend on the order.  Exponents near either end: additions.
template <int N> __device__ __forceinline__ double sum_block(const double (&v)[N]) {
  static_assert(N < 64, "57 bits and the sum's carry fit 63");
  int emax = 0;
#pragma unroll
  for (int u = 0; u < N; ++u) emax = max(emax, (__double2hiint(v[u]) >> 20) & 0x7FF);
  if (emax < 100 || emax > 2000) {
    double t = 0.0;
#pragma unroll
    for (int u = 0; u < N; ++u) t += v[u];
    return t;
  }
  long long acc = 0;
#pragma unroll
  for (int u = 0; u < N; ++u) {
    const long long b = __double_as_longlong(v[u]);
    const int sh = emax - ((int)(b >> 52) & 0x7FF);
    const long long m = ((b & 0xFFFFFFFFFFFFFll) | (1ll << 52)) << 4;
    const long long x = sh > 62 ? 0 : m >> sh;
    acc += b < 0 ? -x : x;
  }
  if (acc == 0) return 0.0;
  unsigned long long mag = acc < 0 ? 0ull - (unsigned long long)acc : (unsigned long long)acc;
  const int lz = __clzll((long long)mag);
  mag <<= lz;
  const unsigned lo = (unsigned)mag & 0x7FFu;
  unsigned long long r = mag >> 11;
  r += (lo > 0x400u || (lo == 0x400u && (r & 1))) ? 1 : 0;
  r += (unsigned long long)(emax + 6 - lz) << 52;  // (the mantissa's leading bit adds one to the exponent)
  return __longlong_as_double((long long)(r | (acc < 0 ? 1ull << 63 : 0ull)));
}
template <int N> __device__ __forceinline__ zd sum_block(const zd (&v)[N]) {
  double a[N], b[N];
#pragma unroll
  for (int u = 0; u < N; ++u) {
    a[u] = v[u].x;
    b[u] = v[u].y;
  }
  return make_zd(sum_block(a), sum_block(b));
}
template <int N> __device__ __forceinline__ float sum_block(const float (&v)[N]) {
  float t = 0.f;
#pragma unroll
  for (int u = 0; u < N; ++u) t += v[u];
  return t;
}

// (acc 2^-49 + sh) 2^e rounded once to FP64, in integer arithmetic: GB300 runs about 1.7 FP64 operations
// (conversions included) per SM per cycle, and at eight of them per output the epilogue of a 128 x 64
// tile took about 19 us.  sh (|sh| < 2^-18) joins acc in units of 2^-81 (acc:lo, 96 bits); the magnitude is
// normalised with a count of leading zeros and rounded to nearest even, subnormal results included.
__device__ __forceinline__ double to_fp64(long long acc, float sh, int e) {
  const uint32_t sb = __float_as_uint(sh);
  const int se = (int)((sb >> 23) & 0xFF);
  const unsigned long long sm = (sb & 0x7FFFFFu) | 0x800000u;
  const int sft = se - 150 + 81;  // sh 2^81 = sm 2^sft (a zero or denormal sh has sft < -24)
  long long si = sft >= 0 ? (long long)(sm << sft) : (sft > -25 ? (long long)(sm >> -sft) : 0);
  if (sb >> 31) si = -si;
  acc += si >> 32;
  uint32_t lo = (uint32_t)si;
  const bool neg = acc < 0;
  unsigned long long m = (unsigned long long)acc;
  if (neg) {  // two's complement of the 96 bits
    lo = 0u - lo;
    m = ~m + (lo == 0 ? 1ull : 0ull);
  }
  int ex = 63 - 49 + e;  // exponent of bit 63 of m
  if ((m >> 32) == 0) {
    m = (m << 32) | lo;
    lo = 0;
    ex -= 32;
  }
  if (m == 0) return 0.0;
  const int lz = __clzll((long long)m);
  const unsigned long long low = ((unsigned long long)lo) << lz;  // lz < 32 whenever lo != 0
  m = (m << lz) | (low >> 32);
  ex -= lz;
  // m 2^(ex - 63), rounded at bit `drop`: 11 bits off a normal result, more off a subnormal one
  const bool normal = ex >= -1022;
  const int drop = normal ? 11 : min(65, 11 - 1022 - ex);
  unsigned long long b = drop < 64 ? m >> drop : 0ull;
  const unsigned long long rem = drop < 65 ? m << (64 - drop) : 0ull;  // the dropped bits, aligned to the top
  if (rem > 1ull << 63 || (rem == 1ull << 63 && ((uint32_t)low != 0u || (b & 1)))) ++b;
  // (a carry to 2^53 moves the exponent up by itself: the fields add, up to infinity)
  if (normal) b += (unsigned long long)(ex + 1022) << 52;
  if (ex > 1023) b = 0x7FF0000000000000ull;
  return __longlong_as_double((long long)(b | (neg ? 1ull << 63 : 0ull)));
}

// The same where neither zero, NaN, overflow nor subnormal results can occur (|e| < 1000): sh is split into
// 32-bit integer and fraction by FP32 conversions (the fraction of a negative sh rounds at 2^-74), and the 96 bits
// are normalised as three words with funnel shifts.  About half the instructions; with the other per-output work
// thinned out too, a 6144 x 6144 x 128 update went from 515 to 330 us (splits included; its MMAs are about 160).
__device__ __forceinline__ double to_fp64_fast(long long acc, float sh, int e, uint32_t flip) {
  const float x = sh * 562949953421312.0f;  // 2^49: |x| < 2^31
  const int xi = __float2int_rd(x);
  uint32_t l = __float2uint_rz((x - __int2float_rn(xi)) * 4294967296.0f);  // the fraction, [0, 1)
  acc += xi;
  const uint32_t neg = (uint32_t)((int)(acc >> 32) >> 31);  // all ones for a negative sum: two's complement
  const unsigned long long mag = ((unsigned long long)acc ^ (((unsigned long long)neg << 32) | neg)) + (l == 0 ? neg & 1u : 0u);
  l = (l ^ neg) + (neg & 1u);
  uint32_t h = (uint32_t)(mag >> 32), m = (uint32_t)mag;
  int ex = 63 - 49 + e + 1022;
  if (h == 0) {
    h = m;
    m = l;
    l = 0;
    ex -= 32;
    if (h == 0) {
      h = m;
      m = 0;
      ex -= 32;
      if (h == 0) return 0.0;
    }
  }
  const int lz = __clz((int)h);
  h = __funnelshift_l(m, h, lz);
  m = __funnelshift_l(l, m, lz);
  const uint32_t t = (m & 0x7FFu) | ((l << lz) != 0u ? 1u : 0u), up = (t + 0x3FFu + ((m >> 11) & 1u)) >> 11;
  const uint32_t w0 = __funnelshift_r(m, h, 11), r0 = w0 + up;
  const uint32_t w1 = (h >> 11) + (r0 < w0 ? 1u : 0u) + ((uint32_t)(ex - lz) << 20);
  return __hiloint2double((int)(w1 | ((neg ^ flip) & 0x80000000u)), (int)r0);
}

}  // namespace gev
