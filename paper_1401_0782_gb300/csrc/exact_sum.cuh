// Sums of doubles over a warp without rounding until the end, in fixed point on the
// integer pipe (a warp's FP64 instruction occupies its FP64 pipe for 64 cycles): every
// value becomes an integer multiple of a unit far below the last bit of the largest
// one, integers add exactly, and the total is rounded once.  The result does not depend
// on the order.  In place of the FP64 trees of p^T A p (means over ten inputs): T over 16
// columns of 24x24x120 378 ms (377 with trees), T and its gradient over 8 columns of
// 16x16x64 at two energies 84.8 ms (83.8).
#pragma once
#include <cuda_runtime.h>

#include "cplx.cuh"

namespace rsn {

// bits of a double as a multiple of 2^(top - 1075 - guard), rounded; top: the largest
// biased exponent of the sum's values
__host__ __device__ __forceinline__ long long to_fixed(long long bits, int top, int guard) {
  const int e = (int)(bits >> 52) & 0x7ff;
  long long m = bits & 0xfffffffffffffll;
  m = (e ? m | 0x10000000000000ll : m) << guard;
  const int sh = top - (e ? e : 1);
  m = sh < 62 ? (m + ((1ll << sh) >> 1)) >> sh : 0;
  return bits < 0 ? -m : m;
}

typedef __int128 i128;
typedef unsigned __int128 u128;

// the same with 128 bits: GUARD bits below the last bit of the largest value leave
// 74 - GUARD for the number of values
template <int GUARD>
__host__ __device__ __forceinline__ i128 to_fixed128(long long bits, int top) {
  const int e = (int)(bits >> 52) & 0x7ff;
  const long long m = (bits & 0xfffffffffffffll) | (e ? 0x10000000000000ll : 0ll);
  const int sh = top - (e ? e : 1);
  const i128 v = sh < 120 ? ((i128)m << GUARD) >> sh : 0;
  return bits < 0 ? -v : v;
}

// v * 2^-shift in [1, 2) * 2^63 with the lost bits in the last place: a double rounds it
// as it would round v
__host__ __device__ __forceinline__ unsigned long long top64(u128 v, int& shift) {
  unsigned long long hi = (unsigned long long)(v >> 64), lo = (unsigned long long)v;
  shift = 0;
  if (hi == 0) return lo;
#ifdef __CUDA_ARCH__
  const int lz = __clzll((long long)hi);
#else
  const int lz = __builtin_clzll(hi);
#endif
  shift = 64 - lz;
  const unsigned long long m = lz ? (hi << lz) | (lo >> (64 - lz)) : hi;
  const unsigned long long rest = lz ? lo << lz : lo;
  return m | (rest ? 1ull : 0ull);
}

__device__ __forceinline__ int top_exponent(double a) { return (__double2hiint(a) & 0x7fffffff) >> 20; }
__device__ __forceinline__ i128 shfl_xor128(i128 v, int w) {
  const unsigned long long hi = __shfl_xor_sync(0xffffffffu, (unsigned long long)(v >> 64), w);
  const unsigned long long lo = __shfl_xor_sync(0xffffffffu, (unsigned long long)v, w);
  return (i128)(((u128)hi << 64) | lo);
}

// The sums of re and of im over the warp: even lanes return that of re, odd ones of im.
// (Sums below 2^-950, infinities and NaN take the plain tree.)
__device__ __forceinline__ double warp_sum2_exact(double re, double im) {
  const bool odd = (threadIdx.x & 1) != 0;
  const int tr = __reduce_max_sync(0xffffffffu, top_exponent(re));
  const int ti = __reduce_max_sync(0xffffffffu, top_exponent(im));
  if (min(tr, ti) < 80 || max(tr, ti) >= 0x7ff) {
    double v[2] = {re, im};
    return warp_sum_many<2>(v);
  }
  const long long a = to_fixed(__double_as_longlong(re), tr, 5), b = to_fixed(__double_as_longlong(im), ti, 5);
  long long s = (odd ? b : a) + __shfl_xor_sync(0xffffffffu, odd ? a : b, 1);
#pragma unroll
  for (int w = 2; w < 32; w <<= 1) s += __shfl_xor_sync(0xffffffffu, s, w);
  // unit 2^(top - 1080)
  return __ll2double_rn(s) * __longlong_as_double((long long)((odd ? ti : tr) - 57) << 52);
}

// The sum of n >= 1 complex values over a warp, in every lane: in 64 bits, or, for many
// values, in 128.  Not inlined: inside an operator kernel it upset the allocation of
// the march's registers (FP32 register kernel, 24 uneven junctions: 619 us a launch,
// 506 as a call).
static __device__ __noinline__ double2 warp_sum_parts(const double2* part, int n) {
  constexpr int KEEP = 4, GUARD = 40;  // values a lane keeps between the passes; n < 2^33
  const int lane = threadIdx.x & 31;
  const bool odd = (lane & 1) != 0;
  double2 w[KEEP];
  int tr = 1, ti = 1;  // (denormals have the exponent 0 and the unit of 1)
#pragma unroll
  for (int k = 0; k < KEEP; ++k) {
    w[k] = make_double2(0.0, 0.0);
    if (lane + 32 * k < n) w[k] = __ldcg(part + lane + 32 * k);
  }
#pragma unroll
  for (int k = 0; k < KEEP; ++k) {
    tr = max(tr, top_exponent(w[k].x));
    ti = max(ti, top_exponent(w[k].y));
  }
  for (int t = lane + 32 * KEEP; t < n; t += 32) {
    const double2 v = __ldcg(part + t);
    tr = max(tr, top_exponent(v.x));
    ti = max(ti, top_exponent(v.y));
  }
  tr = __reduce_max_sync(0xffffffffu, tr);
  ti = __reduce_max_sync(0xffffffffu, ti);
  if (max(tr, ti) >= 0x7ff) {  // infinities or NaN
    double v[2] = {0.0, 0.0};
    for (int t = lane; t < n; t += 32) {
      const double2 p = __ldcg(part + t);
      v[0] += p.x;
      v[1] += p.y;
    }
    const double t = warp_sum_many<2>(v);
    return make_double2(__shfl_sync(0xffffffffu, t, 0), __shfl_sync(0xffffffffu, t, 1));
  }
  if (n <= 512 && min(tr, ti) >= 80) {
    // 64 bits: at least one bit below the last one of the largest value for up to 256
    // values (110 of them, rounded to a quarter of it: 0.8 of it rms, which is less than
    // the rounding of a total a few times as large)
    const int guard = 9 - (32 - __clz(n - 1));
    long long re = 0, im = 0;
#pragma unroll
    for (int k = 0; k < KEEP; ++k) {
      re += to_fixed(__double_as_longlong(w[k].x), tr, guard);
      im += to_fixed(__double_as_longlong(w[k].y), ti, guard);
    }
    for (int t = lane + 32 * KEEP; t < n; t += 32) {
      const double2 v = __ldcg(part + t);
      re += to_fixed(__double_as_longlong(v.x), tr, guard);
      im += to_fixed(__double_as_longlong(v.y), ti, guard);
    }
    long long s = (odd ? im : re) + __shfl_xor_sync(0xffffffffu, odd ? re : im, 1);
#pragma unroll
    for (int x = 2; x < 32; x <<= 1) s += __shfl_xor_sync(0xffffffffu, s, x);
    const double v = __ll2double_rn(s) * __longlong_as_double((long long)((odd ? ti : tr) - 52 - guard) << 52);
    return make_double2(__shfl_sync(0xffffffffu, v, 0), __shfl_sync(0xffffffffu, v, 1));
  }
  i128 re = 0, im = 0;
#pragma unroll
  for (int k = 0; k < KEEP; ++k) {
    re += to_fixed128<GUARD>(__double_as_longlong(w[k].x), tr);
    im += to_fixed128<GUARD>(__double_as_longlong(w[k].y), ti);
  }
  for (int t = lane + 32 * KEEP; t < n; t += 32) {
    const double2 v = __ldcg(part + t);
    re += to_fixed128<GUARD>(__double_as_longlong(v.x), tr);
    im += to_fixed128<GUARD>(__double_as_longlong(v.y), ti);
  }
  i128 s = (odd ? im : re) + shfl_xor128(odd ? re : im, 1);
#pragma unroll
  for (int x = 2; x < 32; x <<= 1) s += shfl_xor128(s, x);
  int shift;
  const unsigned long long m = top64((u128)(s < 0 ? -s : s), shift);
  const double v = scalbn(__ull2double_rn(m), shift + (odd ? ti : tr) - 1075 - GUARD), u = s < 0 ? -v : v;
  return make_double2(__shfl_sync(0xffffffffu, u, 0), __shfl_sync(0xffffffffu, u, 1));
}

}  // namespace rsn
