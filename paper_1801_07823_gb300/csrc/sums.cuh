// Sums of doubles over a warp and over a few of its results, by alignment to the
// largest and integer addition, for the scalars on the critical path of the
// persistent kernels.  An FP64 addition takes 64 clocks on this device and a
// warp's tree of them five of those and ten shuffles; here the mantissas are
// aligned to the largest exponent, rounded to 58 bits and added exactly, which
// is also the closer sum (32 roundings of at most 2^-59 of the largest value
// against five of 2^-53 of the sum).
#pragma once
#include "digit.cuh"

namespace swsum {

// s 2^(e - 1080); e = 2047: not finite.
struct Aligned {
  long long s;
  int e;
};
__device__ __forceinline__ Aligned warp_sum(double v) {
  Aligned a;
  a.e = __reduce_max_sync(0xffffffffu, swdig::expo(v));
  const long long m = swdig::fixed(v, 0, a.e, 5);
  const unsigned l0 = __reduce_add_sync(0xffffffffu, (unsigned)m & 0x1fffffu);
  const unsigned l1 = __reduce_add_sync(0xffffffffu, (unsigned)(m >> 21) & 0x1fffffu);
  const int l2 = __reduce_add_sync(0xffffffffu, (int)(m >> 42));
  a.s = (long long)l0 + ((long long)l1 << 21) + ((long long)l2 << 42);
  return a;
}
// Sum of n <= 16 of them, rounded once.
template <int n>
__device__ __forceinline__ double total(const Aligned* a) {
  int e = 1;
#pragma unroll
  for (int k = 0; k < n; ++k) e = max(e, a[k].e);
  if (e == 2047) return __longlong_as_double(0x7ff8000000000000ll);
  long long H = 0, M = 0;  // the sum is (H 2^32 + M) 2^(e - 1104)
#pragma unroll
  for (int k = 0; k < n; ++k) {
    const int sh = min(e - a[k].e + 8, 95);
    H += a[k].s >> min(sh, 63);
    M += (unsigned)(sh < 32 ? a[k].s << (32 - sh) : a[k].s >> (sh - 32));
  }
  return swdig::to_double(H, M, e - 1104);
}

// Sum of G per-CTA parts in global memory, by one warp (valid in every lane); every CTA forms
// it in the same order.
__device__ __forceinline__ double grid_total(const double* parts, int G) {
  const int lane = threadIdx.x & 31;
  constexpr int kLoads = 5;  // 152 parts: one round trip
  double s = 0.0;
  for (int q0 = 0; q0 < G; q0 += 32 * kLoads) {
    double v[kLoads];
#pragma unroll
    for (int j = 0; j < kLoads; ++j) {
      const int q = q0 + 32 * j + lane;
      v[j] = q < G ? __ldcg(parts + q) : 0.0;
    }
#pragma unroll
    for (int j = 0; j < kLoads; ++j) s += v[j];
  }
  const Aligned a = warp_sum(s);
  return total<1>(&a);
}

}  // namespace swsum
