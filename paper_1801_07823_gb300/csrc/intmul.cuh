// FP64 products and sums by 32-bit integer multiply-adds.
//
// GB300 issues two FP64 FMAs per clock and SM, so an FP64 operator waits for
// that pipe while the integer units (64 operations per clock) idle.  Here its
// products are formed in integers: the operands of a sum share one power of two
// each (that of the largest component), are cut to 59 bits and written as
// h 2^30 + l; three of the four digit products of a pair are kept (the fourth is
// below 2^-58 of the largest product), added up exactly, and the sum is rounded
// to FP64 once.  Before that rounding a sum of eight products (four complex
// ones, one component) is off by less than 2^-53 of the product of the two
// largest components, typically 2^-57 of it; a chain of FP64 FMAs rounds eight
// times.  With Gaussian operands the relative 2-norm error is 0.33e-16
// against 1.5e-16.
//
// Infinities, NaN and operands whose largest component is close to the subnormal range are
// left to FP64 (usable).
#pragma once
#include "digit.cuh"

namespace swint {

struct Num {
  int h, l;  // (h 2^30 + l), |h| < 2^29, |l| < 2^30
};
struct Cplx {
  Num x, y;
};
__device__ __forceinline__ Num operator-(Num a) { return Num{-a.h, -a.l}; }

__device__ __forceinline__ unsigned magnitude(double x) {
  return (unsigned)__double2hiint(x) & 0x7fffffffu;
}
__device__ __forceinline__ unsigned magnitude(double2 v) {
  return max(magnitude(v.x), magnitude(v.y));
}
// The exponent field of the largest of some components, from the largest magnitude().  Below
// 64 the implicit bit that num() always sets would show.
__device__ __forceinline__ bool usable(int e) { return e >= 64 && e < 2047; }

// x 2^(1081 - e) cut to an integer; e at least the exponent field of x.
__device__ __forceinline__ Num num(double x, int e) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int sh = e - (int)((hi >> 20) & 0x7ffu);
  const unsigned mh = (hi & 0xfffffu) | 0x100000u;
  unsigned long long m = ((unsigned long long)((mh << 6) | (lo >> 26)) << 32) | (lo << 6);
  asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(sh));  // shifts of 64 and more give 0
  const int h = (int)(m >> 30), l = (int)(m & 0x3fffffffu);
  return (int)hi < 0 ? Num{-h, -l} : Num{h, l};
}
__device__ __forceinline__ Cplx num(double2 v, int e) { return Cplx{num(v.x, e), num(v.y, e)}; }

// Sums of up to eight products a component: H 2^60 + M 2^30 in units of the operands' last
// places; |H| < 2^61, |M| < 2^63.
struct Sum {
  long long H = 0, M = 0;
  __device__ __forceinline__ void add(Num a, Num b) {
    H += (long long)a.h * b.h;
    M += (long long)a.h * b.l;
    M += (long long)a.l * b.h;
  }
  // the sum of products of operands with exponent fields ea and eb
  __device__ __forceinline__ double value(int ea, int eb) const {
    // H 2^30 + M as H' 2^32 + M', M' = M + (H mod 4) 2^30 carried over by hand
    const unsigned long long low = (unsigned long long)(H & 3) << 30;
    const long long hi = (H >> 2) + (M >> 32);
    const unsigned long long lo = (unsigned)M + low;  // < 2^33
    return swdig::to_double(hi, (long long)lo, ea + eb - 2132);
  }
};
struct Csum {
  Sum x, y;
  __device__ __forceinline__ void add(Cplx a, Cplx b) {  // += a b
    x.add(a.x, b.x);
    x.add(-a.y, b.y);
    y.add(a.x, b.y);
    y.add(a.y, b.x);
  }
  __device__ __forceinline__ double2 value(int ea, int eb) const {
    return make_double2(x.value(ea, eb), y.value(ea, eb));
  }
};

// Links W = eta U / 2: components of at most 1/2.
constexpr int kLinkExp = 1022;
__device__ __forceinline__ bool link_usable(unsigned mag) { return mag <= (unsigned)kLinkExp << 20; }

}  // namespace swint
