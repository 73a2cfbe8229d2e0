// FP64 stencil products on the FP16 tensor cores, by exact digit arithmetic.
//
// GB300 runs FP64 at 4 flop per clock per SM, so a coarse stencil in plain
// FP64 (about 0.5 flop per byte) is bound by the FP64 pipe and leaves memory
// idle.  Here every operand is written as an integer of eight base-256
// digits, the digit products run as FP16 MMAs with FP32 accumulators, in which
// every product and sum is an exact integer, and the integer result is rounded
// to FP64 once.  (Splitting operands so that a matrix unit sums their parts
// without rounding is Ozaki, Ogita, Oishi, Rump, "Error-free transformations
// of matrix multiplication by using fast routines of matrix multiplication",
// Numer. Algorithms 59 (2012).)
//
// Numbers.  A row of A is scaled by the power of two of its largest component
// and rounded to 64 bits (u_0 - 128, u_1, .., u_7), u unsigned bytes; the
// vectors of a site's five neighbours share one power of two and are rounded to 63 bits in balanced digits d_0 .. d_7 in [-128, 127].  Of the 64
// digit products those of level i + j <= 7 are kept; the others are below
// 2^-59 of the largest product.  Against exact arithmetic the products are 2
// to 10 times closer than the FP64 kernels they take the place of (the
// operands' rounding is below FP64's accumulated rounding): measured on Galerkin
// stencils with Gaussian, smooth and localised vectors, relative 2-norm error
// 0.4e-16 to 0.8e-16 against 1.0e-16 to 5.9e-16.  Fixed point has a range: an entry 2^-k
// below its row's largest keeps 64 - k bits, a vector element 63 - k, so that rows and vectors
// graded against each other (large entries on small elements) lose what FP64 would keep; the
// error bound is one of the two scales, not of every term.
//
// MMA shape.  mma.m16n8k16 with M = the real and imaginary parts of eight
// output rows, N = the eight levels, K = four entries times four digits: the
// operand of entry a holds its digits i, that of the vector the digits n - i,
// so an accumulator is a level.  Digits 0..3 of an entry meet the vector's real
// and imaginary part (two MMAs); digits 4..7 only reach levels 4..7, so one MMA
// takes the real and imaginary parts side by side: 12 MMAs for eight rows by
// sixteen columns.  The byte u is read as the FP16 subnormal u 2^-24, which
// costs one byte permutation per two operands and no conversion.  A sum over
// eight k-steps is at most 128 * 4 * 255 * 128 < 2^24, exact in the FP32
// accumulator.  (With K = sixteen columns and N = the vector's digits the same
// MMAs need half as many permutations again and four times the accumulators: 190
// to 210 clocks of a sub-partition per k-step, bound by its integer pipe.)
// tcgen05 would have to see the expanded FP16 operands in shared memory, twice
// the bytes that the L2 delivers; with N = 8 the register path of mma.sync
// (measured 944 multiply-adds per clock and SM) keeps up with the L2.
//
// Layout.  An entry is two 64-bit integers (real, imaginary part, offset by
// 2^63 so that every digit is an unsigned byte).  A block, padded to nP x nP
// with nP a multiple of eight, is a column-major array of 4 x 4 tiles of
// entries; in a tile the two rows of a 128-byte line lie together, and in a
// line the two columns of 64 bytes (tile_place).  One copy serves A and A^dag:
// a load of eight lanes covers one line (A: two rows, four columns) or two
// halves of lines (A^dag: four rows, two columns), and the L1 takes a line a
// clock.  With plain column-major entries, where eight lanes of A touch four
// lines, the loads ran at 33 bytes per clock and SM, half of what the L2 gives.
// The row scales of A are applied to the result of A and, before its digits
// are taken, to the vector of A^dag.
#pragma once
#include <cuda_fp16.h>

#include "sw_internal.h"

namespace swdig {

constexpr int kMaxSteps = 8;            // k-steps summed before the accumulators are emptied
constexpr int kLevels = 8;              // digit levels kept
// Level sums of an item (eight rows of a site): level l, component c, row g at 20 l + 8 c + g.
// Lanes 4 g + t add to levels 2 t + const, so that this stride keeps their banks apart.
constexpr int kSLevel = 20;
constexpr int kSItem = kLevels * kSLevel;
constexpr int kNotFinite = 1 << 20;     // exponent that marks an infinity or NaN

// nc x nc blocks on an E0 x E1 lattice: RG groups of eight rows per site, nP = 8 RG, KQ quads
// of columns per direction, KS k-steps (four quads each) per row.
struct Shape {
  int E0, E1, nc, nP, KQ, KS, RG;
};
inline Shape shape_of(const CoarseGeom& g) {
  Shape s;
  s.E0 = g.E0;
  s.E1 = g.E1;
  s.nc = g.nc;
  s.RG = (g.nc + 7) / 8;
  s.nP = 8 * s.RG;
  s.KQ = 2 * s.RG;
  s.KS = (5 * s.KQ + 3) / 4;
  return s;
}

// Place of (row i, column j) in its 4 x 4 tile.
__host__ __device__ __forceinline__ int tile_place(int i, int j) {
  return (i & 2) * 4 + (j & 2) * 2 + (i & 1) * 2 + (j & 1);
}
// First tile of quad q (four columns of A, four rows of A^dag) of site X's row group 0.
template <bool DAG>
__device__ __forceinline__ int quad_offset(const Shape& s, int X, int q) {
  if (q >= 5 * s.KQ) q = 0;  // padding of the last k-step: its vector digits are zero
  const int d = q / s.KQ, c = 4 * (q - d * s.KQ);
  if (!DAG) return ((X * 5 + d) * s.nP + c) * s.nP;
  return (nbr(X, d, s.E0, s.E1) * 5 + opp(d)) * s.nP * s.nP + 4 * c;
}
// The four quads of k-step ks of site X; entries from one row group to the next.
template <bool DAG>
__device__ __forceinline__ int4 kstep_offsets(const Shape& s, int X, int ks) {
  const int q = 4 * ks;
  return make_int4(quad_offset<DAG>(s, X, q), quad_offset<DAG>(s, X, q + 1),
                   quad_offset<DAG>(s, X, q + 2), quad_offset<DAG>(s, X, q + 3));
}
__device__ __forceinline__ int group_step(const Shape& s, bool dag) { return dag ? 8 * s.nP : 32; }
// The lane's part: lane 4 g + t takes row g and column t of every quad.
__device__ __forceinline__ int lane_offset(const Shape& s, bool dag) {
  const int g = (threadIdx.x & 31) >> 2, t = threadIdx.x & 3;
  return dag ? (g >> 2) * 4 * s.nP + tile_place(t, g) : (g >> 2) * 16 + tile_place(g, t);
}

// Biased exponent of x, 1 for subnormals and zero: x = +-mant 2^(e - 1075).
__device__ __forceinline__ int expo(double x) {
  const int e = (__double2hiint(x) >> 20) & 0x7ff;
  return e > 1 ? e : 1;
}
// x 2^(shift + 1075 - emax + bits) as an integer, rounded to nearest
// (emax >= expo(x) + shift).
__device__ __forceinline__ long long fixed(double x, int shift, int emax, int bits) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  unsigned long long m = b & 0xfffffffffffffull;
  const int e = (int)(b >> 52) & 0x7ff;
  if (e) m |= 1ull << 52;
  m <<= bits;
  const int sh = emax - (e > 1 ? e : 1) - shift;
  if (sh > 0) m = sh < 64 ? (m + (1ull << (sh - 1))) >> sh : 0ull;
  return (long long)b < 0 ? -(long long)m : (long long)m;
}

// Rounds (H 2^32 + M) 2^k to the nearest double (ties to even): the final
// step of a row, in integer arithmetic because the FP64 pipe is the scarce one.
__device__ __forceinline__ double to_double(long long H, long long M, int k) {
  long long hi = H + (M >> 32);
  unsigned lo = (unsigned)M;
  const bool neg = hi < 0;
  if (neg) {
    hi = -hi - (lo ? 1 : 0);
    lo = 0u - lo;
  }
  unsigned long long top = (unsigned long long)hi, low = (unsigned long long)lo << 32;
  int e = 95;  // exponent of bit 63 of top
  if (top == 0) {
    if (low == 0) return 0.0;
    top = low;
    low = 0;
    e = 31;
  }
  const int lz = __clzll((long long)top);
  if (lz) {
    top = (top << lz) | (low >> (64 - lz));
    low <<= lz;
  }
  e += k - lz;
  unsigned long long mant = top >> 11;
  const unsigned rem = (unsigned)top & 0x7ffu;
  if (rem > 0x400u || (rem == 0x400u && (low != 0 || (mant & 1)))) ++mant;
  const bool in_range = e > -1022 && e < 1023;
  unsigned long long bits = ((unsigned long long)(in_range ? e + 1022 : 1022) << 52) + mant;
  if (neg) bits |= 1ull << 63;
  const double v = __longlong_as_double((long long)bits);
  return in_range ? v : scalbn(v, e);
}

// ------------------------------------------------------------ vector digits
// Digits of the neighbour vectors in shared memory: per quad of columns kQuadBytes, real part
// first; column t of the quad and level n at 32 n + 8 t hold the four FP16 digits n, n - 1,
// n - 2, n - 3, so that a lane reads its MMA operand (level lane / 4, column lane & 3) at 8 *
// lane.  The 32 bytes between quads keep the writers of neighbouring columns on separate banks.
constexpr int kQuadBytes = 544;
__device__ __forceinline__ void put_digits(double x, int shift, int emax, unsigned char* dst) {
  const unsigned long long s =
      (unsigned long long)fixed(x, shift, emax, 9) + 0x8080808080808080ull;  // |fixed| < 2^62
  const unsigned hi = (unsigned)(s >> 32), lo = (unsigned)s;
  const __half2 bias = __floats2half2_rn(1152.f, 1152.f);
  unsigned q[4];  // digits 2 k (low half) and 2 k + 1
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const unsigned p = __byte_perm(k < 2 ? hi : lo, 0x64646464u, (k & 1) ? 0x4041u : 0x4243u);
    const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&p), bias);  // 1024 + u - 1152
    q[k] = *reinterpret_cast<const unsigned*>(&h);
  }
  unsigned p2 = 0, p1 = 0;  // (digit n - 2, n - 3), (digit n - 1, n - 2)
#pragma unroll
  for (int n = 0; n < 8; ++n) {
    const unsigned p = (n & 1) ? __byte_perm(q[n >> 1], 0u, 0x1032)
                               : __byte_perm(q[n >> 1], n ? q[(n >> 1) - 1] : 0u, 0x7610);
    *reinterpret_cast<uint2*>(dst + 32 * n) = make_uint2(p, p2);
    p2 = p1;
    p1 = p;
  }
}
// Column c (padded, direction by direction, site by site).
__device__ __forceinline__ void put_column(double2 x, int shift, int emax, unsigned char* B,
                                           int c) {
  unsigned char* dst = B + (size_t)(c >> 2) * kQuadBytes + 8 * (c & 3);
  put_digits(x.x, shift, emax, dst);
  put_digits(x.y, shift, emax, dst + 256);
}
// Exponent of a vector element with its row scale (A^dag; A: shift 0).
__device__ __forceinline__ int column_expo(double2 x, int shift) {
  const int e = max(expo(x.x), expo(x.y));
  return e == 2047 || shift >= 1024 ? kNotFinite : e + shift;
}

// ------------------------------------------------------------ products
// v = *p if go; a predicate and not a branch, behind which the compiler would wait.
__device__ __forceinline__ void ld_entry(uint4& v, const uint4* p, bool go,
                                         unsigned long long pol) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %6, 0;\n\t"
      "@q ld.global.nc.L1::no_allocate.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;\n\t}"
      : "+r"(v.x), "+r"(v.y), "+r"(v.z), "+r"(v.w)
      : "l"(p), "l"(pol), "r"((int)go));
}
__device__ __forceinline__ void mma(float (&c)[4], unsigned a0, unsigned a1, unsigned a2,
                                    unsigned a3, uint2 b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b.x), "r"(b.y));
}
// Accumulators of one item (eight rows of a site): digits 0..3 against the vector's real and
// imaginary part, levels 0..7; digits 4..7, levels 4..7 against both.
struct Acc {
  float re[4], im[4], lo[4];
};
__device__ __forceinline__ void clear(Acc& a) {
#pragma unroll
  for (int k = 0; k < 4; ++k) a.re[k] = a.im[k] = a.lo[k] = 0.f;
}
// A lane's vector digits of a quad.
struct Digits {
  uint2 re, im, lo;
};
__device__ __forceinline__ Digits ld_digits(const unsigned char* b) {
  const int lane = threadIdx.x & 31;
  Digits d;
  d.re = *reinterpret_cast<const uint2*>(b + 8 * lane);
  d.im = *reinterpret_cast<const uint2*>(b + 256 + 8 * lane);
  d.lo = *reinterpret_cast<const uint2*>(b + (lane < 16 ? 8 * lane : 256 + 8 * (lane - 16)));
  return d;
}
__device__ __forceinline__ unsigned less128(unsigned p) {  // u - 128 in the low half
  const unsigned c = 0x00000080u;
  const __half2 h = __hsub2(*reinterpret_cast<__half2*>(&p), *reinterpret_cast<const __half2*>(&c));
  return *reinterpret_cast<const unsigned*>(&h);
}
// Products of an entry (of each lane) with its column's digits.
__device__ __forceinline__ void mma_entry(Acc& a, const uint4& w, const Digits& d) {
  {
    const unsigned a0 = less128(__byte_perm(w.y, 0u, 0x4243)), a2 = __byte_perm(w.y, 0u, 0x4041);
    const unsigned a1 = less128(__byte_perm(w.w, 0u, 0x4243)), a3 = __byte_perm(w.w, 0u, 0x4041);
    mma(a.re, a0, a1, a2, a3, d.re);
    mma(a.im, a0, a1, a2, a3, d.im);
  }
  mma(a.lo, __byte_perm(w.x, 0u, 0x4243), __byte_perm(w.z, 0u, 0x4243),
      __byte_perm(w.x, 0u, 0x4041), __byte_perm(w.z, 0u, 0x4041), d.lo);
}
__device__ __forceinline__ int as_int(float v) { return __float2int_rn(v * 16777216.f); }

// Adds the accumulators of an item into its level sums S (shared memory, exact
// integers, so the order of the additions does not matter).  A: re = Ar vr - Ai vi,
// im = Ar vi + Ai vr; A^dag: re = Ar vr + Ai vi, im = Ar vi - Ai vr.
__device__ __forceinline__ void empty(const Acc& a, int* S, bool dag) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int sgn = dag ? 1 : -1;
  int* hi = S + 2 * t * kSLevel + g;
  int* lo = S + (4 + 2 * (t & 1)) * kSLevel + g;
  const bool vim = t >= 2;  // of the digits 4..7: products with the vector's imaginary part
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    atomicAdd(hi + e * kSLevel, as_int(a.re[e]) + sgn * as_int(a.im[2 + e]));
    atomicAdd(hi + e * kSLevel + 8, as_int(a.im[e]) - sgn * as_int(a.re[2 + e]));
    atomicAdd(lo + e * kSLevel + (vim ? 8 : 0), as_int(a.lo[e]));
    atomicAdd(lo + e * kSLevel + (vim ? 0 : 8), (vim ? sgn : -sgn) * as_int(a.lo[2 + e]));
  }
}

// Up to kGroups consecutive items of a site share the vector operands: R items from row group
// rg of local site ls on, the run's item-th.
constexpr int kGroups = 4;
struct Super {
  int ls, rg, R, item;
};
// Stencil and vectors of a run of items.  Its k-steps are counted super by super.
struct Run {
  const uint4* T;            // entries from the lane's offset on
  const int4* quads;         // quad offsets of the run's sites, [site][KS] (shared memory)
  const unsigned char* B;    // vector digits
  int* S;                    // level sums of the items
  const Super* sup;
  int step;                  // group_step
  bool dag;
  unsigned long long pol;
};
using Words = uint4[kGroups][4];  // a lane's entries of one k-step: [item][quad]

__device__ __forceinline__ void fetch_quad(Words& w, const Run& r, int c, int off, const Super& u,
                                           bool go) {
#pragma unroll
  for (int k = 0; k < kGroups; ++k)
    ld_entry(w[k][c], r.T + (off + (u.rg + k) * r.step), go && k < u.R, r.pol);
}
__device__ __forceinline__ void prefetch(const Shape& s, const Run& r, int f, int n, Words& w) {
  if (n <= 0) return;
  const int j = f / s.KS, ks = f - j * s.KS;
  const Super u = r.sup[j];
  const int4 o = r.quads[u.ls * s.KS + ks];
  fetch_quad(w, r, 0, o.x, u, true);
  fetch_quad(w, r, 1, o.y, u, true);
  fetch_quad(w, r, 2, o.z, u, true);
  fetch_quad(w, r, 3, o.w, u, true);
}
// k-steps ks, ks + 1, .. of super j with R items: up to n, not past its last; ks, j and n are
// moved on.  The entries of the next k-step (of whatever super) are asked for as soon as those
// of the present one are used, a whole k-step (up to 8 KB per warp) ahead; vector digits, which
// come from shared memory behind those loads, a quad ahead.
template <int R>
__device__ __forceinline__ void walk(const Shape& s, const Run& r, int& j, int& ks, int& n,
                                     Words& w) {
  const Super u = r.sup[j];
  int* S = r.S + u.item * kSItem;
  const unsigned char* b = r.B + (size_t)(u.ls * s.KS + ks) * (4 * kQuadBytes);
  const int4* q = r.quads + u.ls * s.KS + ks;
  Digits d = ld_digits(b);
  Acc acc[R];
#pragma unroll
  for (int k = 0; k < R; ++k) clear(acc[k]);
  for (int left = kMaxSteps;;) {
    ++ks;
    ++q;
    --n;
    const bool end = ks == s.KS, more = n > 0;
    Super v = u;  // of the next k-step
    if (end && more) {
      v = r.sup[j + 1];
      q = r.quads + v.ls * s.KS;
    }
    const int4 o = more ? *q : make_int4(0, 0, 0, 0);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const Digits next = ld_digits(c < 3 || (more && !end) ? b + kQuadBytes : b);
      b += kQuadBytes;
#pragma unroll
      for (int k = 0; k < R; ++k) mma_entry(acc[k], w[k][c], d);
      fetch_quad(w, r, c, c == 0 ? o.x : c == 1 ? o.y : c == 2 ? o.z : o.w, v, more);
      d = next;
    }
    const bool stop = end || !more;
    if (--left == 0 || stop) {
#pragma unroll
      for (int k = 0; k < R; ++k) {
        empty(acc[k], S + k * kSItem, r.dag);
        clear(acc[k]);
      }
      left = kMaxSteps;
    }
    if (stop) break;
  }
  if (ks == s.KS) {
    ks = 0;
    ++j;
  }
}
// The products of a warp's share: k-steps f .. f + n - 1 of the run; w holds the entries of the
// first (prefetch).
__device__ __forceinline__ void products(const Shape& s, const Run& r, int f, int n, Words& w) {
  int j = f / s.KS, ks = f - j * s.KS;
  while (n > 0) {
    switch (r.sup[j].R) {
      case 1: walk<1>(s, r, j, ks, n, w); break;
      case 2: walk<2>(s, r, j, ks, n, w); break;
      case 3: walk<3>(s, r, j, ks, n, w); break;
      default: walk<4>(s, r, j, ks, n, w); break;
    }
  }
}

// Takes the value of pair q = 2 row + component of an item out of its level
// sums (and clears them): ea is the exponent of the stencil row (A; 1023 for
// A^dag), ev of the site's vectors.
__device__ __forceinline__ double take(int* S, int q, int ea, int ev) {
  S += (q & 1) * 8 + (q >> 1);
  long long H = 0, M = 0;
#pragma unroll
  for (int l = 0; l < 4; ++l) {
    H = H * 256 + S[l * kSLevel];
    M = M * 256 + S[(4 + l) * kSLevel];
    S[l * kSLevel] = 0;
    S[(4 + l) * kSLevel] = 0;
  }
  if (ea >= 2047 || ev >= kNotFinite) return __longlong_as_double(0x7ff8000000000000ll);
  return to_double(H, M, ea + ev - 2 * 1023 - 67);
}

}  // namespace swdig
