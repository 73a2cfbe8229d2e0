// Packing of a coarse stencil into digit entries and the stencil application on
// them (digit.cuh has the number format, the layout and the reasons).
#include <atomic>

#include "digit.cuh"
#include "many.h"

namespace {

using namespace swdig;

// One warp per (site, row): the largest exponent of row i of A.
__global__ void __launch_bounds__(256) k_row_expo(const double2* __restrict__ Y, Shape s,
                                                  int* __restrict__ ex) {
  const long row = (long)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  const int X = (int)(row / s.nP), i = (int)(row - (long)X * s.nP);
  int em = 1;
  if (i < s.nc)
    for (int c = lane; c < 5 * s.nc; c += 32) {
      const double2 v = Y[((long)X * 5 * s.nc + c) * s.nc + i];
      em = max(em, max(expo(v.x), expo(v.y)));
    }
  em = __reduce_max_sync(0xffffffffu, em);
  if (lane == 0) ex[row] = em;
}

__global__ void k_pack_digits(const double2* __restrict__ Y, Shape s, const int* __restrict__ ex,
                              uint4* __restrict__ T, long n) {
  const long e = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  const long xd = e / (s.nP * s.nP);  // X 5 + d
  const int ij = (int)(e - xd * s.nP * s.nP), i = ij % s.nP, j = ij / s.nP;
  double2 v = make_double2(0.0, 0.0);
  if (i < s.nc && j < s.nc) v = Y[(xd * s.nc + j) * s.nc + i];
  const int em = ex[(xd / 5) * s.nP + i];
  const unsigned long long a = (unsigned long long)fixed(v.x, 0, em, 10) + (1ull << 63);
  const unsigned long long b = (unsigned long long)fixed(v.y, 0, em, 10) + (1ull << 63);
  T[xd * s.nP * s.nP + ((j >> 2) * (s.nP >> 2) + (i >> 2)) * 16 + tile_place(i, j)] =
      make_uint4((unsigned)a, (unsigned)(a >> 32), (unsigned)b, (unsigned)(b >> 32));
}

// y_X = sum_d Y[X][d] x_{X+d} (DAG: the adjoint).  A CTA of four warps takes
// (site, part) units: it writes the digits of the five neighbour vectors to
// shared memory, its warps share the unit's k-steps, and each thread finishes
// (row, component) pairs.  The kernel is bound by reading the entries (16 bytes
// each, as many as the FP64 stencil): kCtas CTAs per SM keep some warps reading
// while others are between units, and every warp asks for the first entries of
// its next unit before it finishes the present one.
constexpr int kNT = 128;
constexpr int kCtas = 3;
constexpr int kPer = 5;     // complex vector elements per thread: nc <= 128
constexpr int kSupers = 16 / kGroups;

// One member of a batch per blockIdx.y.
template <bool DAG, int W>
__global__ void __launch_bounds__(kNT, kCtas) k_digit_apply(Shape s, const uint4* __restrict__ T,
                                                            const int* __restrict__ ex,
                                                            const double2* __restrict__ Y,
                                                            Pack<2, W> io, int parts,
                                                            const int* skip,
                                                            unsigned long long* exec) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int em;
  __shared__ Super sup[2][kSupers];  // of this unit and the next
  const double2* in = io.v[0][blockIdx.y];
  double2* out = io.v[1][blockIdx.y];
  unsigned char* B = smem;
  int4* quads = reinterpret_cast<int4*>(smem + (size_t)s.KS * 4 * kQuadBytes);
  int* S = reinterpret_cast<int*>(quads + 2 * s.KS);
  const int warp = threadIdx.x >> 5;
  unsigned long long pol;  // entries are read once
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  const int nunits = s.E0 * s.E1 * parts;
  for (int k = threadIdx.x; k < s.RG * kSItem; k += kNT) S[k] = 0;
  // unit u: row groups ra .. rb of site X; this warp's k-steps f .. f + n - 1
  int X = 0, ra = 0, rb = 0, f = 0, n = 0, slot = 0;
  Run run{T + lane_offset(s, DAG), nullptr, B, S, nullptr, group_step(s, DAG), DAG, pol};
  Words w = {};
  auto enter = [&](int u) {  // collective
    X = u / parts;
    const int p = u - X * parts;
    ra = s.RG * p / parts;
    rb = s.RG * (p + 1) / parts;
    const int nsup = (rb - ra + kGroups - 1) / kGroups;
    run.quads = quads + slot * s.KS;
    run.sup = sup[slot];
    for (int k = threadIdx.x; k < s.KS; k += kNT)
      quads[slot * s.KS + k] = kstep_offsets<DAG>(s, X, k);
    if (threadIdx.x < nsup) {
      const int a = (rb - ra) * threadIdx.x / nsup, b = (rb - ra) * (threadIdx.x + 1) / nsup;
      sup[slot][threadIdx.x] = Super{0, ra + a, b - a, a};
    }
    const int all = nsup * s.KS;
    f = all * warp / (kNT / 32);
    n = all * (warp + 1) / (kNT / 32) - f;
    __syncthreads();
    prefetch(s, run, f, n, w);
  };
  int u = blockIdx.x;
  if (u < nunits) enter(u);  // tables and first entries: constant, asked for before the wait
  after_previous();
  if (skip && skip[4 * blockIdx.y]) return;
  if (exec && blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(exec, 1ull);
  while (u < nunits) {
    if (threadIdx.x == 0) em = -kNotFinite;
    double2 x[kPer];
    int shift[kPer], e = -kNotFinite;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int c = threadIdx.x + k * kNT, d = c / s.nP, j = c - d * s.nP;
      x[k] = make_double2(0.0, 0.0);
      shift[k] = 0;
      if (d < 5 && j < s.nc) {
        const int nb = nbr(X, d, s.E0, s.E1);
        x[k] = in[(long)nb * s.nc + j];
        if (DAG) shift[k] = ex[(long)nb * s.nP + j] - 1023;
        e = max(e, column_expo(x[k], shift[k]));
      }
    }
    e = __reduce_max_sync(0xffffffffu, e);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) atomicMax(&em, e);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int c = threadIdx.x + k * kNT;
      if (c < 16 * s.KS) put_column(x[k], shift[k], em, B, c);
    }
    __syncthreads();
    products(s, run, f, n, w);
    const int Xc = X, rac = ra, rbc = rb, ev = em;
    u += gridDim.x;
    slot ^= 1;
    if (u < nunits)
      enter(u);
    else
      __syncthreads();
    for (int c = threadIdx.x; c < (rbc - rac) * 16; c += kNT) {
      const int i = 8 * rac + (c >> 1), comp = c & 1;
      const int ea = DAG ? 1023 : ex[(long)Xc * s.nP + i];
      double v = take(S + (c >> 4) * kSItem, c & 15, ea, ev);
      if (i >= s.nc) continue;
      if (ev >= kNotFinite || ea >= 2047) {  // not finite: the plain sum says how
        v = 0.0;
        for (int d = 0; d < 5; ++d) {
          const int nb = nbr(Xc, d, s.E0, s.E1);
          for (int j = 0; j < s.nc; ++j) {
            double2 a = DAG ? Y[(((long)nb * 5 + opp(d)) * s.nc + i) * s.nc + j]
                            : Y[(((long)Xc * 5 + d) * s.nc + j) * s.nc + i];
            if (DAG) a.y = -a.y;
            const double2 z = in[(long)nb * s.nc + j];
            v = comp ? fma(a.y, z.x, fma(a.x, z.y, v)) : fma(-a.y, z.y, fma(a.x, z.x, v));
          }
        }
      }
      reinterpret_cast<double*>(out + (long)Xc * s.nc + i)[comp] = v;
    }
    __syncthreads();  // em, B and S are rewritten by the next unit
  }
}

}  // namespace

long digit_entries(const CoarseGeom& g) {
  const Shape s = shape_of(g);
  return (long)s.E0 * s.E1 * 5 * s.nP * s.nP;
}
long digit_rows(const CoarseGeom& g) { return (long)g.E0 * g.E1 * shape_of(g).nP; }

void launch_pack_digits(const CoarseGeom& g, const double2* Y, uint4* T, int* ex, cudaStream_t st) {
  const Shape s = shape_of(g);
  k_row_expo<<<s.E0 * s.E1 * s.RG, 256, 0, st>>>(Y, s, ex);
  SW_LAUNCH_CHECK();
  const long n = digit_entries(g);
  k_pack_digits<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(Y, s, ex, T, n);
  SW_LAUNCH_CHECK();
}

void many_digit(const CoarseGeom& g, const DigitStencil& t, const double2* Y, int dagger,
                const Many<2>& io, int device, cudaStream_t st, const int* ctl,
                unsigned long long* exec) {
  const Shape s = shape_of(g);
  const int sites = s.E0 * s.E1;
  // rows of a site are split over CTAs while there are fewer units than CTA slots
  int parts = 1;
  while (2 * parts <= s.RG && (long)sites * parts * io.n < kCtas * 152) parts *= 2;
  const int units = sites * parts;
  const size_t smem = (size_t)s.KS * (4 * kQuadBytes + 32) + (size_t)s.RG * kSItem * sizeof(int);
  const int slots = (kCtas * 152 + io.n - 1) / io.n;  // per member
  const dim3 grid(units < slots ? units : slots, io.n);
  with_width(io.n, [&](auto w) {
    constexpr int W = decltype(w)::value;
    // the flag is set after the attributes: a thread that sees it may launch
    static std::atomic<bool> wide[64];
    if (!wide[device & 63].load()) {
      constexpr int most = 40 * (4 * kQuadBytes + 32) + 16 * kSItem * (int)sizeof(int);  // nc = 128
      for (auto f : {k_digit_apply<true, W>, k_digit_apply<false, W>})
        SW_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
      wide[device & 63].store(true);
    }
    auto k = dagger ? k_digit_apply<true, W> : k_digit_apply<false, W>;
    launch_early(k, grid, kNT, smem, st, s, t.T, t.ex, Y, Pack<2, W>(io), parts, ctl, exec);
  });
}
void launch_digit_apply(const CoarseGeom& g, const DigitStencil& t, const double2* Y, int dagger,
                        const double2* in, double2* out, int device, cudaStream_t st,
                        const int* skip, unsigned long long* exec) {
  many_digit(g, t, Y, dagger, Many<2>(0, in, out), device, st, skip, exec);
}
