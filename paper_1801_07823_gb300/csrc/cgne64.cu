// Coarsest-level CGNE in FP64 (CG on the normal error, Sec. IV and Table
// kcycle) as one persistent cooperative kernel, its stencil products formed
// by exact digit arithmetic on the tensor cores (digit.cuh).
//
// Iteration (same as cgne.cu): P1 w = A p, x += alpha p, r -= alpha w, |r|^2;
// grid barrier; P2 p = A^dag r + beta p, |p|^2; grid barrier.
//
// Work.  One CTA of 12 warps per SM.  A CTA owns a contiguous run of items (eight
// rows of one site; pairs of them where that leaves enough for every SM), so that
// its entries, rows and vectors are the same ones in every iteration, and what can be worked out once (offsets, shares, row
// exponents) is kept in shared memory.  Per phase eleven warps write the digits of
// the sites' neighbour vectors to shared memory while the last one adds up
// the previous phase's norm parts and forms alpha or beta, which are needed only
// at the update; all warps share the run's k-steps (a share may begin and end
// inside an item: level sums are exact integers, added in shared memory in
// any order); one thread per (row, component) rounds the product, updates its
// vector and keeps its part of the norm.  Between a CTA's arrival at a grid
// barrier and its wait it updates x, which nobody else reads, and asks for the
// first entries of its next phase.
//
// A run longer than shared memory holds is walked in chunks of whole sites.
//
// Measured, microseconds per iteration, against the FP64-pipe kernel this one
// took the place of: 28.4 against 73.3 at 16^2 sites x 64 dof, 16.2 against 28.7
// at 8^2 x 64, 9.9 against 16.6 at 4^2 x 24.  At 16^2 x 64 the 84 MB of entries
// stay in the L2 (ncu: 97 % hits), and a phase spends 6 us in the products (a
// k-step of eight rows takes about 190 clocks of its sub-partition, of which the
// twelve MMAs need 104), 1 us each in reading and splitting the vectors, in the
// update, and in the norm with its fence, and 1 us in the barrier; at 4^2 x 24
// that fixed part is all.
//
// Where it is all, the cluster form is faster: up to 16 CTAs of one cluster, the
// cluster's hardware barrier instead of arrivals counted in the L2, norm parts in
// every CTA's shared memory.  With more than six items per CTA (kClusterItems) the
// products on a tenth of the SMs take longer than that saves.  It needs 16 SMs in one
// GPC, so a context that shares the SMs with others keeps the grid form.
// Solve at 64^2 with Nv 8/12 (4^2 x 24): 35.2 -> 32.3 ms.
//
// The fraction l2frac of the entries' lines, sized on the host to what the L2
// can keep, is loaded with evict-last priority and the rest evict-first.
//
// Grid barriers use one monotone arrival counter; waits are bounded
// (SW_ERR_TIMEOUT on the host), and a CTA that gives up leaves at its next
// barrier.  Norm parts are added per CTA and over CTAs in a fixed order, so
// every CTA takes the same decision and every run gives the same bits.
#include <algorithm>
#include <atomic>

#include "sums.cuh"

namespace {

using namespace swdig;
using namespace swsum;

constexpr int kThreads = 384;
constexpr int kWarps = kThreads / 32;
constexpr int kPut = kThreads - 32;  // threads that write vector digits
constexpr int kMaxCols = 1792;       // padded vector columns per chunk
constexpr int kMaxPairs = 1024;      // (row, component) pairs per chunk
constexpr int kMaxSites = 56;        // sites per chunk
constexpr int kMaxSupers = 128;      // supers per chunk
constexpr int kMaxBytes = 176 * 1024;  // shared memory of a chunk
constexpr int kCluster = 16;         // CTAs of the cluster form, at most
constexpr int kClusterItems = 6 * kCluster;  // its largest problem

struct Args {
  Shape s;
  DigitStencil t;
  const double2* b;
  double2 *x, *r, *p;
  double* partials;  // [2][gridDim.x]
  unsigned* bar;     // [0] monotone arrival counter, two arrivals per CTA and barrier
  int* status;       // [0] iterations, [1] barrier timeout, [2] non-finite residual
  int maxit;
  double tol;
  int stall_test;    // 1: CTA 0 never arrives at the first barrier
  float l2frac;      // fraction of the entries' lines loaded with L2 evict-last priority
  int cs;            // sites per chunk
  int unit;          // items that stay together
};

enum { kInit = 0, kP1 = 1, kP2 = 2 };

struct Shared {
  Aligned sum[kWarps];
  double own[kMaxPairs];         // r or p before its update
  int elem[kMaxPairs];           // 2 * element + component of a pair, -1: padding
  int src[kMaxCols];             // element of a vector column, -1: padding
  short row_ex[kMaxPairs];       // exponent of a pair's row of A
  short shift[kMaxCols];         // row scale of a column's element (A^dag)
  unsigned char site[kMaxPairs], col_site[kMaxCols];
  Super sup[kMaxSupers];
  int f0[kWarps], n[kWarps];     // the warps' shares of the k-steps
  int em[2][kMaxSites];
  double rr, stop2, coef;
  double parts[2][kCluster];     // norm parts of the cluster form
  int nsup, state;  // state 0: continue, 1: converged / cap, 2: non-finite
  int ok;
};

// A chunk of this CTA's items; dynamic shared memory of a chunk.
struct Chunk {
  int a, b, s0, ns, ncomp;
};
struct Place {
  int i0, i1;
  bool single;       // one chunk: its tables are made once
  unsigned char* B;  // vector digits
  double2* cols;     // vector columns
  int4* quads;       // [2][cs][KS] quad offsets of A and of A^dag
  int* S;            // level sums
  unsigned long long pol;
};

// Tables of the chunk that begins at item a (collective, synchronises).
__device__ Chunk enter_chunk(const Args& A, Shared& sh, const Place& pl, int a) {
  const Shape& s = A.s;
  Chunk c;
  c.a = a;
  c.s0 = a / s.RG;
  c.b = min(pl.i1, (c.s0 + A.cs) * s.RG);
  c.ns = (c.b - 1) / s.RG - c.s0 + 1;
  c.ncomp = (c.b - c.a) * 16;
  __syncthreads();
  for (int q = threadIdx.x; q < c.ncomp; q += kThreads) {
    const int it = c.a + (q >> 4), X = it / s.RG, i = (it - X * s.RG) * 8 + ((q >> 1) & 7);
    sh.elem[q] = i < s.nc ? 2 * (X * s.nc + i) + (q & 1) : -1;
    sh.row_ex[q] = (short)A.t.ex[(long)X * s.nP + i];
    sh.site[q] = (unsigned char)(X - c.s0);
  }
  const int per = 16 * s.KS;
  for (int e = threadIdx.x; e < c.ns * per; e += kThreads) {
    const int ls = e / per, k = e - ls * per, d = k / s.nP, j = k - d * s.nP;
    sh.src[e] = -1;
    sh.col_site[e] = (unsigned char)ls;
    pl.cols[e] = make_double2(0.0, 0.0);
    if (d < 5 && j < s.nc) {
      const int nb = nbr(c.s0 + ls, d, s.E0, s.E1);
      sh.src[e] = nb * s.nc + j;
      sh.shift[e] = (short)(A.t.ex[(long)nb * s.nP + j] - 1023);
    }
  }
  for (int e = threadIdx.x; e < c.ns * s.KS; e += kThreads) {
    const int ls = e / s.KS, ks = e - ls * s.KS;
    pl.quads[e] = kstep_offsets<false>(s, c.s0 + ls, ks);
    pl.quads[A.cs * s.KS + e] = kstep_offsets<true>(s, c.s0 + ls, ks);
  }
  if (threadIdx.x == 0) {  // supers: each site's items of the chunk, split evenly
    int n = 0;
    for (int it = c.a; it < c.b;) {
      const int X = it / s.RG, rg = it - X * s.RG, m = min(c.b - it, s.RG - rg);
      const int parts = (m + kGroups - 1) / kGroups;
      for (int p = 0; p < parts; ++p) {
        const int g0 = m * p / parts, g1 = m * (p + 1) / parts;
        sh.sup[n++] = Super{X - c.s0, rg + g0, g1 - g0, it - c.a + g0};
      }
      it += m;
    }
    sh.nsup = n;
  }
  __syncthreads();
  if (threadIdx.x < kWarps) {
    // shares of equal work, a k-step of R items counting as 2 R + 1; the last warp, which
    // has the scalars to do, gets half a share less
    const int w = threadIdx.x;
    int total = 0;
    for (int j = 0; j < sh.nsup; ++j) total += (2 * sh.sup[j].R + 1) * s.KS;
    auto begin = [&](int w) {  // k-step at which warp w's share begins
      const int want = min(total, (int)((long)total * 2 * w / (2 * kWarps - 1)));
      int f = 0, sum = 0;
      for (int j = 0; j < sh.nsup; ++j) {
        const int one = 2 * sh.sup[j].R + 1, all = one * s.KS;
        if (sum + all > want) return f + (want - sum + one / 2) / one;
        sum += all;
        f += s.KS;
      }
      return f;
    };
    const int f0 = begin(w);
    sh.f0[w] = f0;
    sh.n[w] = (w + 1 < kWarps ? begin(w + 1) : sh.nsup * s.KS) - f0;
  }
  __syncthreads();
  return c;
}

// Component q & 1 of complex element q >> 1.
__device__ __forceinline__ double ld_comp(const double2* v, int q) {
  return __ldcg(reinterpret_cast<const double*>(v) + q);
}
__device__ __forceinline__ void st_comp(double2* v, int q, double x) {
  reinterpret_cast<double*>(v)[q] = x;
}
// Named barriers (0 is __syncthreads).
__device__ __forceinline__ void bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Sum of the previous phase's partials (in global memory, or in shared memory in the cluster
// form), in the same order in every CTA, and the scalar the phase needs (one warp).
template <bool CLUSTER>
__device__ void scalars(const Args& A, Shared& sh, int mode, const double* partials, int k) {
  const int lane = threadIdx.x & 31, G = gridDim.x;
  double s;
  if (CLUSTER) {
    const Aligned a = warp_sum(lane < G ? partials[lane] : 0.0);
    s = total<1>(&a);
  } else {
    s = grid_total(partials, G);
  }
  if (lane != 0) return;
  if (mode == kInit) {  // s = |b|^2
    sh.rr = s;
    sh.stop2 = A.tol * fabs(A.tol) * s;  // below 0: no residual meets it
    sh.state = !isfinite(s) ? 2 : ((A.maxit <= 0 || !(s > sh.stop2)) ? 1 : 0);
    sh.coef = 0.0;
    return;
  }
  if (mode == kP2) sh.state = !isfinite(s) ? 2 : ((k < A.maxit && s > sh.stop2) ? 0 : 1);
  const double rr = sh.rr;
  sh.coef = mode == kP1 ? rr / s : s / rr;  // s = |p|^2: alpha; s = |r|^2 after k iterations: beta
  if (mode == kP2) sh.rr = s;
}

// Digits of the chunk's neighbour vectors (the first kPut threads).
__device__ void put_vectors(const Chunk& c, int cols, Shared& sh, bool dag, const double2* v,
                            int* em, const Place& pl) {
#pragma unroll 1
  for (int e = threadIdx.x; e < cols; e += kPut) {
    const int q = sh.src[e];
    if (q >= 0)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                       (unsigned)__cvta_generic_to_shared(pl.cols + e)),
                   "l"(v + q)
                   : "memory");
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll 1
  for (int e = threadIdx.x; (e & ~31) < cols; e += kPut) {  // warp-uniform
    const bool in = e < cols;
    const int ls = in ? sh.col_site[e] : -1;
    const int ex = in && sh.src[e] >= 0 ? column_expo(pl.cols[e], dag ? sh.shift[e] : 0)
                                        : -kNotFinite;
    if (__all_sync(0xffffffffu, ls == __shfl_sync(0xffffffffu, ls, 0))) {
      const int m = __reduce_max_sync(0xffffffffu, ex);
      if ((threadIdx.x & 31) == 0) atomicMax(em + ls, m);
    } else if (in) {
      atomicMax(em + ls, ex);
    }
  }
  bar_sync(1, kPut);
#pragma unroll 1
  for (int e = threadIdx.x; e < cols; e += kPut)
    put_column(pl.cols[e], dag && sh.src[e] >= 0 ? sh.shift[e] : 0, em[sh.col_site[e]], pl.B, e);
}

// The run of a chunk in the given orientation.
__device__ __forceinline__ Run run_of(const Args& A, const Shared& sh, const Place& pl, bool dag) {
  return Run{A.t.T + lane_offset(A.s, dag), pl.quads + (dag ? A.cs * A.s.KS : 0),
             pl.B, pl.S, sh.sup, group_step(A.s, dag), dag, pl.pol};
}

// One stencil application over this CTA's items with the update of r (kP1) or
// p (kP2; kInit: p = A^dag r) and this thread's share of the new squared norm;
// w holds the first entries if there is one chunk.  em[par] is clear at the
// start of a chunk, which clears the other half for the next.  False: the solve
// has stopped.
template <bool CLUSTER>
__device__ bool phase(const Args& A, const Place& pl, Chunk& c, Shared& sh, int mode,
                      const double* partials, int k, int& par, Words& w, double& acc) {
  const bool dag = mode != kP1;
  const Shape& s = A.s;
  const double2* v = dag ? A.r : A.p;
  double2* y = dag ? A.p : A.r;
  const int warp = threadIdx.x >> 5;
  const Run run = run_of(A, sh, pl, dag);
  acc = 0.0;
  bool first = true;
  for (int a = pl.i0; a < pl.i1; a = c.b, first = false, par ^= 1) {
    if (!pl.single) {
      c = enter_chunk(A, sh, pl, a);
      prefetch(s, run, sh.f0[warp], sh.n[warp], w);
    }
    if (threadIdx.x < kPut) {
#pragma unroll 1
      for (int q = threadIdx.x; q < c.ncomp; q += kPut)
        if (sh.elem[q] >= 0 && mode != kInit)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(
                           (unsigned)__cvta_generic_to_shared(sh.own + q)),
                       "l"(reinterpret_cast<const double*>(y) + sh.elem[q])
                       : "memory");
        else
          sh.own[q] = 0.0;
      put_vectors(c, c.ns * 16 * s.KS, sh, dag, v, sh.em[par], pl);
      bar_arrive(2, kThreads);
      bar_sync(3, kPut);
    } else {
      if (first) scalars<CLUSTER>(A, sh, mode, partials, k);
      __syncwarp();
      bar_sync(2, kThreads);
    }
    if (threadIdx.x < kMaxSites) sh.em[par ^ 1][threadIdx.x] = -kNotFinite;
    products(s, run, sh.f0[warp], sh.n[warp], w);
    __syncthreads();
    if (dag && sh.state) return false;
    const double coef = dag ? sh.coef : -sh.coef;
#pragma unroll 1
    for (int q = threadIdx.x; q < c.ncomp; q += kThreads) {
      const double t = take(pl.S + (q >> 4) * kSItem, q & 15, dag ? 1023 : sh.row_ex[q],
                            sh.em[par][sh.site[q]]);
      const int e = sh.elem[q];
      if (e < 0) continue;
      // r - alpha A p, or A^dag r + beta p
      const double nw = dag ? fma(coef, sh.own[q], t) : fma(coef, t, sh.own[q]);
      st_comp(y, e, nw);
      acc = fma(nw, nw, acc);
    }
  }
  return true;
}

// The CTA's norm part and arrival at grid barrier `gen`, then `work` while the
// others arrive, then the wait.  A CTA arrives twice: once when its vectors
// are visible and once, after the sum that meanwhile is formed, when its norm
// part is.  False if a wait gave up here or elsewhere.
template <typename F>
__device__ bool grid_barrier(const Args& A, Shared& sh, double acc, double* partials,
                             unsigned gen, bool withhold, F&& work) {
  const Aligned a = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) sh.sum[threadIdx.x >> 5] = a;
  __syncthreads();
  if (withhold) return false;  // the others' wait must run out
  if (threadIdx.x == kPut) {
    __threadfence();
    atomicAdd(A.bar, 1u);
  }
  if (threadIdx.x == 0) {
    partials[blockIdx.x] = total<kWarps>(sh.sum);
    __threadfence();
    atomicAdd(A.bar, 1u);
  }
  work();
  if (threadIdx.x == 0) {
    const unsigned target = 2 * gen * gridDim.x;
    unsigned v;
    long spins = 0;
    for (;;) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(A.bar) : "memory");
      if (v >= target) break;
      if (++spins > kSpinLimit) {
        atomicExch(A.status + 1, 1);
        break;
      }
    }
    __threadfence();
    sh.ok = *((volatile int*)(A.status + 1)) == 0;
  }
  __syncthreads();
  return sh.ok;
}

// The same between the CTAs of a cluster: parts go to every CTA's shared memory, and the
// hardware's cluster barrier orders them and the vectors.  All CTAs form the same sums and
// so leave together; nothing here waits for a CTA that might not come.
template <typename F>
__device__ void cluster_barrier(Shared& sh, double acc, int ph, F&& work) {
  const Aligned a = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) sh.sum[threadIdx.x >> 5] = a;
  __syncthreads();
  if (threadIdx.x < gridDim.x) {
    const double v = total<kWarps>(sh.sum);
    unsigned there;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(there)
                 : "r"((unsigned)__cvta_generic_to_shared(&sh.parts[ph][blockIdx.x])),
                   "r"(threadIdx.x));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(there), "d"(v) : "memory");
  }
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  work();
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// CLUSTER: the grid is one cluster.
template <bool CLUSTER>
__global__ void __launch_bounds__(kThreads, 1) k_cgne64(Args A) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ Shared sh;
  const Shape& s = A.s;
  const int G = gridDim.x;
  const long items = (long)s.E0 * s.E1 * s.RG;
  Place pl;
  pl.B = smem;
  pl.cols = reinterpret_cast<double2*>(pl.B + (size_t)A.cs * s.KS * 4 * kQuadBytes);
  pl.quads = reinterpret_cast<int4*>(pl.cols + A.cs * s.KS * 16);
  pl.S = reinterpret_cast<int*>(pl.quads + 2 * A.cs * s.KS);
  pl.i0 = (int)(items / A.unit * blockIdx.x / G) * A.unit;
  pl.i1 = (int)(items / A.unit * (blockIdx.x + 1) / G) * A.unit;
  asm volatile("createpolicy.fractional.L2::evict_last.L2::evict_first.b64 %0, %1;"
               : "=l"(pl.pol)
               : "f"(A.l2frac));
  if (CLUSTER) {  // every CTA has begun before another writes to its shared memory
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
  for (int q = threadIdx.x; q < A.cs * s.RG * kSItem; q += kThreads) pl.S[q] = 0;
  if (threadIdx.x < kMaxSites) sh.em[0][threadIdx.x] = sh.em[1][threadIdx.x] = -kNotFinite;
  Chunk c = enter_chunk(A, sh, pl, pl.i0);
  pl.single = c.b == pl.i1;
  const int nall = (pl.i1 - pl.i0) * 16;  // (row, component) pairs of this CTA
  auto pair = [&](int q) {                // component index of this CTA's pair q, -1: padding
    if (pl.single) return sh.elem[q];
    const int it = pl.i0 + (q >> 4), X = it / s.RG, i = (it - X * s.RG) * 8 + ((q >> 1) & 7);
    return i < s.nc ? 2 * (X * s.nc + i) + (q & 1) : -1;
  };
  // x = 0, r = b, ||r||^2
  double acc = 0.0;
  for (int q = threadIdx.x; q < nall; q += kThreads) {
    const int e = pair(q);
    if (e < 0) continue;
    const double v = reinterpret_cast<const double*>(A.b)[e];
    st_comp(A.x, e, 0.0);
    st_comp(A.r, e, v);
    acc = fma(v, v, acc);
  }
  Words w = {};
  const int warp = threadIdx.x >> 5;
  int ph = 0, k = 0, par = 0, mode = kInit;
  for (unsigned gen = 1;; ++gen) {
    // after the update of r (and at the start): x += alpha p
    const double alpha = mode == kP2 ? sh.coef : 0.0;
    const auto work = [&] {
      if (pl.single) prefetch(s, run_of(A, sh, pl, mode != kP1), sh.f0[warp], sh.n[warp], w);
      if (mode == kP2) {
#pragma unroll 1
        for (int q = threadIdx.x; q < nall; q += kThreads) {
          const int e = pair(q);
          if (e >= 0) st_comp(A.x, e, fma(alpha, ld_comp(A.p, e), ld_comp(A.x, e)));
        }
      }
    };
    if (CLUSTER)
      cluster_barrier(sh, acc, ph, work);
    else if (!grid_barrier(A, sh, acc, A.partials + ph * G, gen, A.stall_test && blockIdx.x == 0, work))
      return;
    if (!phase<CLUSTER>(A, pl, c, sh, mode, CLUSTER ? sh.parts[ph] : A.partials + ph * G, k, par, w,
                        acc))
      break;
    ph ^= 1;
    if (mode == kP1) ++k;
    mode = mode == kP1 ? kP2 : kP1;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    A.status[0] = k;
    if (sh.state == 2) A.status[2] = 1;
  }
}

}  // namespace

// Fraction of `bytes` that the L2 can keep resident across a sweep (three
// quarters of its capacity, the rest left to vectors and other traffic).
static float l2_fraction(long bytes, int device) {
  int l2 = 0;
  SW_CUDA(cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, device));
  const double f = 0.75 * (double)l2 / (double)(bytes > 0 ? bytes : 1);
  return (float)(f < 1.0 ? f : 1.0);
}

bool launch_cgne64(const CoarseGeom& g, const DigitStencil& t, const double2* b, double2* x,
                   double2* r, double2* p, double* partials, unsigned* bar, int* status, int maxit,
                   double tol, int device, cudaStream_t st, int stall_test, int sms_use) {
  static std::atomic<int> cached_sms[64];
  const Shape s = shape_of(g);
  const int site = s.KS * (4 * kQuadBytes + 16 * 16 + 32) + s.RG * kSItem * (int)sizeof(int);
  int cs = std::min(kMaxBytes / site, std::min(kMaxSites, kMaxCols / (16 * s.KS)));
  cs = std::min(cs, std::min(kMaxPairs / (16 * s.RG), kMaxSupers / ((s.RG + kGroups - 1) / kGroups) - 2));
  const int smem = cs * site;
  int sms = cached_sms[device & 63].load();
  if (sms == 0) {
    int occ = 0, coop = 0, n = 0, most = 0;
    SW_CUDA(cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, device));
    cudaFuncAttributes fa;
    SW_CUDA(cudaFuncGetAttributes(&fa, k_cgne64<false>));
    most -= (int)fa.sharedSizeBytes;
    for (auto f : {k_cgne64<false>, k_cgne64<true>})
      SW_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    SW_CUDA(cudaFuncSetAttribute(k_cgne64<true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    SW_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_cgne64<false>, kThreads, most));
    SW_CUDA(cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, device));
    SW_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, device));
    if (!coop || occ < 1 || n > kReduceBlocks) return false;
    sms = n;
    cached_sms[device & 63].store(sms);
  }
  SW_CUDA(cudaMemsetAsync(bar, 0, 2 * sizeof(unsigned), st));
  SW_CUDA(cudaMemsetAsync(status, 0, 3 * sizeof(int), st));
  // one CTA per SM it may use, at most one per item (partials hold 2 x kReduceBlocks)
  const int unit = s.RG % 2 == 0 && s.E0 * s.E1 * s.RG >= 4 * sms ? 2 : 1;
  const int items = s.E0 * s.E1 * s.RG / unit;
  int grid = sms_use < sms ? (sms_use > 0 ? sms_use : 1) : sms;
  grid = grid < items ? grid : items;
  Args a{s, t, b, x, r, p, partials, bar, status, maxit, tol, stall_test,
         l2_fraction(16 * digit_entries(g), device), cs, unit};
  const int all = s.E0 * s.E1 * s.RG;
  if (all <= kClusterItems && sms_use >= sms && !stall_test) {
    int n = 1;
    while (2 * n <= std::min(all, kCluster)) n *= 2;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = n;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int fits = 0;
    if (cudaOccupancyMaxActiveClusters(&fits, k_cgne64<true>, &cfg) == cudaSuccess && fits > 0) {
      a.unit = 1;
      SW_CUDA(cudaLaunchKernelEx(&cfg, k_cgne64<true>, a));
      sw_count_launch();
      return true;
    }
    cudaGetLastError();
  }
  void* params[] = {&a};
  SW_CUDA(cudaLaunchCooperativeKernel((const void*)k_cgne64<false>, dim3(grid), dim3(kThreads),
                                      params, smem, st));
  sw_count_launch();
  return true;
}
