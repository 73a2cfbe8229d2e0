// CG on the even/odd (checkerboard) normal system of the staggered operator,
// the paper's comparison solver (Sec. II, Eq. normal; Sec. IV, Fig. iterworst):
//   [m D_eo; D_oe m] [x_e; x_o] = [b_e; b_o]  ->
//   (m^2 - D_eo D_oe) x_e = m b_e - D_eo b_o,  x_o = (b_o - D_oe x_e) / m,
// with even/odd the site parity eps(x) = (-1)^(x0 + x1).  m^2 - D_eo D_oe is
// Hermitian positive definite (D_oe = -D_eo^dag).  The full residual is
// b - D x = ((m b_e - D_eo b_o) - (m^2 - D_eo D_oe) x_e) / m on even sites
// and 0 on odd ones, so CG stops when its residual is below m tol ||b||.
//
// Layout: half-lattice vectors, site (x0, x1) of parity p at (x1 L0 + x0) / 2.
//
// The iteration is one persistent cooperative kernel (k_cg_eo).  As eight
// launches per iteration it took 55 us at 256^2, most of it launch gaps; now 14.8
// us, and 13 on any smaller lattice: three barriers (1.2 us each), two sums over
// the grid with an FP64 division each (1.5 us), three round trips to the L2 and
// chains of dependent FP64 operations at 64 clocks each.  A CTA owns a contiguous run
// of the half lattice; per iteration three grid barriers order
//   A  t_o = D_oe p with p = r + beta p_old formed where it is read (two FMAs per
//      neighbour instead of one more barrier), and p written in the other buffer
//   B  q = m^2 p - D_eo t, <p, q>          -> alpha
//   C  x += alpha p, r -= alpha q, |r|^2   -> beta, stopping test
// Every CTA forms the two scalars from all CTAs' parts in the same order.
//
// A solve shares the device: it gives its SMs back when other calls are in flight (run_cg_eo).
// Beside a CG on 256^2 a 64^2 solve takes 31 ms (alone 25.4), 34 on the CG's own stream; while
// one launch held the SMs to the end, the solve waited for that end.  A context with too small
// a share of the SMs for its lattice queues a launch per operation on all of them instead
// (cg_queued).
#include <chrono>
#include <cmath>
#include <cstring>

#include <algorithm>
#include <atomic>

#include "lease.h"
#include "many.h"
#include "sums.cuh"

namespace {

__device__ __forceinline__ void cfma(double2& acc, double2 a, double2 b) {
  acc.x = fma(a.x, b.x, acc.x);
  acc.x = fma(-a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y);
  acc.y = fma(a.y, b.x, acc.y);
}

// out_p(s) = a src_p(s) + c * sum_mu [W_mu(s) in(s+mu) - conj(W_mu(s-mu)) in(s-mu)]
// for the sites s of parity p; in is the opposite-parity half.  One thread per
// site, 2D grid over (x0 / 2, x1) so each row's threads read consecutive
// addresses.
__global__ void k_hop_eo(const double2* __restrict__ W, int par, double a, const double2* src,
                         double c, const double2* __restrict__ in, double2* __restrict__ out,
                         int L0, int L1) {
  int hx = blockIdx.x * blockDim.x + threadIdx.x;
  int x1 = blockIdx.y;
  if (hx >= L0 / 2) return;
  int x0 = 2 * hx + ((x1 + par) & 1);
  long N = (long)L0 * L1;
  long s = (long)x1 * L0 + x0;
  int xp0 = x0 + 1 == L0 ? 0 : x0 + 1, xm0 = x0 == 0 ? L0 - 1 : x0 - 1;
  int xp1 = x1 + 1 == L1 ? 0 : x1 + 1, xm1 = x1 == 0 ? L1 - 1 : x1 - 1;
  long sp0 = (long)x1 * L0 + xp0, sm0 = (long)x1 * L0 + xm0;
  long sp1 = (long)xp1 * L0 + x0, sm1 = (long)xm1 * L0 + x0;
  double2 h = make_double2(0.0, 0.0);
  cfma(h, W[s], in[sp0 >> 1]);
  cfma(h, W[N + s], in[sp1 >> 1]);
  double2 w = W[sm0], v = in[sm0 >> 1];
  h.x -= w.x * v.x + w.y * v.y;
  h.y -= w.x * v.y - w.y * v.x;
  w = W[N + sm1];
  v = in[sm1 >> 1];
  h.x -= w.x * v.x + w.y * v.y;
  h.y -= w.x * v.y - w.y * v.x;
  double2 o = src ? src[s >> 1] : make_double2(0.0, 0.0);
  o.x = fma(c, h.x, a * o.x);
  o.y = fma(c, h.y, a * o.y);
  out[s >> 1] = o;
}

// lexicographic <-> checkerboard halves
__global__ void k_split_eo(const double2* __restrict__ lex, double2* __restrict__ e,
                           double2* __restrict__ o, int L0, int L1) {
  long s = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= (long)L0 * L1) return;
  int x0 = (int)(s % L0), x1 = (int)(s / L0);
  (((x0 + x1) & 1) ? o : e)[s >> 1] = lex[s];
}
__global__ void k_join_eo(const double2* __restrict__ e, const double2* __restrict__ o,
                          double2* __restrict__ lex, int L0, int L1) {
  long s = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= (long)L0 * L1) return;
  int x0 = (int)(s % L0), x1 = (int)(s / L0);
  lex[s] = (((x0 + x1) & 1) ? o : e)[s >> 1];
}

void hop_eo(const sw_gauge* g, int par, double a, const double2* src, double c, const double2* in,
            double2* out, cudaStream_t s) {
  dim3 grid((g->L0 / 2 + 127) / 128, g->L1);
  k_hop_eo<<<grid, 128, 0, s>>>(g->W_lex, par, a, src, c, in, out, g->L0, g->L1);
  SW_LAUNCH_CHECK();
}

// ---------------------------------------------------------------- the iteration
constexpr int kCgThreads = 512;
constexpr int kCgWarps = kCgThreads / 32;
constexpr int kCgSlots = 256;  // above the multigrid levels' 4 x 64
constexpr int kCgKeep = 4;  // iterations of a launch before it yields its SMs
// Whether a launch per operation on all SMs beats the persistent kernel on `sms` of them.
// Measured, us per iteration: queued 24 + half / 8300 (64^2 24.5, 512^2 42.3, 1024^2 87,
// 2048 x 1024 151); persistent about 10 + half / (73 sms) (256^2 on 152 / 38 / 19 / 2 SMs: 14.8 /
// 24.4 / 37 / 225; 1024^2 on 152 / 76 / 50: 58 / 104 / 150).
bool cg_queued(long half, int sms) { return half * (114 - sms) > 117000L * sms; }
// Iterations of a launch, 3 to 6 ms: work that other contexts queue on the stream gets its turn.
// A launch costs about 20 us.
int cg_slice(long half) { return (int)std::min(256L, std::max(32L, (1L << 25) / half)); }

struct CgArgs {
  const double2* W;
  double2 *x, *r, *q, *t;
  double2* p[2];
  double* partials;  // [2][gridDim.x]
  unsigned* bar;     // monotone arrival counter
  int* status;       // [0] iterations (their complement: not finished), [1] barrier timeout,
                     // [2] non-finite residual, [3] to yield
  const int* yield;  // host word: other calls are in flight
  double2* state;    // |r|^2 and beta of a solve that is to go on (k0 > 0)
  int L0, L1, k0, slice, maxit;  // iterations before this launch, of it at most, in all
  double m2, rr, stop;
};
struct CgShared {
  swsum::Aligned sum[kCgWarps];
  double total;
  int ok, yield;
};

// Neighbours of site h of the half of parity par: half-lattice indices of the
// other parity (forward 0, 1, backward 0, 1), and the lexicographic sites of the
// links between.
struct CgSite {
  long s, sm0, sm1;
  int n[4];
};
__device__ __forceinline__ CgSite cg_site(int h, int par, int L0, int L1) {
  const int half = L0 >> 1;
  const int x1 = h / half, x0 = 2 * (h - x1 * half) + ((x1 + par) & 1);
  const long row = (long)x1 * L0;
  CgSite c;
  c.s = row + x0;
  const long sp0 = row + (x0 + 1 == L0 ? 0 : x0 + 1);
  const long sp1 = (x1 + 1 == L1 ? 0 : row + L0) + x0;
  c.sm0 = row + (x0 == 0 ? L0 - 1 : x0 - 1);
  c.sm1 = (x1 == 0 ? (long)(L1 - 1) * L0 : row - L0) + x0;
  c.n[0] = (int)(sp0 >> 1);
  c.n[1] = (int)(sp1 >> 1);
  c.n[2] = (int)(c.sm0 >> 1);
  c.n[3] = (int)(c.sm1 >> 1);
  return c;
}
// sum_mu [W_mu(s) v(s+mu) - conj(W_mu(s-mu)) v(s-mu)]
__device__ __forceinline__ double2 cg_hop(const double2* __restrict__ W, long N, const CgSite& c,
                                          const double2 (&v)[4]) {
  double2 h = make_double2(0.0, 0.0);
  cfma(h, __ldg(W + c.s), v[0]);
  cfma(h, __ldg(W + N + c.s), v[1]);
  auto back = [&](double2 w, double2 u) {
    h.x = fma(-w.x, u.x, h.x);
    h.x = fma(-w.y, u.y, h.x);
    h.y = fma(-w.x, u.y, h.y);
    h.y = fma(w.y, u.x, h.y);
  };
  back(__ldg(W + c.sm0), v[2]);
  back(__ldg(W + N + c.sm1), v[3]);
  return h;
}

// Grid barrier; with parts: also the sum over the grid of every thread's v (in sh.total).
// False if a wait gave up here or elsewhere.
__device__ bool cg_barrier(const CgArgs& a, CgShared& sh, unsigned gen, double v, double* parts) {
  if (parts) {
    const swsum::Aligned w = swsum::warp_sum(v);
    if ((threadIdx.x & 31) == 0) sh.sum[threadIdx.x >> 5] = w;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (parts) parts[blockIdx.x] = swsum::total<kCgWarps>(sh.sum);
    __threadfence();
    atomicAdd(a.bar, 1u);
    const unsigned target = gen * gridDim.x;
    unsigned n;
    long spins = 0;
    for (;;) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(n) : "l"(a.bar) : "memory");
      if (n >= target) break;
      if (++spins > kSpinLimit) {
        atomicExch(a.status + 1, 1);
        break;
      }
    }
    __threadfence();
    sh.ok = *((volatile int*)(a.status + 1)) == 0;
    sh.yield = *((volatile int*)(a.status + 3));
  }
  if (parts) {
    __syncthreads();
    if (threadIdx.x < 32) {
      const double s = swsum::grid_total(parts, gridDim.x);
      if (threadIdx.x == 0) sh.total = s;
    }
  }
  __syncthreads();
  return sh.ok;
}

// Two CTAs' registers per SM although one runs: beside a CTA that takes most of them (104 per
// thread without the bound, 62 with it, at the same speed) the Dslash and the coarse stencils of
// other contexts had no room and waited for the end of the kernel.
__global__ void __launch_bounds__(kCgThreads, 2) k_cg_eo(CgArgs a) {
  __shared__ CgShared sh;
  __shared__ double coef;
  const long N = (long)a.L0 * a.L1, half = N / 2;
  const int h0 = (int)(half * blockIdx.x / gridDim.x), h1 = (int)(half * (blockIdx.x + 1) / gridDim.x);
  double rr = a.k0 > 0 ? a.state->x : a.rr, beta = a.k0 > 0 ? a.state->y : 0.0;
  unsigned gen = 0;
  int k = a.k0;
  const bool watch = blockIdx.x == 0 && threadIdx.x == 32;
  for (;;) {
    // one thread looks at the host word, while phase A runs, and tells all CTAs before the
    // iteration's last barrier
    const int want = watch ? *(const volatile int*)a.yield : 0;
    const double2* po = a.p[k & 1];
    double2* pn = a.p[(k + 1) & 1];
    for (int h = h0 + threadIdx.x; h < h1; h += kCgThreads) {
      const CgSite c = cg_site(h, 1, a.L0, a.L1);
      double2 v[4], w[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = __ldcg(a.r + c.n[j]);
      double2 own = __ldcg(a.r + h);
      if (k > 0) {
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = __ldcg(po + c.n[j]);
        const double2 o = __ldcg(po + h);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          v[j].x = fma(beta, w[j].x, v[j].x);
          v[j].y = fma(beta, w[j].y, v[j].y);
        }
        own.x = fma(beta, o.x, own.x);
        own.y = fma(beta, o.y, own.y);
      }
      pn[h] = own;
      a.t[h] = cg_hop(a.W, N, c, v);
    }
    if (!cg_barrier(a, sh, ++gen, 0.0, nullptr)) return;
    double acc = 0.0;
    for (int h = h0 + threadIdx.x; h < h1; h += kCgThreads) {
      const CgSite c = cg_site(h, 0, a.L0, a.L1);
      double2 v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = __ldcg(a.t + c.n[j]);
      const double2 p = __ldcg(pn + h), d = cg_hop(a.W, N, c, v);
      const double2 q = make_double2(fma(a.m2, p.x, -d.x), fma(a.m2, p.y, -d.y));
      a.q[h] = q;
      acc = fma(p.x, q.x, fma(p.y, q.y, acc));
    }
    if (!cg_barrier(a, sh, ++gen, acc, a.partials)) return;
    if (threadIdx.x == 0) coef = rr / sh.total;  // alpha
    __syncthreads();
    const double alpha = coef;
    acc = 0.0;
    for (int h = h0 + threadIdx.x; h < h1; h += kCgThreads) {
      const double2 p = __ldcg(pn + h), q = __ldcg(a.q + h);
      double2 x = __ldcg(a.x + h), r = __ldcg(a.r + h);
      x.x = fma(alpha, p.x, x.x);
      x.y = fma(alpha, p.y, x.y);
      r.x = fma(-alpha, q.x, r.x);
      r.y = fma(-alpha, q.y, r.y);
      a.x[h] = x;
      a.r[h] = r;
      acc = fma(r.x, r.x, fma(r.y, r.y, acc));
    }
    if (want) a.status[3] = 1;
    if (!cg_barrier(a, sh, ++gen, acc, a.partials + gridDim.x)) return;
    ++k;
    const double rn = sh.total;
    if (!isfinite(rn) || k >= a.maxit || !(sqrt(rn) > a.stop)) {
      if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.status[0] = k;
        if (!isfinite(rn)) a.status[2] = 1;
      }
      return;
    }
    if (threadIdx.x == 0) coef = rn / rr;  // beta
    __syncthreads();
    beta = coef;
    rr = rn;
    if (k - a.k0 >= (sh.yield ? kCgKeep : a.slice)) {
      if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.status[0] = ~k;
        *a.state = make_double2(rr, beta);
      }
      return;
    }
  }
}

// CG from the residual a.r (|r|^2 in slot kCgSlots + 1) for at most a.maxit iterations, a launch
// per operation, eight iterations queued at a time, on all SMs and without a lease.  Returns
// the iterations.
int run_cg_queued(sw_gauge* g, const CgArgs& a) {
  sw_ctx* c = g->ctx;
  cudaStream_t s = c->stream;
  const long h = g->N / 2;
  constexpr int s_pq = 3, s_stop = 5, kQueue = 8;
  int s_rr[2] = {1, 2};
  double2* p = a.p[1];
  int* ctl = c->many_ctl;
  c->h_slots[kCgSlots + s_stop] = make_double2(a.stop, 0.0);
  SW_CUDA(cudaMemcpyAsync(c->slots + kCgSlots + s_stop, c->h_slots + kCgSlots + s_stop,
                          sizeof(double2), cudaMemcpyHostToDevice, s));
  SW_CUDA(cudaMemsetAsync(ctl, 0, 4 * sizeof(int), s));
  blas_copy(c, p, a.r, h);
  const int* done = c->h_many->ctl;
  for (int issued = 0;;) {
    for (int q = 0; q < kQueue && issued < a.maxit; ++q, ++issued) {
      hop_eo(g, 1, 0.0, nullptr, 1.0, p, a.t, s);  // t_o = D_oe p
      hop_eo(g, 0, a.m2, p, -1.0, a.t, a.q, s);    // q = m^2 p - D_eo t
      many_setup_dot(c, h, Many<2>(kCgSlots, p, a.q), s_pq, ctl);
      many_cg_step(c, h, Many<4>(kCgSlots, a.x, a.r, p, a.q), s_rr[0], s_pq, s_rr[1], s_stop,
                   a.maxit, ctl);
      many_xpay(c, h, Many<2>(kCgSlots, p, a.r), s_rr[1], s_rr[0], ctl);
      std::swap(s_rr[0], s_rr[1]);
    }
    SW_CUDA(cudaMemcpyAsync(c->h_many->ctl, ctl, 4 * sizeof(int), cudaMemcpyDeviceToHost, s));
    SW_CUDA(cudaStreamSynchronize(s));
    if (done[2]) throw SwError{SW_ERR_NAN, "non-finite CG residual"};
    if (done[0]) return done[1];
  }
}

// The persistent kernel from the residual a.r (rr = |r|^2), for at most a.maxit iterations;
// returns them.  The SMs are given back and asked for again after a slice, and every kCgKeep
// iterations while other calls are in flight: the solve goes on from x, r, p, |r|^2 and beta,
// with the same bits.
int run_cg_eo(sw_ctx* c, CgArgs a) {
  static std::atomic<bool> checked[64];
  if (!checked[c->device & 63].load()) {
    int coop = 0, occ = 0;
    SW_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, c->device));
    SW_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_cg_eo, kCgThreads, 0));
    SW_REQUIRE(coop && occ >= 1, SW_ERR_CUDA, "the device cannot run the persistent CG kernel");
    checked[c->device & 63].store(true);
  }
  a.partials = c->partials;
  a.bar = c->bar;
  a.status = c->cgstat;
  a.yield = &c->h_many->yield;
  a.state = c->slots + kCgSlots + 5;
  const long half = (long)a.L0 * a.L1 / 2;
  a.slice = cg_slice(half);
  int* h = c->h_ctl;
  for (a.k0 = 0;; a.k0 = ~h[0]) {
    SmLease lease(c, &c->h_many->yield);  // held until the kernel has finished
    // one CTA per SM; fewer where a CTA would have less than a warp of sites
    long grid = (half + 31) / 32;
    if (grid > lease.sms()) grid = lease.sms();
    if (grid > kReduceBlocks) grid = kReduceBlocks;
    SW_CUDA(cudaMemsetAsync(a.bar, 0, 2 * sizeof(unsigned), c->stream));
    SW_CUDA(cudaMemsetAsync(a.status, 0, 4 * sizeof(int), c->stream));
    void* params[] = {&a};
    SW_CUDA(cudaLaunchCooperativeKernel((const void*)k_cg_eo, dim3((unsigned)grid),
                                        dim3(kCgThreads), params, 0, c->stream));
    sw_count_launch();
    SW_CUDA(cudaMemcpyAsync(h, c->cgstat, 4 * sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    SW_CUDA(cudaStreamSynchronize(c->stream));
    if (h[1]) throw SwError{SW_ERR_TIMEOUT, "even/odd CG: a grid barrier wait gave up"};
    if (h[2]) throw SwError{SW_ERR_NAN, "non-finite CG residual"};
    if (h[0] >= 0) return h[0];
  }
}

}  // namespace

// Solves D x = b by CG on the even normal system; b, x lexicographic device
// buffers.  work: 7 half vectors + 1 full.  Returns iterations (negative on
// non-convergence) and fills the true residual.
int cg_eo_device(sw_gauge* g, double m, const double2* b, double2* x, double tol, int maxit,
                 double2* work, int* iters, double* true_resid) {
  sw_ctx* c = g->ctx;
  cudaStream_t s = c->stream;
  long N = g->N, h = N / 2;
  double2 *be = work, *bo = work + h, *xe = work + 2 * h, *r = work + 3 * h, *p = work + 4 * h,
          *q = work + 5 * h, *t = work + 6 * h, *full = work + 7 * h;
  int blocks = (int)((N + 255) / 256);
  k_split_eo<<<blocks, 256, 0, s>>>(b, be, bo, g->L0, g->L1);
  SW_LAUNCH_CHECK();
  constexpr int sb = kCgSlots;
  blas_norm2(c, b, N, sb + 0);
  double bn = std::sqrt(slot_read(c, sb + 0).x);
  if (!std::isfinite(bn)) throw SwError{SW_ERR_NAN, "non-finite right-hand side"};
  // rhs = m b_e - D_eo b_o (in place of b_e), x_e = 0
  hop_eo(g, 0, m, be, -1.0, bo, be, s);
  blas_zero(c, xe, h);
  double stop = bn > 0.0 ? tol * m * bn : 0.0;
  int total = 0, sms = 0;
  SW_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device));
  const bool queued = cg_queued(h, SmLease::share(c, sms));
  // CG with reliable restarts: when the recurrence residual meets the target,
  // the true residual rhs - M x_e is recomputed; if it is still above the
  // target (recurrence drift at small m), CG restarts from it.
  for (int attempt = 0; attempt < 8 && bn > 0.0 && total < maxit; ++attempt) {
    hop_eo(g, 1, 0.0, nullptr, 1.0, xe, t, s);
    hop_eo(g, 0, m * m, xe, -1.0, t, q, s);
    blas_sub(c, r, be, q, h);
    blas_norm2(c, r, h, sb + 1);
    double rr0 = slot_read(c, sb + 1).x;
    if (!std::isfinite(rr0)) throw SwError{SW_ERR_NAN, "non-finite CG residual"};
    if (std::sqrt(rr0) <= stop) break;
    CgArgs a{};
    a.W = g->W_lex;
    a.x = xe;
    a.r = r;
    a.q = q;
    a.t = t;
    a.p[0] = full;  // overwritten by the residual check afterwards
    a.p[1] = p;
    a.L0 = g->L0;
    a.L1 = g->L1;
    a.maxit = maxit - total;
    a.m2 = m * m;
    a.rr = rr0;
    a.stop = stop;
    total += queued ? run_cg_queued(g, a) : run_cg_eo(c, a);
  }
  *iters = total;
  // x_o = (b_o - D_oe x_e) / m
  hop_eo(g, 1, 1.0 / m, bo, -1.0 / m, xe, t, s);
  k_join_eo<<<blocks, 256, 0, s>>>(xe, t, x, g->L0, g->L1);
  SW_LAUNCH_CHECK();
  launch_dslash_lex(g, m, 0, x, full, s);
  blas_sub(c, full, b, full, N);
  blas_norm2(c, full, N, sb + 4);
  double rn = std::sqrt(slot_read(c, sb + 4).x);
  *true_resid = bn > 0.0 ? rn / bn : 0.0;
  return (bn == 0.0 || *true_resid <= tol) ? SW_OK : SW_ERR_NOCONV;
}

extern "C" int sw_cg_eo_solve(sw_gauge* g, double mass, const void* b, void* x, double tol,
                              int maxiter, int on_device, sw_solve_stats* st) {
  if (!g || !b || !x) return SW_ERR_ARG;
  sw_ctx* c = g->ctx;
  const CallScope scope(c);
  try {
    c->err.clear();
    SW_CUDA(cudaSetDevice(c->device));
    cudaError_t stale = cudaGetLastError();
    if (stale != cudaSuccess) report_stale_error(stale);
    SW_REQUIRE(std::isfinite(mass) && mass > 0.0, SW_ERR_ARG, "mass must be > 0");
    SW_REQUIRE(tol > 0.0 && maxiter >= 0, SW_ERR_ARG, "tol must be > 0, maxiter >= 0");
    auto t0 = std::chrono::steady_clock::now();
    long N = g->N;
    double2* work = nullptr;
    cudaError_t e = cudaMalloc(&work, (size_t)(7 * (N / 2) + N + 2 * N) * sizeof(double2));
    if (e != cudaSuccess) {
      cudaGetLastError();
      throw SwError{SW_ERR_OOM, "CG work buffers"};
    }
    double2* db = work + 7 * (N / 2) + N;
    double2* dx = db + N;
    int iters = 0, rc = SW_OK;
    double tr = 0.0;
    try {
      if (!on_device)
        SW_CUDA(cudaMemcpyAsync(db, b, N * sizeof(double2), cudaMemcpyHostToDevice, c->stream));
      rc = cg_eo_device(g, mass, on_device ? (const double2*)b : db,
                        on_device ? (double2*)x : dx, tol, maxiter, work, &iters, &tr);
      if (!on_device)
        SW_CUDA(cudaMemcpyAsync(x, dx, N * sizeof(double2), cudaMemcpyDeviceToHost, c->stream));
      SW_CUDA(cudaStreamSynchronize(c->stream));
    } catch (...) {
      dev_free(work, "CG work");
      throw;
    }
    dev_free(work, "CG work");
    if (st) {
      std::memset(st, 0, sizeof(*st));
      st->converged = rc == SW_OK;
      st->outer_iters = iters;
      st->fine_applies = iters + 1;
      st->true_resid = tr;
      st->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    }
    if (rc != SW_OK) c->err = "CG reached maxiter";
    return rc;
  } catch (const SwError& err) {
    c->err = err.msg;
    return err.code;
  }
}
