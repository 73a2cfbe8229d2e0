// Multigrid hierarchy: setup and K-cycle solve (Sec. IV, Table kcycle).
//
// Setup per level l (0 = fine): nv near-null vectors psi = psi0 + e, e from CG
// on A A^dag e = -A A^dag psi0 (tolerance setup_tol, setup_maxiter
// iterations); global modified Gram-Schmidt; chiral doubling and modified
// Gram-Schmidt per (aggregate, chirality) -> P; Galerkin stencil
// Y = P^dag A P and its adjoint stencil.
//
// Solve: flexible GCR(outer_restart) on S z_e = b_e - A_eo b_o with
// S = I - A_eo A_oe, preconditioned by the K-cycle: MR(smoother_iters, omega)
// on S; restrict (r_e, 0); GCR(inter_restart, max inter_maxiter, tol
// inter_tol) on A_hat preconditioned by the next K-cycle, or CGNE (tol
// coarsest_tol, max coarsest_maxiter) on the coarsest level; prolong and keep
// the even part; r2 = r1 - S e; MR post-smoother on r2; p = x1 + e + x3.
// Then z_o = b_o - A_oe z_e and x = B^-1 z.
//
// Krylov coefficients stay on the device (Coef slots); the host reads back
// only the residual norms its stopping tests branch on.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <tuple>

#include "lease.h"
#include "many.h"
#include "sw_internal.h"
#include "sw_mg.h"

namespace {

double2* dalloc(long n) {
  void* p = nullptr;
  if (n <= 0) n = 1;
  cudaError_t e = cudaMalloc(&p, n * sizeof(double2));
  if (e != cudaSuccess) {
    cudaGetLastError();
    throw SwError{SW_ERR_OOM, std::string("cudaMalloc of ") + std::to_string(n * 16) +
                                  " bytes failed: " + cudaGetErrorString(e)};
  }
  sw_poison(p, n * sizeof(double2));
  return (double2*)p;
}

}  // namespace

void sw_mg_release(sw_mg* mg) {
  for (double2* p : mg->allocs) dev_free(p, "hierarchy buffer");
  mg->allocs.clear();
}

double2* ScopedBuffers::get(long n) {
  double2* p = dalloc(n);
  list.push_back(p);
  return p;
}

ScopedBuffers::~ScopedBuffers() {
  for (double2* p : list) dev_free(p, "call scratch");
}

double2* mg_alloc(sw_mg* mg, long n) {
  double2* p = dalloc(n);
  mg->allocs.push_back(p);
  return p;
}

// ---------------------------------------------------------------- operators
long level_len(const sw_mg* mg, int l) {
  const MgLevel& L = mg->lev[l];
  if (l == 0) return mg->fine_D ? mg->g->N : mg->g->N / 2;
  return L.ndof;
}

// FP64 stencil of a coarse level (dagger: its adjoint) on the members of v, on
// its digit entries where the level keeps them.  ctl: see many.h.
void coarse_op(sw_mg* mg, int l, int dagger, const Many<2>& v, const int* ctl) {
  sw_ctx* c = mg->ctx;
  const MgLevel& L = mg->lev[l];
  const CoarseGeom cg{L.E0, L.E1, L.nc};
  unsigned long long* exec = c->timing ? c->exec + l : nullptr;
  if (L.dg.T)
    many_digit(cg, L.dg, L.Y, dagger, v, c->device, c->stream, ctl, exec);
  else
    many_coarse(cg, L.Y, dagger, v, c->stream, ctl, exec);
}

// Operator of level l in the solve on (in, out, tmp) of every member: S on level
// 0 (even half), A_hat below.  lowp: inside the preconditioner of a
// mixed-precision hierarchy -- the fine Schur operator then runs in FP32 and
// intermediate stencils in scaled FP16.
void level_op(sw_mg* mg, int l, const Many<3>& v, bool lowp, const int* ctl = nullptr) {
  sw_ctx* c = mg->ctx;
  int tk = timing_begin(c, l, v.n);
  if (l == 0 && mg->fine_D) {
    for (int m = 0; m < v.n; ++m)
      launch_dslash_ps(mg->g, mg->mass, 0, v.v[0][m], v.v[1][m], c->stream);
  } else if (l == 0 && lowp && mg->mixed) {
    many_S32(mg->g, mg->g->W_ps32, mg->binv32, v, c->stream);
  } else if (l == 0) {
    many_S(mg->g, mg->binv, v, c->stream);
  } else {
    const MgLevel& L = mg->lev[l];
    Many<2> io;
    for (int m = 0; m < v.n; ++m) io.add(0, v.v[0][m], v.v[1][m]);
    if (lowp && mg->mixed && L.Yh)
      many_coarse_h(CoarseGeom{L.E0, L.E1, L.nc}, L.Yh, L.Ysc, 0, io, c->stream);
    else
      coarse_op(mg, l, 0, io, ctl);
  }
  timing_end(c, tk);
}
// Normal operator used by the setup on level l: A A^dag on (in, out, t, u) of every
// member (full fine vectors on level 0).  Its products are FP64 FMAs in a fixed order on
// every level, not the digit products of the solves (see mg_setup).
void level_normal(sw_mg* mg, int l, const Many<4>& v, const int* ctl) {
  sw_ctx* c = mg->ctx;
  if (l == 0 && mg->fine_D) {
    for (int m = 0; m < v.n; ++m) {
      launch_dslash_ps(mg->g, mg->mass, 1, v.v[0][m], v.v[2][m], c->stream);
      launch_dslash_ps(mg->g, mg->mass, 0, v.v[2][m], v.v[1][m], c->stream);
    }
  } else if (l == 0) {
    many_normal_A(mg->g, mg->binv, v, c->stream, ctl);
  } else {
    for (int dagger = 1; dagger >= 0; --dagger) {
      Many<2> io;
      for (int m = 0; m < v.n; ++m) io.add(0, v.v[dagger ? 0 : 2][m], v.v[dagger ? 2 : 1][m]);
      const MgLevel& L = mg->lev[l];
      const int tk = timing_begin(c, l, v.n);
      many_coarse(CoarseGeom{L.E0, L.E1, L.nc}, L.Y, dagger, io, c->stream, ctl,
                  c->timing ? c->exec + l : nullptr);
      timing_end(c, tk);
    }
  }
}

static void check_norm(double v, const char* where) {
  if (!std::isfinite(v)) throw SwError{SW_ERR_NAN, std::string("non-finite norm in ") + where};
}

// ---------------------------------------------------------------- Krylov
// CG on the normal error (Craig): x = op^dag y with op op^dag y = b.  The
// stopping test runs on the device (iter_check); the host queues kIterBatch
// iterations at a time and reads the control block between batches, so the
// iterations need no host round trip.  Iterates and counts are those of the
// sequential loop: every kernel after the stopping iteration is a no-op.
constexpr int kIterBatch = 8;

// Autotuner records, keyed by (device, nc, batch width, coarse sites, SMs used): the
// pipeline depth of the batched tensor-core kernel.
struct TuneRec {
  int stages;
  double us_per_iter;
};
static std::mutex g_tune_mutex;
static std::map<std::tuple<int, int, int, int, int>, TuneRec> g_tune;  // + SMs used

static int cgne(sw_mg* mg, int l, const double2* b, double2* x) {
  sw_ctx* c = mg->ctx;
  MgLevel& L = mg->lev[l];
  long n = level_len(mg, l);
  if (mg->persistent_cgne) {
    SmLease lease(c);  // held until the kernel has finished
    const char* dfenv = std::getenv("SW_COARSEST_DF64");
    const CoarseGeom cg{L.E0, L.E1, L.nc};
    const int tk = timing_begin(c, kCatCgne);
    bool ran = mg->mixed && L.Ydf && dfenv && dfenv[0] == '1' &&
               launch_cgne_df(cg, L.Ydf, b, x, L.gr, L.cp, L.cdf, L.cdf + L.ndof, c->partials,
                              c->bar, c->cgstat, mg->p.coarsest_maxiter, mg->p.coarsest_tol,
                              c->device, c->stream, mg->stall_test, lease.sms());
    if (!ran && L.dg.T)
      ran = launch_cgne64(cg, L.dg, b, x, L.gr, L.cp, c->partials, c->bar, c->cgstat,
                          mg->p.coarsest_maxiter, mg->p.coarsest_tol, c->device, c->stream,
                          mg->stall_test, lease.sms());
    timing_end(c, tk);
    if (ran) {
      SW_CUDA(cudaMemcpyAsync(c->h_ctl, c->cgstat, 3 * sizeof(int), cudaMemcpyDeviceToHost,
                              c->stream));
      SW_CUDA(cudaStreamSynchronize(c->stream));
      if (!c->pending.empty()) timing_harvest(c);
      if (c->timing) c->t_count[kCatCgne + 1] += c->h_ctl[0];  // iterations, for flop counts
      if (c->h_ctl[1])
        throw SwError{SW_ERR_TIMEOUT, "coarsest CGNE: a grid barrier wait gave up"};
      if (c->h_ctl[2]) throw SwError{SW_ERR_NAN, "non-finite norm in CGNE residual"};
      if (mg->verbose > 1)
        std::fprintf(stderr, "[sw]     coarsest CGNE launch: %d iterations\n", c->h_ctl[0]);
      return c->h_ctl[0];
    }
  }
  int sb = slot_base(l);
  int s_rr[2] = {sb + 10, sb + 11}, s_pp = sb + 12;
  int* ctl = c->ctl + 4 * l;
  int maxit = mg->p.coarsest_maxiter;
  blas_zero(c, x, n);
  blas_copy(c, L.gr, b, n);
  blas_norm2(c, L.gr, n, s_rr[0]);
  double rr = slot_read(c, s_rr[0]).x;
  check_norm(rr, "CGNE residual");
  double stop = mg->p.coarsest_tol * std::sqrt(rr);
  const auto op = [&](int dagger, const double2* in, double2* out, const int* skip) {
    const int tk = timing_begin(c, l);
    coarse_op(mg, l, dagger, Many<2>(0, in, out), skip);
    timing_end(c, tk);
  };
  op(1, L.gr, L.cp, nullptr);
  iter_init(c, ctl, s_rr[0], stop, maxit);
  int cur = 0;
  for (int issued = 0;;) {
    for (int q = 0; q < kIterBatch && issued < maxit; ++q, ++issued) {
      blas_norm2(c, L.cp, n, s_pp, ctl);
      blas_axpy(c, x, L.cp, n, coef_ratio(s_rr[cur], s_pp, 1.0), ctl);
      op(0, L.cp, L.cw, ctl);
      blas_axpy(c, L.gr, L.cw, n, coef_ratio(s_rr[cur], s_pp, -1.0), ctl);
      blas_norm2(c, L.gr, n, s_rr[1 - cur], ctl);
      iter_check(c, ctl, s_rr[1 - cur], stop, maxit);
      op(1, L.gr, L.cw, ctl);
      blas_xpay(c, L.cp, L.cw, n, coef_ratio(s_rr[1 - cur], s_rr[cur], 1.0), ctl);
      cur = 1 - cur;
    }
    iter_read(c, ctl, c->h_ctl);
    if (c->h_ctl[2]) throw SwError{SW_ERR_NAN, "non-finite norm in CGNE residual"};
    if (c->h_ctl[0] || issued >= maxit) break;
  }
  return c->h_ctl[1];
}

// CG on the Hermitian positive semi-definite A A^dag (setup) for all members of the
// set in lockstep: x from zero, right-hand sides -q.  Stopping tests on the device;
// the host looks at them after kIterBatch iterations.  Returns the iterations of each.
struct SetupVecs {
  std::vector<double2*> x, r, p, q, t, u;
};
static std::vector<int> cg_setup(sw_mg* mg, int l, const SetupVecs& v, int w) {
  sw_ctx* c = mg->ctx;
  const long n = mg->lev[l].ndof;
  const int maxit = mg->p.setup_maxiter;
  constexpr int s_pq = 22, s_stop = 23;
  int s_rr[2] = {20, 21};
  Many<4> start, op, step;
  Many<2> pq, pr;
  for (int m = 0; m < w; ++m) {
    const int slot = slot_base(l) + (m + 1) * kSlotPage;
    start.add(slot, v.x[m], v.r[m], v.p[m], v.q[m]);
    op.add(slot, v.p[m], v.q[m], v.t[m], v.u[m]);
    step.add(slot, v.x[m], v.r[m], v.p[m], v.q[m]);
    pq.add(slot, v.p[m], v.q[m]);
    pr.add(slot, v.p[m], v.r[m]);
  }
  int* ctl = c->many_ctl;
  many_cg_start(c, n, start, s_rr[0], s_stop, mg->p.setup_tol, maxit, ctl);
  for (int issued = 0;;) {
    SW_CUDA(cudaMemcpyAsync(c->h_many->ctl, ctl, 4 * w * sizeof(int), cudaMemcpyDeviceToHost,
                            c->stream));
    SW_CUDA(cudaStreamSynchronize(c->stream));
    if (!c->pending.empty()) timing_harvest(c);
    bool done = true;
    for (int m = 0; m < w; ++m) {
      if (c->h_many->ctl[4 * m + 2])
        throw SwError{SW_ERR_NAN, "non-finite norm in setup CG residual"};
      done = done && c->h_many->ctl[4 * m];
    }
    if (done) break;
    for (int q = 0; q < kIterBatch && issued < maxit; ++q, ++issued) {
      level_normal(mg, l, op, ctl);
      many_setup_dot(c, n, pq, s_pq, ctl);
      many_cg_step(c, n, step, s_rr[0], s_pq, s_rr[1], s_stop, maxit, ctl);
      many_xpay(c, n, pr, s_rr[1], s_rr[0], ctl);
      std::swap(s_rr[0], s_rr[1]);
    }
  }
  std::vector<int> its(w);
  for (int m = 0; m < w; ++m) its[m] = c->h_many->ctl[4 * m + 1];
  return its;
}

int mg_coarsest_solve(sw_mg* mg, const double2* b, double2* x) {
  return cgne(mg, mg->nlev - 1, b, x);
}

// ---------------------------------------------------------------- setup
// Digit entries of a level for the solves.  They are a second copy of its stencil, without
// which coarse_op and cgne work on Y: none where the kernels cannot index them, where there
// would be more than SW_DIGIT_ENTRIES (environment), or where the device has no memory left.
static void make_digits(sw_mg* mg, MgLevel& L) {
  const CoarseGeom geom{L.E0, L.E1, L.nc};
  const long n = digit_entries(geom);
  const char* lim = std::getenv("SW_DIGIT_ENTRIES");
  if (n > kMaxDigitEntries || (lim && n > std::atol(lim))) return;
  uint4* T = nullptr;
  try {
    T = (uint4*)mg_alloc(mg, n + (digit_rows(geom) + 3) / 4);
  } catch (const SwError& e) {
    if (e.code != SW_ERR_OOM) throw;
    if (mg->verbose) std::fprintf(stderr, "[sw] no memory for digit entries: %s\n", e.msg.c_str());
    return;
  }
  int* ex = (int*)(T + n);
  launch_pack_digits(geom, L.Y, T, ex, mg->ctx->stream);
  L.dg = DigitStencil{T, ex};
}

// The null vectors depend on every rounding of their relaxation: CG on A A^dag multiplies a
// rounding difference about a thousandfold per step where a KD block is nearly singular
// (|B^-1| up to 1/m), and to order one in some hundreds of steps on any field.  Eight steps at
// 512^2 with other sums and products of the same accuracy moved single elements of the level-2
// stencil by 3e-2.  So that a configuration has one hierarchy, whatever kernels the solves use,
// the operations of a setup have one order: plain FP64 products, and sums as trees over slices
// that depend on n alone (Tree in many.cu), the same for any grouping of the vectors.
void mg_setup(sw_mg* mg, const double* const* psi0, uint64_t seed) {
  sw_ctx* c = mg->ctx;
  sw_gauge* g = mg->g;
  cudaStream_t s = c->stream;
  long N = g->N;
  mg->binv = mg_alloc(mg, N * 4);
  launch_binv_build(g, mg->mass, mg->binv, s);
  mg->lev[0].stmp = mg_alloc(mg, N);
  if (mg->mixed) {
    mg->binv32 = (float2*)mg_alloc(mg, N * 2);
    launch_to_f32(mg->binv, mg->binv32, N * 4, s);
  }
  for (int l = 0; l + 1 < mg->nlev; ++l) {
    ScopedBuffers tmp;  // returned before the next level
    MgLevel& L = mg->lev[l];
    MgLevel& C = mg->lev[l + 1];
    int nv = L.nv;
    long n = L.ndof;
    // Null vectors advance in groups whose vectors are small enough for a launch per
    // operation and vector to be mostly latency (64^2: 4096 elements, 3 us); from 2 M
    // elements on one vector fills the device by itself and the scratch is one
    // vector's.
    const int w = (int)std::min<long>(nv, std::max<long>(1, (1L << 21) / n));
    double2* V = tmp.get(n * nv);
    double2* lex = l == 0 ? tmp.get(n) : nullptr;
    SetupVecs wk;
    for (auto* f : {&wk.x, &wk.r, &wk.p, &wk.q, &wk.t, &wk.u}) {
      f->assign(w, nullptr);
      if (f == &wk.u && l > 0) continue;
      double2* base = tmp.get(n * w);
      for (int m = 0; m < w; ++m) (*f)[m] = base + (long)m * n;
    }
    const int sb = slot_base(l);
    const auto page = [&](int m) { return sb + (m + 1) * kSlotPage; };
    const size_t it0 = mg->setup_iters.size();
    const int passes = mg->p.setup_passes;
    mg->setup_iters.resize(it0 + (size_t)nv * passes);
    for (int i0 = 0; i0 < nv; i0 += w) {
      const int m1 = std::min(w, nv - i0);
      Many<1> psi;
      Many<2> psi_e;
      Many<4> first;
      for (int m = 0; m < m1; ++m) {
        double2* v = V + (long)(i0 + m) * n;
        double2* target = l == 0 ? lex : v;
        if (psi0 && psi0[l])
          SW_CUDA(cudaMemcpyAsync(target, psi0[l] + 2 * (long)(i0 + m) * n, n * sizeof(double2),
                                  cudaMemcpyHostToDevice, s));
        else
          launch_gaussian(sw_stream_seed(seed, l, i0 + m), n, target, s);
        if (l == 0) launch_pack(g, lex, v, s);
        psi.add(page(m), v);
        psi_e.add(page(m), v, wk.x[m]);
        first.add(page(m), v, wk.q[m], wk.t[m], wk.u[m]);
      }
      for (int pass = 0; pass < passes; ++pass) {
        if (pass > 0) {
          many_setup_norm(c, n, psi, 30);
          many_normalise(c, n, psi, 30);
        }
        level_normal(mg, l, first, nullptr);  // e solves A A^dag e = -A A^dag psi
        const std::vector<int> its = cg_setup(mg, l, wk, m1);
        for (int m = 0; m < m1; ++m) mg->setup_iters[it0 + (size_t)(i0 + m) * passes + pass] = its[m];
        many_add(c, n, psi_e);
      }
    }
    // global modified Gram-Schmidt: vector j is normalised and taken out of the later ones
    for (int j = 0; j < nv; ++j) {
      double2* vj = V + (long)j * n;
      many_setup_norm(c, n, Many<1>(page(j), vj), 32, c->h_many->norm + j);
      many_normalise(c, n, Many<1>(page(j), vj), 32);
      Many<2> dots, later;
      for (int i = j + 1; i < nv; ++i) {
        dots.add(page(i), vj, V + (long)i * n);
        later.add(page(i), V + (long)i * n, vj);
      }
      many_setup_dot(c, n, dots, 31);
      many_project(c, n, later, 31);
    }
    SW_CUDA(cudaStreamSynchronize(s));
    for (int i = 0; i < nv; ++i)
      if (!(c->h_many->norm[i] > 0.0) || !std::isfinite(c->h_many->norm[i]))
        throw SwError{SW_ERR_BREAKDOWN, "global Gram-Schmidt: vector " + std::to_string(i) +
                                            " on level " + std::to_string(l + 1) + " has norm 0"};
    // chiral doubling + block orthonormalisation
    L.P = mg_alloc(mg, n * nv);
    SW_CUDA(cudaMemsetAsync(c->flag, 0, sizeof(int), s));
    if (l == 0)
      launch_block_ortho_fine(g, L.b0, L.b1, nv, V, L.P, c->flag, s);
    else
      launch_block_ortho_coarse(CoarseGeom{L.E0, L.E1, L.nc}, L.b0, L.b1, nv, V, L.P, c->flag, s);
    int hflag = 0;
    SW_CUDA(cudaMemcpyAsync(&hflag, c->flag, sizeof(int), cudaMemcpyDeviceToHost, s));
    SW_CUDA(cudaStreamSynchronize(s));
    if (hflag)
      throw SwError{SW_ERR_BREAKDOWN,
                    "block orthonormalisation met a zero vector on level " + std::to_string(l + 1)};
    // Galerkin coarse operator and its adjoint stencil
    long ysz = (long)C.E0 * C.E1 * 5 * C.nc * C.nc;
    C.Y = mg_alloc(mg, ysz);
    if (l == 0) {
      double2* Wv = tmp.get(N * 2 * nv);
      if (mg->fine_D)
        launch_build_W_identity(g, nv, L.P, Wv, s);  // Galerkin of D itself: P^dag D P
      else
        launch_build_W(g, nv, mg->binv, L.P, Wv, s);
      launch_build_Y_fine(g, mg->mass, L.b0, L.b1, nv, L.P, Wv, C.Y, s);
    } else {
      double2* T = tmp.get((long)L.E0 * L.E1 * 5 * L.nc * 2 * nv);
      launch_build_Y_coarse(CoarseGeom{L.E0, L.E1, L.nc}, L.b0, L.b1, nv, L.Y, L.P, T, C.Y, s);
    }
    if (mg->mixed) {
      CoarseGeom cg{C.E0, C.E1, C.nc};
      if (l + 2 < mg->nlev) {  // intermediate level: scaled FP16 copy
        C.Yh = (__half2*)mg_alloc(mg, (ysz + 3) / 4);
        C.Ysc = (float*)mg_alloc(mg, ((long)C.E0 * C.E1 * 5 + 3) / 4);
        launch_to_half_scaled(cg, C.Y, C.Yh, C.Ysc, s);
      } else {  // coarsest level: double-float copy
        C.Ydf = (float4*)mg_alloc(mg, ysz);
        launch_to_df64(C.Y, C.Ydf, ysz, s);
        C.cdf = (float4*)mg_alloc(mg, 2 * C.ndof);
      }
    }
    SW_CUDA(cudaStreamSynchronize(s));
  }
  // solve workspace
  for (int l = 0; l < mg->nlev; ++l) {
    MgLevel& L = mg->lev[l];
    long n = level_len(mg, l);
    L.rhs = mg_alloc(mg, n);
    L.sol = mg_alloc(mg, n);
    L.gr = mg_alloc(mg, n);
    L.gtmp = mg_alloc(mg, n);
    int nb = l == 0 ? mg->p.outer_restart : mg->p.inter_restart;
    if (l == mg->nlev - 1) nb = 0;
    L.gp.assign(nb, nullptr);
    L.gq.assign(nb, nullptr);
    for (int k = 0; k < nb; ++k) { L.gp[k] = mg_alloc(mg, n); L.gq[k] = mg_alloc(mg, n); }
    L.cp = mg_alloc(mg, n);
    L.cw = mg_alloc(mg, n);
    if (l + 1 < mg->nlev) {
      L.kx1 = mg_alloc(mg, n); L.kr1 = mg_alloc(mg, n); L.kq = mg_alloc(mg, n);
      L.ke = mg_alloc(mg, n); L.kx3 = mg_alloc(mg, n);
    }
    if (l == 0) {
      L.tmp = L.stmp;
      mg->bps = mg_alloc(mg, N);
      mg->xps = mg_alloc(mg, N);
      mg->lexb = mg_alloc(mg, N);
      mg->lexx = mg_alloc(mg, N);
      mg->lext = mg_alloc(mg, N);
    }
  }
  // last, and with the setup's scratch returned: what a hierarchy can do without
  for (int l = 1; l < mg->nlev; ++l)
    if (l + 1 == mg->nlev || !mg->mixed) make_digits(mg, mg->lev[l]);
  SW_CUDA(cudaStreamSynchronize(s));
}

// ================================================================ lockstep solves
// One solve, or several right-hand sides of one mixed-precision hierarchy, which
// advance through the same K-cycle together: every step is one launch for all
// of them (own work vectors, own page of Krylov scalars, own stopping tests), and
// all of them reach the coarsest level together and share one batched
// coarsest CGNE launch, which reads the coarsest stencil once for the whole
// batch.  A right-hand side that has met a stopping test drops out of the step
// while the others go on.

namespace {

using Set = std::vector<int>;

struct Solve {
  sw_mg* mg;
  bool batch;
  std::vector<long long> fine, inter_it, inter_solves, coarse_it, coarse_solves;
  Solve(sw_mg* m, bool many)
      : mg(m), batch(many), fine(width(), 0), inter_it(width(), 0), inter_solves(width(), 0),
        coarse_it(width(), 0), coarse_solves(width(), 0) {}
  int width() const { return batch ? kMaxBatch : 1; }
  LevelWs& at(int l, int r) { return batch ? mg->batch.lv[l][r] : mg->lev[l]; }
  int slot(int l, int r) const { return slot_base(l) + (batch ? (r + 1) * kSlotPage : 0); }
};

// Waits for the norms that the last sums left in pinned memory.
const double* norms(sw_ctx* c) {
  SW_CUDA(cudaStreamSynchronize(c->stream));
  if (!c->pending.empty()) timing_harvest(c);
  return c->h_many->norm;
}

// SW_VERBOSE >= 3: the 2-norm of a single solve's work vector on stderr (a trace of where a
// non-finite value first appears).  Costs a host round trip per call.
void trace_norm(Solve& S, int l, const char* what, const double2* v) {
  sw_mg* mg = S.mg;
  if (mg->verbose < 3 || S.batch) return;
  blas_norm2(mg->ctx, v, level_len(mg, l), slot_base(l) + 63);
  std::fprintf(stderr, "[sw]       level %d %s |v| %.6e\n", l + 1, what,
               std::sqrt(slot_read(mg->ctx, slot_base(l) + 63).x));
}

void apply(Solve& S, int l, const Set& set, const Many<3>& v, bool lowp) {
  if (l == 0)
    for (int r : set) S.fine[r]++;
  level_op(S.mg, l, v, lowp);
}

// MR smoother with zero initial guess (always part of the preconditioner).  Before the
// coarse correction: x1 = kx1 and r1 = kr1 from b.  After it, on the residual in
// kr1: out = (x1 + e) + x3, the residual it would leave is not formed.
void mr(Solve& S, int l, const Set& set, bool post, const std::vector<const double2*>& b,
        const std::vector<double2*>& out) {
  sw_mg* mg = S.mg;
  sw_ctx* c = mg->ctx;
  const long n = level_len(mg, l);
  const double om = mg->p.omega;
  const int iters = mg->p.smoother_iters;
  constexpr int sq = 8;
  for (int it = 0; it < iters; ++it) {
    const bool last = post && it == iters - 1;
    Many<3> op, step;
    Many<2> qr;
    Many<4> first;
    Many<5> end;
    for (int r : set) {
      LevelWs& W = S.at(l, r);
      const int slot = S.slot(l, r);
      const double2* res = post || it > 0 ? W.kr1 : b[r];
      double2* x = post ? W.kx3 : W.kx1;
      op.add(slot, res, W.kq, W.tmp);
      qr.add(slot, W.kq, res);
      if (last)
        end.add(slot, out[r], x, res, W.kx1, W.ke);
      else if (it == 0)
        first.add(slot, x, W.kr1, res, W.kq);
      else
        step.add(slot, x, W.kr1, W.kq);
    }
    apply(S, l, set, op, true);
    many_dot_norm(c, n, qr, sq);
    if (mg->verbose >= 3 && !S.batch) {
      const double2 a = slot_read(c, slot_base(l) + sq), q2 = slot_read(c, slot_base(l) + sq + 1);
      std::fprintf(stderr, "[sw]       level %d MR %d (q, r) %.6e %+.6ei |q|^2 %.6e\n", l + 1,
                   it, a.x, a.y, q2.x);
    }
    many_mr_first(c, n, first, sq, om);
    many_mr(c, n, step, sq, om);
    many_mr_last(c, n, end, sq, om, it == 0);
  }
  if (iters > 0) return;
  Many<3> init;
  Many<2> sum, more;
  for (int r : set) {
    LevelWs& W = S.at(l, r);
    init.add(S.slot(l, r), W.kx1, W.kr1, b[r]);
    if (!post) continue;
    sum.add(0, out[r], W.kx1);
    more.add(0, out[r], W.ke);
  }
  if (!post) many_init(c, n, init, sq, nullptr);
  many_copy(c, n, sum);
  many_add(c, n, more);
}

void solve_level(Solve& S, int l, const Set& set);

// K-cycle preconditioner: out_r = M(g_r) on level l for every member of the set.
void kcycle(Solve& S, int l, const Set& set, const std::vector<const double2*>& g,
            const std::vector<double2*>& out) {
  sw_mg* mg = S.mg;
  cudaStream_t s = mg->ctx->stream;
  const MgLevel& L = mg->lev[l];
  const CoarseGeom cg{L.E0, L.E1, L.nc};
  trace_norm(S, l, "K-cycle input", g[set[0]]);
  mr(S, l, set, false, g, out);
  trace_norm(S, l, "pre-smoothed x", S.at(l, set[0]).kx1);
  trace_norm(S, l, "pre-smoothed r", S.at(l, set[0]).kr1);
  Many<2> down, up;
  Many<3> op, sub;
  for (int r : set) {
    LevelWs& W = S.at(l, r);
    LevelWs& C = S.at(l + 1, r);
    down.add(0, W.kr1, C.rhs);
    up.add(0, C.sol, W.ke);
    op.add(0, W.ke, W.kq, W.tmp);
    sub.add(0, W.kr1, W.kr1, W.kq);
  }
  if (l == 0)
    many_restrict_fine(mg->g, L.b0, L.b1, L.nv, L.P, down, s, mg->fine_D ? 1 : 0);
  else
    many_restrict_coarse(cg, L.b0, L.b1, L.nv, L.P, down, s);
  trace_norm(S, l + 1, "restricted r", S.at(l + 1, set[0]).rhs);
  solve_level(S, l + 1, set);
  if (l == 0)
    many_prolong_fine(mg->g, L.b0, L.b1, L.nv, L.P, up, s, mg->fine_D ? 1 : 0);
  else
    many_prolong_coarse(cg, L.b0, L.b1, L.nv, L.P, up, s);
  apply(S, l, set, op, true);
  many_sub(mg->ctx, level_len(mg, l), sub);  // r2 = r1 - op e
  mr(S, l, set, true, g, out);
}

struct SetResult {
  std::vector<int> it, restarts;
  std::vector<char> conv;
  explicit SetResult(int n) : it(n, 0), restarts(n, 0), conv(n, 0) {}
};

// Flexible restarted GCR for every member of the set (see the oracle's fgcr for the
// steps), to |r| <= tol[r] (rel: times |b_r|).  confirm: on the true residual.
SetResult fgcr(Solve& S, int l, const Set& set, const std::vector<const double2*>& b,
               const std::vector<double2*>& x, std::vector<double> tol, bool rel, int restart,
               int maxiter, bool confirm) {
  sw_mg* mg = S.mg;
  sw_ctx* c = mg->ctx;
  const long n = level_len(mg, l);
  const int nb = S.width();
  const bool lowp = l > 0;  // intermediate solves are part of the preconditioner
  constexpr int s_rr = 0, s_qq = 2, s_a = 3, s_b = 4;
  double* host = c->h_many->norm;
  SetResult res(nb);
  std::vector<int> k(nb, 0);
  std::vector<double> rn(nb, 0.0);
  Many<3> init;
  for (int r : set) init.add(S.slot(l, r), x[r], S.at(l, r).gr, b[r]);
  many_init(c, n, init, s_rr, host);
  const double* hn = norms(c);
  for (size_t m = 0; m < set.size(); ++m) {
    rn[set[m]] = std::sqrt(hn[m]);
    check_norm(rn[set[m]], "GCR residual");
    if (rel) tol[set[m]] *= rn[set[m]];
  }
  // r = b - op x from x, with its norm
  const auto true_residual = [&](const Set& who, bool keep) {
    Many<3> op, sub;
    for (int r : who) {
      LevelWs& W = S.at(l, r);
      op.add(0, x[r], W.gtmp, W.tmp);
      sub.add(S.slot(l, r), keep ? W.gr : W.gtmp, b[r], W.gtmp);
    }
    apply(S, l, who, op, lowp);
    many_sub_norm(c, n, sub, s_rr, host);
    hn = norms(c);
    for (size_t m = 0; m < who.size(); ++m) {
      rn[who[m]] = std::sqrt(hn[m]);
      check_norm(rn[who[m]], "GCR true residual");
    }
  };
  for (Set act = set; !act.empty();) {
    Set cand, go;
    for (int r : act)
      if (rn[r] <= tol[r]) {
        if (confirm)
          cand.push_back(r);
        else
          res.conv[r] = 1;
      } else if (res.it[r] < maxiter) {
        go.push_back(r);
      }
    if (!cand.empty()) {
      true_residual(cand, false);
      Many<2> keep;
      for (int r : cand) {
        if (rn[r] <= tol[r]) {
          res.conv[r] = 1;
          continue;
        }
        keep.add(0, S.at(l, r).gr, S.at(l, r).gtmp);
        k[r] = 0;
        res.restarts[r]++;
        if (res.it[r] < maxiter) go.push_back(r);
      }
      many_copy(c, n, keep);
      std::sort(go.begin(), go.end());
    }
    act = go;
    if (go.empty()) break;
    std::vector<const double2*> g(nb, nullptr);
    std::vector<double2*> p(nb, nullptr);
    Many<3> op, scale;
    Many<1> alone;
    Many<2> dots;
    Many<4> upd;
    int most = 0;
    for (int r : go) {
      LevelWs& W = S.at(l, r);
      const int slot = S.slot(l, r);
      double2* q = W.gq[k[r]];
      g[r] = W.gr;
      p[r] = W.gp[k[r]];
      op.add(slot, p[r], q, W.tmp);
      if (k[r] > 0)
        dots.add(slot, W.gq[0], q);
      else
        alone.add(slot, q);
      scale.add(slot, q, p[r], W.gr);
      upd.add(slot, x[r], W.gr, p[r], q);
      most = std::max(most, k[r]);
    }
    kcycle(S, l, go, g, p);
    apply(S, l, go, op, lowp);
    many_norm(c, n, alone, s_qq);
    many_dot(c, n, dots, s_b);
    for (int j = 0; j < most; ++j) {
      Many<5> mgs;
      for (int r : go) {
        if (k[r] <= j) continue;
        LevelWs& W = S.at(l, r);
        mgs.add(S.slot(l, r), W.gq[k[r]], p[r], W.gq[j], W.gp[j],
                j + 1 < k[r] ? W.gq[j + 1] : nullptr);
      }
      many_mgs(c, n, mgs, s_b, s_qq);
    }
    many_scale_dot(c, n, scale, s_qq, s_a);
    many_update(c, n, upd, s_a, s_rr, host);
    Set again;
    for (int r : go) {
      ++k[r];
      ++res.it[r];
      if (!S.batch && l == 1 && mg->verbose > 1)
        std::fprintf(stderr, "[sw]   level-2 GCR %d |r| %.3e (tol %.3e)\n", res.it[r], rn[r], tol[r]);
      if (!S.batch && l == 0 && mg->verbose)
        std::fprintf(stderr, "[sw] outer %d |r| %.3e  inter %lld/%lld coarsest %lld/%lld\n",
                     res.it[r], rn[r], S.inter_it[r], S.inter_solves[r], S.coarse_it[r],
                     S.coarse_solves[r]);
      if (k[r] == restart && res.it[r] < maxiter) {
        again.push_back(r);
        k[r] = 0;
        res.restarts[r]++;
      }
    }
    hn = norms(c);
    for (size_t m = 0; m < go.size(); ++m) {
      rn[go[m]] = std::sqrt(hn[m]);
      check_norm(rn[go[m]], "GCR residual");
    }
    if (!again.empty()) true_residual(again, true);
  }
  return res;
}

void cgne_b(Solve& S, int l, const Set& set, int stall = 0);

void solve_level(Solve& S, int l, const Set& set) {
  sw_mg* mg = S.mg;
  if (l == mg->nlev - 1) {
    if (S.batch) return cgne_b(S, l, set);
    S.coarse_it[0] += cgne(mg, l, S.at(l, 0).rhs, S.at(l, 0).sol);
    S.coarse_solves[0]++;
    return;
  }
  std::vector<const double2*> b(S.width(), nullptr);
  std::vector<double2*> x(S.width(), nullptr);
  for (int r : set) {
    b[r] = S.at(l, r).rhs;
    x[r] = S.at(l, r).sol;
  }
  const SetResult res = fgcr(S, l, set, b, x, std::vector<double>(S.width(), mg->p.inter_tol), true,
                             mg->p.inter_restart, mg->p.inter_maxiter, false);
  for (int r : set) {
    S.inter_it[r] += res.it[r];
    S.inter_solves[r]++;
  }
}

// ---------------------------------------------------------------- autotuner
// Pipeline depth of the tensor-core batched CGNE, chosen on first use per
// (device, nc, width, coarse sites) by timing each candidate for a few
// iterations on the call's own data (the real solve then starts from scratch).

int tc_stages(sw_mg* mg, const MgLevel& L, int nb, double2* const* bptr, double2* const* xptr,
              int sms) {
  sw_ctx* c = mg->ctx;
  BatchWs& B = mg->batch;
  const int K = tc_width(nb);
  const bool f32 = mg->p.batch_iterates == SW_PREC_FP32;
  // batch widths of FP32-iterate runs are recorded as 100 + K
  const auto key = std::make_tuple(c->device, L.nc, f32 ? 100 + K : K, L.E0 * L.E1, sms);
  {
    std::lock_guard<std::mutex> lk(g_tune_mutex);
    auto it = g_tune.find(key);
    if (it != g_tune.end()) return it->second.stages;
  }
  int opts[8];
  const int nopt = tc_stage_options(L.nc, K, opts);
  SW_REQUIRE(nopt > 0, SW_ERR_ARG, "no tensor-core tiling fits shared memory");
  // each candidate: a warm-up launch, then the fastest of kReps launches of
  // kTuneIters iterations (the minimum is robust against other streams' work)
  constexpr int kTuneIters = 16, kReps = 3;
  const CoarseGeom cg{L.E0, L.E1, L.nc};
  const float keep = tc_l2_fraction(cg, c->device);
  cudaEvent_t e0, e1;
  SW_CUDA(cudaEventCreate(&e0));
  SW_CUDA(cudaEventCreate(&e1));
  TuneRec best{opts[0], 1e30};
  // candidates: every pipeline depth, with the stencil tiles streamed through
  // L2 (choice S) or partly kept there (choice 10 + S)
  for (int k = 0; k < 2 * nopt; ++k) {
    const int choice = opts[k % nopt] + (k >= nopt ? 10 : 0);
    float fastest = 1e30f;
    for (int rep = 0; rep <= kReps; ++rep) {  // rep 0 is a warm-up
      SW_CUDA(cudaEventRecord(e0, c->stream));
      bool ran = launch_cgne_tc(cg, choice % 10, f32, B.At, B.Ad, nb, bptr, xptr, B.X, B.R, B.P,
                                B.Rt, B.Pt, B.partials, B.bar, B.status, kTuneIters, 0.0,
                                c->device, c->stream, 0, sms, choice >= 10 ? keep : 0.f);
      SW_CUDA(cudaEventRecord(e1, c->stream));
      SW_CUDA(cudaEventSynchronize(e1));
      SW_REQUIRE(ran, SW_ERR_ARG, "tensor-core batched CGNE has no variant for this shape");
      int st0 = 0;
      SW_CUDA(cudaMemcpy(&st0, B.status, sizeof(int), cudaMemcpyDeviceToHost));
      SW_REQUIRE(st0 == 0, SW_ERR_TIMEOUT, "batched coarsest CGNE: a wait gave up while tuning");
      float ms = 0.f;
      SW_CUDA(cudaEventElapsedTime(&ms, e0, e1));
      if (rep > 0 && ms < fastest) fastest = ms;
    }
    const double us = 1e3 * fastest / kTuneIters;
    if (us < best.us_per_iter) best = TuneRec{choice, us};
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  std::lock_guard<std::mutex> lk(g_tune_mutex);
  g_tune[key] = best;
  return best.stages;
}

void cgne_b(Solve& S, int l, const Set& set, int stall) {
  if (set.empty()) return;
  sw_mg* mg = S.mg;
  sw_ctx* c = mg->ctx;
  MgLevel& L = mg->lev[l];
  BatchWs& B = mg->batch;
  const int nb = (int)set.size();
  const bool tc = tc_supported(L.nc) && !B.Yf;
  const bool f32 = mg->p.batch_iterates == SW_PREC_FP32;
  double2** hp = c->h_many->ptr;  // pinned; the wait for the status below ends its use
  for (int i = 0; i < nb; ++i) {
    hp[i] = B.lv[l][set[i]].rhs;
    hp[kMaxBatch + i] = B.lv[l][set[i]].sol;
  }
  SW_CUDA(cudaMemcpyAsync(B.dptr, hp, sizeof(c->h_many->ptr), cudaMemcpyHostToDevice, c->stream));
  SmLease lease(c);
  std::vector<int> its(nb, 0);
  // the CUDA-core FP32 kernel (SW_BATCH_FP32=1) takes at most 16 at a time
  const int chunk = tc ? kMaxBatch : 16;
  for (int i0 = 0; i0 < nb; i0 += chunk) {
    const int m = std::min(chunk, nb - i0);
    bool ran;
    int tk;
    if (tc) {
      const int choice = tc_stages(mg, L, m, B.dptr + i0, B.dptr + kMaxBatch + i0, lease.sms());
      const CoarseGeom cg{L.E0, L.E1, L.nc};
      tk = timing_begin(c, kCatCgne);
      ran = launch_cgne_tc(cg, choice % 10, f32, B.At, B.Ad, m, B.dptr + i0,
                           B.dptr + kMaxBatch + i0, B.X, B.R, B.P, B.Rt, B.Pt, B.partials,
                           B.bar, B.status, mg->p.coarsest_maxiter, mg->p.coarsest_tol,
                           c->device, c->stream, stall, lease.sms(),
                           choice >= 10 ? tc_l2_fraction(cg, c->device) : 0.f);
    } else {
      tk = timing_begin(c, kCatCgne);
      ran = launch_cgne_batch(CoarseGeom{L.E0, L.E1, L.nc}, B.Yf, B.Yd, m, B.dptr + i0,
                              B.dptr + kMaxBatch + i0, B.X, B.R, B.P, B.Rf, B.Pf, B.partials,
                              B.bar, B.status, mg->p.coarsest_maxiter, mg->p.coarsest_tol,
                              c->device, c->stream, lease.sms());
    }
    timing_end(c, tk);
    if (!ran)
      throw SwError{SW_ERR_ARG, "no batched coarsest solver for nc = " + std::to_string(L.nc)};
    const int* hst = c->h_many->status;
    SW_CUDA(cudaMemcpyAsync(c->h_many->status, B.status, sizeof(c->h_many->status),
                            cudaMemcpyDeviceToHost, c->stream));
    SW_CUDA(cudaStreamSynchronize(c->stream));
    if (!c->pending.empty()) timing_harvest(c);
    if (hst[0])
      throw SwError{SW_ERR_TIMEOUT,
                    "batched coarsest CGNE: a wait gave up or a buffer was misaligned"};
    if (hst[1]) throw SwError{SW_ERR_NAN, "non-finite norm in batched CGNE"};
    int kernel_it = 0;  // the launch runs as many iterations as its slowest right-hand side
    for (int i = 0; i < m; ++i) {
      its[i0 + i] = hst[2 + i];
      kernel_it = std::max(kernel_it, hst[2 + i]);
    }
    if (c->timing) c->t_count[kCatCgne + 1] += kernel_it;
  }
  for (int i = 0; i < nb; ++i) {
    S.coarse_it[set[i]] += its[i];
    S.coarse_solves[set[i]]++;
  }
}

// Per-right-hand-side work vectors for nb right-hand sides (grown on demand)
// and, on the first call, the arrays all of them share.
void batch_alloc(sw_mg* mg, int nb) {
  BatchWs& B = mg->batch;
  sw_ctx* c = mg->ctx;
  long N = mg->g->N;
  if (B.lv.empty()) B.lv.assign(mg->nlev, std::vector<LevelWs>());
  if (nb > B.nb) {
    const int cap = std::min(kMaxBatch, std::max(nb, 2 * B.nb));
    for (int l = 0; l < mg->nlev; ++l) {
      long n = level_len(mg, l);
      bool last = l == mg->nlev - 1;
      int nbas = last ? 0 : (l == 0 ? mg->p.outer_restart : mg->p.inter_restart);
      B.lv[l].resize(cap);
      for (int r = B.nb; r < cap; ++r) {
        LevelWs& W = B.lv[l][r];
        W.rhs = mg_alloc(mg, n);
        W.sol = mg_alloc(mg, n);
        if (last) continue;
        W.gr = mg_alloc(mg, n);
        W.gtmp = mg_alloc(mg, n);
        W.gp.assign(nbas, nullptr);
        W.gq.assign(nbas, nullptr);
        for (int k = 0; k < nbas; ++k) {
          W.gp[k] = mg_alloc(mg, n);
          W.gq[k] = mg_alloc(mg, n);
        }
        W.kx1 = mg_alloc(mg, n); W.kr1 = mg_alloc(mg, n); W.kq = mg_alloc(mg, n);
        W.ke = mg_alloc(mg, n); W.kx3 = mg_alloc(mg, n);
        if (l == 0) W.tmp = mg_alloc(mg, n);
      }
    }
    B.nb = cap;
  }
  if (B.shared) return;
  MgLevel& C = mg->lev[mg->nlev - 1];
  const long nc = C.ndof;
  const long sites = (long)C.E0 * C.E1;
  const CoarseGeom cg{C.E0, C.E1, C.nc};
  B.X = mg_alloc(mg, nc * kMaxBatch);
  B.R = mg_alloc(mg, nc * kMaxBatch);
  B.P = mg_alloc(mg, nc * kMaxBatch);
  const char* fp32 = std::getenv("SW_BATCH_FP32");
  if (tc_supported(C.nc) && !(fp32 && fp32[0] == '1')) {
    // tensor-core kernel: stacked TF32 blocks of A and A^dag, right-hand-side tiles
    const long tiles = sites * 5 * tc_tile_floats(C.nc);
    B.At = (float*)mg_alloc(mg, (tiles + 3) / 4);
    B.Ad = (float*)mg_alloc(mg, (tiles + 3) / 4);
    launch_stack_tiles(cg, C.Y, B.At, 0, c->stream);
    launch_stack_tiles(cg, C.Y, B.Ad, 1, c->stream);
    const long vt = sites * 2L * kMaxBatch * C.nc;
    B.Rt = (float*)mg_alloc(mg, (vt + 3) / 4);
    B.Pt = (float*)mg_alloc(mg, (vt + 3) / 4);
  } else {
    // CUDA-core FP32 kernel: FP32 forward and adjoint blocks
    B.Rf = (float2*)mg_alloc(mg, (nc * 16 + 1) / 2);
    B.Pf = (float2*)mg_alloc(mg, (nc * 16 + 1) / 2);
    long ysz = sites * 5 * C.nc * C.nc;
    B.Yf = (float2*)mg_alloc(mg, (ysz + 1) / 2);
    launch_to_f32(C.Y, B.Yf, ysz, c->stream);
    B.Yd = (float2*)mg_alloc(mg, (ysz + 1) / 2);
    launch_adjoint_f32(cg, C.Y, B.Yd, c->stream);
  }
  int sms = 0;
  SW_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device));
  B.partials = (double*)mg_alloc(mg, (long)kMaxBatch * sms);  // 2 phases x 64 x SMs doubles
  B.bar = (unsigned*)mg_alloc(mg, 1);
  B.status = (int*)mg_alloc(mg, (2 + kMaxBatch + 3) / 4);
  B.dptr = (double2**)mg_alloc(mg, kMaxBatch);  // 2 x 64 pointers
  B.bps = mg_alloc(mg, N * kMaxBatch);
  B.xps = mg_alloc(mg, N * kMaxBatch);
  B.lex = mg_alloc(mg, N * kMaxBatch);
  B.shared = true;
}

}  // namespace

// ---------------------------------------------------------------- solve
int mg_solve_device(sw_mg* mg, const double2* b_lex, double2* x_lex, double tol,
                    sw_solve_stats* st) {
  sw_ctx* c = mg->ctx;
  sw_gauge* g = mg->g;
  cudaStream_t s = c->stream;
  long N = g->N, half = N / 2;
  auto t0 = std::chrono::steady_clock::now();
  MgLevel& L = mg->lev[0];
  launch_pack(g, b_lex, mg->bps, s);
  int sb = slot_base(0);
  blas_norm2(c, mg->bps, N, sb + 40);
  double bn = std::sqrt(slot_read(c, sb + 40).x);
  check_norm(bn, "right-hand side");
  if (bn == 0.0) {
    blas_zero(c, x_lex, N);
    SW_CUDA(cudaStreamSynchronize(s));
    if (st) {
      std::memset(st, 0, sizeof(*st));
      st->converged = 1;
    }
    return SW_OK;
  }
  Solve S(mg, false);
  const std::vector<double> tol_abs(1, tol * bn);
  SetResult r(1);
  if (mg->fine_D) {
    // Galerkin MG of D itself: flexible GCR on the full D, no KD preconditioning
    r = fgcr(S, 0, {0}, {mg->bps}, {L.sol}, tol_abs, false, mg->p.outer_restart,
             mg->p.outer_maxiter, true);
    launch_unpack(g, L.sol, x_lex, s);
  } else {
    // b~_e = b_e - A_eo b_o = b_e - C_eo B_o^-1 b_o
    launch_block_apply(g, mg->binv, 1, 0, mg->bps + half, L.stmp + half, s);
    launch_hop(g, 0, -1.0, mg->bps, L.stmp + half, L.rhs, s);
    r = fgcr(S, 0, {0}, {L.rhs}, {L.sol}, tol_abs, false, mg->p.outer_restart,
             mg->p.outer_maxiter, true);
    // z_o = b_o - C_oe B_e^-1 z_e ; x = B^-1 z
    launch_block_apply(g, mg->binv, 0, 0, L.sol, L.stmp, s);
    launch_hop(g, 1, -1.0, mg->bps + half, L.stmp, L.stmp + half, s);
    launch_block_apply(g, mg->binv, 0, 0, L.sol, mg->xps, s);
    launch_block_apply(g, mg->binv, 1, 0, L.stmp + half, mg->xps + half, s);
    launch_unpack(g, mg->xps, x_lex, s);
  }
  // true residual ||b - D x|| / ||b|| in FP64
  launch_dslash_lex(g, mg->mass, 0, x_lex, mg->lext, s);
  blas_sub(c, mg->lext, b_lex, mg->lext, N);
  blas_norm2(c, mg->lext, N, sb + 41);
  double tr = std::sqrt(slot_read(c, sb + 41).x) / bn;
  auto t1 = std::chrono::steady_clock::now();
  if (st) {
    st->converged = r.conv[0] ? 1 : 0;
    st->outer_iters = r.it[0];
    st->restarts = r.restarts[0];
    st->fine_applies = S.fine[0];
    st->inter_iters = S.inter_it[0];
    st->inter_solves = S.inter_solves[0];
    st->coarsest_iters = S.coarse_it[0];
    st->coarsest_solves = S.coarse_solves[0];
    st->true_resid = tr;
    st->seconds = std::chrono::duration<double>(t1 - t0).count();
  }
  return r.conv[0] ? SW_OK : SW_ERR_NOCONV;
}

int mg_solve_batch_device(sw_mg* mg, int nb, const double2* Bl, double2* Xl, double tol,
                          sw_solve_stats* st) {
  sw_ctx* c = mg->ctx;
  sw_gauge* g = mg->g;
  cudaStream_t s = c->stream;
  SW_REQUIRE(nb >= 1 && nb <= kMaxBatch, SW_ERR_ARG, "batch of 1..64 right-hand sides");
  SW_REQUIRE(mg->mixed && !mg->fine_D, SW_ERR_ARG, "batched solves need a mixed hierarchy");
  auto t0 = std::chrono::steady_clock::now();
  batch_alloc(mg, nb);
  BatchWs& B = mg->batch;
  long N = g->N, half = N / 2;
  MgLevel& L = mg->lev[0];
  Solve S(mg, true);
  Many<1> bs;
  for (int r = 0; r < nb; ++r) {
    launch_pack(g, Bl + (long)r * N, B.bps + (long)r * N, s);
    bs.add(S.slot(0, r), B.bps + (long)r * N);
  }
  many_norm(c, N, bs, 40, c->h_many->norm);
  const double* hn = norms(c);
  std::vector<double> bn(nb), tol_abs(kMaxBatch, 0.0);
  Set all;
  for (int r = 0; r < nb; ++r) {
    bn[r] = std::sqrt(hn[r]);
    check_norm(bn[r], "right-hand side");
    tol_abs[r] = tol * bn[r];
    if (bn[r] > 0.0) all.push_back(r);
  }
  std::vector<const double2*> bt(kMaxBatch, nullptr);
  std::vector<double2*> z(kMaxBatch, nullptr);
  Many<2> odd;
  Many<3> rhs;
  for (int r = 0; r < nb; ++r) {
    // b~_e = b_e - C_eo B_o^-1 b_o
    double2* bps = B.bps + (long)r * N;
    double2* t = B.xps + (long)r * N;
    LevelWs& W = B.lv[0][r];
    odd.add(0, bps + half, t);
    rhs.add(0, bps, t, W.rhs);
    bt[r] = W.rhs;
    z[r] = W.sol;
  }
  many_block_apply(g, mg->binv, 1, 0, odd, s);
  many_hop(g, 0, -1.0, rhs, s);
  SetResult res(kMaxBatch);
  if (!all.empty())
    res = fgcr(S, 0, all, bt, z, tol_abs, false, mg->p.outer_restart, mg->p.outer_maxiter, true);
  Many<2> even, xe, xo;
  Many<3> zo, diff;
  for (int r = 0; r < nb; ++r) {
    if (bn[r] == 0.0) {
      blas_zero(c, Xl + (long)r * N, N);
      continue;
    }
    // z_o = b_o - C_oe B_e^-1 z_e ; x = B^-1 z
    double2* t = B.lex + (long)r * N;
    double2* xps = B.xps + (long)r * N;
    even.add(0, z[r], xps);  // the even half of x as well
    zo.add(0, B.bps + (long)r * N + half, xps, t + half);
    xo.add(0, t + half, xps + half);
    diff.add(S.slot(0, r), t, Bl + (long)r * N, t);
  }
  if (!all.empty()) {
    many_block_apply(g, mg->binv, 0, 0, even, s);
    many_hop(g, 1, -1.0, zo, s);
    many_block_apply(g, mg->binv, 1, 0, xo, s);
  }
  for (int r : all) {
    launch_unpack(g, B.xps + (long)r * N, Xl + (long)r * N, s);
    launch_dslash_lex(g, mg->mass, 0, Xl + (long)r * N, B.lex + (long)r * N, s);
  }
  many_sub_norm(c, N, diff, 41, c->h_many->norm);
  hn = norms(c);
  std::vector<double> rr(nb, 0.0);
  for (size_t m = 0; m < all.size(); ++m) rr[all[m]] = hn[m];
  double secs = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  bool ok = true;
  for (int r = 0; r < nb; ++r) {
    bool conv = bn[r] == 0.0 || res.conv[r];
    ok = ok && conv;
    if (!st) continue;
    sw_solve_stats& o = st[r];
    std::memset(&o, 0, sizeof(o));
    o.converged = conv ? 1 : 0;
    o.outer_iters = res.it[r];
    o.restarts = res.restarts[r];
    o.fine_applies = S.fine[r];
    o.inter_iters = S.inter_it[r];
    o.inter_solves = S.inter_solves[r];
    o.coarsest_iters = S.coarse_it[r];
    o.coarsest_solves = S.coarse_solves[r];
    o.true_resid = bn[r] > 0.0 ? std::sqrt(rr[r]) / bn[r] : 0.0;
    o.seconds = secs;
  }
  return ok ? SW_OK : SW_ERR_NOCONV;
}

int mg_batch_stall(sw_mg* mg, int nb) {
  SW_REQUIRE(nb >= 1 && nb <= kMaxBatch, SW_ERR_ARG, "batch of 1..64 right-hand sides");
  SW_REQUIRE(mg->mixed && !mg->fine_D, SW_ERR_ARG, "batched solves need a mixed hierarchy");
  batch_alloc(mg, nb);
  const int l = mg->nlev - 1;
  for (int r = 0; r < nb; ++r) blas_zero(mg->ctx, mg->batch.lv[l][r].rhs, level_len(mg, l));
  Set set;
  for (int r = 0; r < nb; ++r) set.push_back(r);
  Solve S(mg, true);
  cgne_b(S, l, set, 1);
  return SW_OK;
}

int mg_autotune_entries(int max, int* nc, int* K, int* sites, int* stages, double* us) {
  std::lock_guard<std::mutex> lk(g_tune_mutex);
  int n = 0;
  for (const auto& kv : g_tune) {
    if (n < max) {
      if (nc) nc[n] = std::get<1>(kv.first);
      if (K) K[n] = std::get<2>(kv.first);
      if (sites) sites[n] = std::get<3>(kv.first);
      if (stages) stages[n] = kv.second.stages;
      if (us) us[n] = kv.second.us_per_iter;
    }
    ++n;
  }
  return n;
}
