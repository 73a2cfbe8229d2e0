// Vector operations of the Krylov loops over the members of a batch (many.h).
//
// Each is one launch for all members (grid.y), and neighbouring steps of a
// recurrence share a pass: an update with the sum that the next step needs of
// its result.  A GCR step with k directions takes k + 3 launches where one
// per operation took 3 k + 6, and a batch as many as a single solve.  At the sizes
// of the coarse levels a launch is latency: a few microseconds, half of it the
// reduction, whose tree is therefore not made of FP64 additions (sums.cuh).
// Measured, one launch per operation and member before -> this: 16 right-hand
// sides at 128^2 221 -> 78 ms (22000 -> 1200 launches), setup and solve at 64^2
// 122 -> 27 ms, FP64 solve at 64^2 45 -> 38 ms.  What is left of a small
// operation is 2 us between launches, a chain of loads, FMAs (64 clocks each)
// and the exchange of the CTAs' parts: 2.7 us for an update, 5 with a sum.
//
// Every sum runs in an order that depends on n alone: a grid-stride slice per
// thread, aligned sums over warps and CTAs (the setup's: trees of FP64 additions, see
// mg_setup), and the last CTA to finish adds the CTAs' parts.  A member's scalars do not depend on the others of its batch.
#include "many.h"

#include "sums.cuh"

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

__device__ __forceinline__ void cadd(double2& o, double2 a, double2 v) {  // o += a v
  o.x = fma(a.x, v.x, o.x); o.x = fma(-a.y, v.y, o.x);
  o.y = fma(a.x, v.y, o.y); o.y = fma(a.y, v.x, o.y);
}
__device__ __forceinline__ double2 neg(double2 a) { return make_double2(-a.x, -a.y); }
__device__ __forceinline__ void dot(double* acc, double2 x, double2 y) {  // += conj(x) y
  acc[0] = fma(x.x, y.x, acc[0]); acc[0] = fma(x.y, y.y, acc[0]);
  acc[1] = fma(x.x, y.y, acc[1]); acc[1] = fma(-x.y, y.x, acc[1]);
}
__device__ __forceinline__ void norm(double* acc, double2 x) {
  acc[0] = fma(x.x, x.x, acc[0]); acc[0] = fma(x.y, x.y, acc[0]);
}

// An operation: K operands, R sums; coef(S, comp): component comp of its coefficient from the
// member's slots; elem: one element; store: what the sums are for.
struct NoCoef {
  __device__ double coef(const double2*, int) const { return 0.0; }
};
struct NoSums {
  template <typename V>
  __device__ void store(const V&, double2*, const double*, int*) const {}
};
struct Init : NoCoef {
  static constexpr int K = 3, R = 1;
  int s_rr;
  template <typename V>
  __device__ void elem(const V& v, long i, double2, double* acc) const {
    const double2 b = v(2)[i];
    v(0)[i] = make_double2(0.0, 0.0);
    v(1)[i] = b;
    norm(acc, b);
  }
  template <typename V>
  __device__ void store(const V&, double2* S, const double* t, int*) const { S[s_rr] = make_double2(t[0], 0.0); }
};
struct DotNorm : NoCoef {
  static constexpr int K = 2, R = 3;
  int s;
  template <typename V>
  __device__ void elem(const V& v, long i, double2, double* acc) const {
    const double2 q = v(0)[i], r = v(1)[i];
    dot(acc, q, r);
    norm(acc + 2, q);
  }
  template <typename V>
  __device__ void store(const V&, double2* S, const double* t, int*) const {
    S[s] = make_double2(t[0], t[1]);
    S[s + 1] = make_double2(t[2], 0.0);
  }
};
struct MrCoef : NoSums {
  int s;
  double om;
  __device__ double coef(const double2* S, int comp) const {
    return (comp ? S[s].y : S[s].x) / S[s + 1].x * om;
  }
};
struct MrFirst : MrCoef {
  static constexpr int K = 4, R = 0;
  template <typename V>
  __device__ void elem(const V& v, long i, double2 a, double*) const {
    double2 x = make_double2(0.0, 0.0), r = v(2)[i];
    const double2 q = v(3)[i];
    cadd(x, a, r);
    cadd(r, neg(a), q);
    v(0)[i] = x;
    v(1)[i] = r;
  }
};
struct MrLast : MrCoef {
  static constexpr int K = 5, R = 0;
  bool first;
  template <typename V>
  __device__ void elem(const V& v, long i, double2 a, double*) const {
    double2 x = first ? make_double2(0.0, 0.0) : v(1)[i];
    const double2 r = v(2)[i], x1 = v(3)[i], e = v(4)[i];
    cadd(x, a, r);
    v(0)[i] = make_double2((x1.x + e.x) + x.x, (x1.y + e.y) + x.y);
  }
};
struct Mr : MrCoef {
  static constexpr int K = 3, R = 0;
  template <typename V>
  __device__ void elem(const V& v, long i, double2 a, double*) const {
    double2 x = v(0)[i], r = v(1)[i];
    const double2 q = v(2)[i];
    cadd(x, a, r);
    cadd(r, neg(a), q);
    v(0)[i] = x;
    v(1)[i] = r;
  }
};
struct Sub : NoCoef, NoSums {
  static constexpr int K = 3, R = 0;
  template <typename V>
  __device__ void elem(const V& v, long i, double2, double*) const {
    const double2 a = v(1)[i], b = v(2)[i];
    v(0)[i] = make_double2(a.x - b.x, a.y - b.y);
  }
};
// Base of the operations whose sums are plain FP64 trees (the setup's).
struct Tree {};
struct Dot : NoCoef {
  static constexpr int K = 2, R = 2;
  int s;
  template <typename V>
  __device__ void elem(const V& v, long i, double2, double* acc) const { dot(acc, v(0)[i], v(1)[i]); }
  template <typename V>
  __device__ void store(const V&, double2* S, const double* t, int*) const { S[s] = make_double2(t[0], t[1]); }
};
struct Norm : NoCoef {
  static constexpr int K = 1, R = 1;
  int s;
  template <typename V>
  __device__ void elem(const V& v, long i, double2, double* acc) const { norm(acc, v(0)[i]); }
  template <typename V>
  __device__ void store(const V&, double2* S, const double* t, int*) const { S[s] = make_double2(t[0], 0.0); }
};
struct SetupDot : Dot, Tree {};
struct SetupNorm : Norm, Tree {};
struct Mgs {
  static constexpr int K = 5, R = 2;
  int s, s_qq;
  __device__ double coef(const double2* S, int comp) const { return comp ? -S[s].y : -S[s].x; }
  template <typename V>
  __device__ void elem(const V& v, long i, double2 a, double* acc) const {
    double2 q = v(0)[i], p = v(1)[i];
    cadd(q, a, v(2)[i]);
    cadd(p, a, v(3)[i]);
    v(0)[i] = q;
    v(1)[i] = p;
    if (v(4))
      dot(acc, v(4)[i], q);
    else
      norm(acc, q);
  }
  template <typename V>
  __device__ void store(const V& v, double2* S, const double* t, int*) const {
    S[v(4) ? s : s_qq] = make_double2(t[0], v(4) ? t[1] : 0.0);
  }
};
struct ScaleDot {
  static constexpr int K = 3, R = 2;
  int s_qq, s_a;
  __device__ double coef(const double2* S, int comp) const { return comp ? 0.0 : 1.0 / sqrt(S[s_qq].x); }
  template <typename V>
  __device__ void elem(const V& v, long i, double2 a, double* acc) const {
    double2 q = v(0)[i], p = v(1)[i];
    q.x *= a.x; q.y *= a.x;
    p.x *= a.x; p.y *= a.x;
    v(0)[i] = q;
    v(1)[i] = p;
    dot(acc, q, v(2)[i]);
  }
  template <typename V>
  __device__ void store(const V&, double2* S, const double* t, int*) const { S[s_a] = make_double2(t[0], t[1]); }
};
struct Update {
  static constexpr int K = 4, R = 1;
  int s_a, s_rr;
  __device__ double coef(const double2* S, int comp) const { return comp ? S[s_a].y : S[s_a].x; }
  template <typename V>
  __device__ void elem(const V& v, long i, double2 a, double* acc) const {
    double2 x = v(0)[i], r = v(1)[i];
    cadd(x, a, v(2)[i]);
    cadd(r, neg(a), v(3)[i]);
    v(0)[i] = x;
    v(1)[i] = r;
    norm(acc, r);
  }
  template <typename V>
  __device__ void store(const V&, double2* S, const double* t, int*) const { S[s_rr] = make_double2(t[0], 0.0); }
};
struct SubNorm : NoCoef {
  static constexpr int K = 3, R = 1;
  int s;
  template <typename V>
  __device__ void elem(const V& v, long i, double2, double* acc) const {
    const double2 a = v(1)[i], b = v(2)[i];
    const double2 o = make_double2(a.x - b.x, a.y - b.y);
    v(0)[i] = o;
    norm(acc, o);
  }
  template <typename V>
  __device__ void store(const V&, double2* S, const double* t, int*) const { S[s] = make_double2(t[0], 0.0); }
};
struct Copy : NoCoef, NoSums {
  static constexpr int K = 2, R = 0;
  template <typename V>
  __device__ void elem(const V& v, long i, double2, double*) const { v(0)[i] = v(1)[i]; }
};
struct CgStart : NoCoef, Tree {
  static constexpr int K = 4, R = 1;
  int s_rr, s_stop, maxit;
  double tol;
  template <typename V>
  __device__ void elem(const V& v, long i, double2, double* acc) const {
    const double2 b = make_double2(0.0 - v(3)[i].x, 0.0 - v(3)[i].y);
    v(0)[i] = make_double2(0.0, 0.0);
    v(1)[i] = b;
    v(2)[i] = b;
    norm(acc, b);
  }
  template <typename V>
  __device__ void store(const V&, double2* S, const double* t, int* ctl) const {
    const double rn = sqrt(t[0]), stop = tol * rn;
    S[s_rr] = make_double2(t[0], 0.0);
    S[s_stop] = make_double2(stop, 0.0);
    ctl[1] = 0;
    ctl[2] = isfinite(rn) ? 0 : 1;
    ctl[0] = maxit <= 0 || !(rn > stop);
  }
};
struct CgStep : Tree {
  static constexpr int K = 4, R = 1;
  int s_rr, s_pq, s_new, s_stop, maxit;
  __device__ double coef(const double2* S, int comp) const { return comp ? 0.0 : S[s_rr].x / S[s_pq].x; }
  template <typename V>
  __device__ void elem(const V& v, long i, double2 a, double* acc) const {
    double2 x = v(0)[i], r = v(1)[i];
    const double2 p = v(2)[i], q = v(3)[i];
    x.x = fma(a.x, p.x, x.x); x.y = fma(a.x, p.y, x.y);
    r.x = fma(-a.x, q.x, r.x); r.y = fma(-a.x, q.y, r.y);
    v(0)[i] = x;
    v(1)[i] = r;
    norm(acc, r);
  }
  template <typename V>
  __device__ void store(const V&, double2* S, const double* t, int* ctl) const {
    S[s_new] = make_double2(t[0], 0.0);
    const double rn = sqrt(t[0]);
    const int k = ++ctl[1];
    if (!isfinite(rn)) ctl[2] = 1;
    if (k >= maxit || !(rn > S[s_stop].x)) ctl[0] = 1;
  }
};
struct Xpay : NoSums {
  static constexpr int K = 2, R = 0;
  int s_new, s_old;
  __device__ double coef(const double2* S, int comp) const { return comp ? 0.0 : S[s_new].x / S[s_old].x; }
  template <typename V>
  __device__ void elem(const V& v, long i, double2 a, double*) const {
    const double2 p = v(0)[i], r = v(1)[i];
    v(0)[i] = make_double2(fma(a.x, p.x, r.x), fma(a.x, p.y, r.y));
  }
};
struct Add : NoCoef, NoSums {
  static constexpr int K = 2, R = 0;
  template <typename V>
  __device__ void elem(const V& v, long i, double2, double*) const {
    const double2 x = v(0)[i], y = v(1)[i];
    v(0)[i] = make_double2(x.x + y.x, x.y + y.y);
  }
};
struct Project : NoSums {
  static constexpr int K = 2, R = 0;
  int s;
  __device__ double coef(const double2* S, int comp) const { return comp ? -S[s].y : -S[s].x; }
  template <typename V>
  __device__ void elem(const V& v, long i, double2 a, double*) const {
    double2 x = v(0)[i];
    cadd(x, a, v(1)[i]);
    v(0)[i] = x;
  }
};
struct Normalise : NoSums {
  static constexpr int K = 1, R = 0;
  int s;
  __device__ double coef(const double2* S, int comp) const { return comp ? 0.0 : 1.0 / sqrt(S[s].x); }
  template <typename V>
  __device__ void elem(const V& v, long i, double2 a, double*) const {
    const double2 x = v(0)[i];
    v(0)[i] = make_double2(a.x * x.x, a.x * x.y);
  }
};

template <typename Op, int W>
__global__ void __launch_bounds__(kThreads) k_many(Op op, Pack<Op::K, W> v, long n, double2* slots,
                                                   double* partials, unsigned* counters,
                                                   double* host, int* ctl) {
  __shared__ double cf[2];
  const int m = blockIdx.y;
  after_previous();
  if (ctl) {
    ctl += 4 * m;
    // a kernel that sets the flag does so in its last CTA, after all of them have read it
    if (!std::is_same<Op, CgStart>::value && *(volatile int*)ctl) return;
  }
  double2* S = slots + v.slot[m];
  if (threadIdx.x < 2) cf[threadIdx.x] = op.coef(S, threadIdx.x);
  __syncthreads();
  const double2 a = make_double2(cf[0], cf[1]);
  const auto get = [&](int k) { return v.v[k][m]; };
  constexpr int R = Op::R;
  double acc[R + 1] = {0.0};
  for (long i = (long)blockIdx.x * kThreads + threadIdx.x; i < n; i += (long)gridDim.x * kThreads)
    op.elem(get, i, a, acc);
  if constexpr (R > 0) {
    constexpr bool tree = std::is_base_of<Tree, Op>::value;
    using Part = typename std::conditional<tree, double, swsum::Aligned>::type;
    __shared__ Part part[R][kWarps];
    __shared__ double sum[R];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const auto cta_sums = [&]() {  // of acc, to sum
      if constexpr (tree) {
        const auto warp = [](double v) {
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          return v;
        };
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const double t = warp(acc[r]);
          if (lane == 0) part[r][w] = t;
        }
        __syncthreads();
        if (w == 0)
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const double t = warp(lane < kWarps ? part[r][lane] : 0.0);
            if (lane == 0) sum[r] = t;
          }
      } else {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const swsum::Aligned t = swsum::warp_sum(acc[r]);
          if (lane == 0) part[r][w] = t;
        }
        __syncthreads();
        if (threadIdx.x < R) sum[threadIdx.x] = swsum::total<kWarps>(part[threadIdx.x]);
      }
      __syncthreads();
    };
    cta_sums();
    if (gridDim.x > 1) {
      double* mine = partials + (long)m * kManyBlocks * 4;
      if (threadIdx.x == 0) {
#pragma unroll
        for (int r = 0; r < R; ++r) mine[4 * blockIdx.x + r] = sum[r];
        __threadfence();
        last = atomicAdd(counters + m, 1u) == gridDim.x - 1;
      }
      __syncthreads();
      if (!last) return;
      __threadfence();
#pragma unroll
      for (int r = 0; r < R; ++r) {
        acc[r] = 0.0;
        for (int j = threadIdx.x; j < (int)gridDim.x; j += kThreads) acc[r] += __ldcg(mine + 4 * j + r);
      }
      cta_sums();
    }
    if (threadIdx.x == 0) {
      double t[R];
#pragma unroll
      for (int r = 0; r < R; ++r) t[r] = sum[r];
      op.store(get, S, t, ctl);
      if (host) host[m] = t[0];
      counters[m] = 0u;
    }
  }
}

// A sum's grid is capped, so that the last CTA adds three parts a thread at most; up to 512
// elements one CTA does without the second stage.
template <typename Op>
void launch(sw_ctx* c, long n, const Op& op, const Many<Op::K>& v, double* host = nullptr,
            int* ctl = nullptr) {
  if (v.n == 0 || n <= 0) return;
  long grid = (n + kThreads - 1) / kThreads;
  constexpr bool tree = std::is_base_of<Tree, Op>::value;  // slices of these: never change
  if (Op::R > 0 && !tree && n <= 2 * kThreads) grid = 1;
  const long most = tree ? kReduceBlocks : kManyBlocks;
  if (Op::R > 0 && grid > most) grid = most;
  with_width(v.n, [&](auto w) {
    constexpr int W = decltype(w)::value;
    launch_early(k_many<Op, W>, dim3((unsigned)grid, v.n), kThreads, 0, c->stream, op,
                 Pack<Op::K, W>(v), n, c->slots, c->many_partials, c->many_counters, host, ctl);
  });
}

}  // namespace

void many_init(sw_ctx* c, long n, const Many<3>& v, int s_rr, double* host) {
  launch(c, n, Init{{}, s_rr}, v, host);
}
void many_dot_norm(sw_ctx* c, long n, const Many<2>& v, int s) { launch(c, n, DotNorm{{}, s}, v); }
void many_mr_first(sw_ctx* c, long n, const Many<4>& v, int s, double om) {
  launch(c, n, MrFirst{{{}, s, om}}, v);
}
void many_mr(sw_ctx* c, long n, const Many<3>& v, int s, double om) {
  launch(c, n, Mr{{{}, s, om}}, v);
}
void many_mr_last(sw_ctx* c, long n, const Many<5>& v, int s, double om, bool first) {
  launch(c, n, MrLast{{{}, s, om}, first}, v);
}
void many_sub(sw_ctx* c, long n, const Many<3>& v) { launch(c, n, Sub{}, v); }
void many_sub_norm(sw_ctx* c, long n, const Many<3>& v, int s, double* host) {
  launch(c, n, SubNorm{{}, s}, v, host);
}
void many_dot(sw_ctx* c, long n, const Many<2>& v, int s) { launch(c, n, Dot{{}, s}, v); }
void many_norm(sw_ctx* c, long n, const Many<1>& v, int s, double* host) {
  launch(c, n, Norm{{}, s}, v, host);
}
void many_mgs(sw_ctx* c, long n, const Many<5>& v, int s, int s_qq) {
  launch(c, n, Mgs{s, s_qq}, v);
}
void many_scale_dot(sw_ctx* c, long n, const Many<3>& v, int s_qq, int s_a) {
  launch(c, n, ScaleDot{s_qq, s_a}, v);
}
void many_update(sw_ctx* c, long n, const Many<4>& v, int s_a, int s_rr, double* host) {
  launch(c, n, Update{s_a, s_rr}, v, host);
}
void many_setup_dot(sw_ctx* c, long n, const Many<2>& v, int s, const int* ctl) {
  launch(c, n, SetupDot{{{}, s}}, v, nullptr, const_cast<int*>(ctl));
}
void many_setup_norm(sw_ctx* c, long n, const Many<1>& v, int s, double* host) {
  launch(c, n, SetupNorm{{{}, s}}, v, host);
}
void many_copy(sw_ctx* c, long n, const Many<2>& v) { launch(c, n, Copy{}, v); }
void many_add(sw_ctx* c, long n, const Many<2>& v) { launch(c, n, Add{}, v); }
void many_project(sw_ctx* c, long n, const Many<2>& v, int s) { launch(c, n, Project{{}, s}, v); }
void many_normalise(sw_ctx* c, long n, const Many<1>& v, int s) { launch(c, n, Normalise{{}, s}, v); }
void many_cg_start(sw_ctx* c, long n, const Many<4>& v, int s_rr, int s_stop, double tol, int maxit,
                   int* ctl) {
  launch(c, n, CgStart{{}, {}, s_rr, s_stop, maxit, tol}, v, nullptr, ctl);
}
void many_cg_step(sw_ctx* c, long n, const Many<4>& v, int s_rr, int s_pq, int s_new, int s_stop,
                  int maxit, int* ctl) {
  launch(c, n, CgStep{{}, s_rr, s_pq, s_new, s_stop, maxit}, v, nullptr, ctl);
}
void many_xpay(sw_ctx* c, long n, const Many<2>& v, int s_new, int s_old, const int* ctl) {
  launch(c, n, Xpay{{}, s_new, s_old}, v, nullptr, const_cast<int*>(ctl));
}
