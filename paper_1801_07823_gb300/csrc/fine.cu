// Fine-level kernels: staggered Dslash (Eq. staggeredD), Kaehler-Dirac block
// inverse B^-1 (Sec. II.A, Eq. localblock), the block hopping term C, and the
// compositions A = D B^-1 = I + C B^-1 (Eq. defA), A^dag and the Schur
// operator I - A_eo A_oe (Table kcycle).
//
// Links are stored pre-multiplied as W_mu(s) = eta_mu(s) U_mu(s) / 2.  In 2D
// eta_mu(s - mu) = eta_mu(s) (eta_1 depends on x0 only), so the backward hop of
// Eq. staggeredD is -conj(W_mu(s - mu)) x(s - mu).
#include "intmul.cuh"
#include "many.h"

namespace {

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ void cfma(double2& acc, double2 a, double2 b) {  // acc += a b
  acc.x = fma(a.x, b.x, acc.x);
  acc.x = fma(-a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y);
  acc.y = fma(a.y, b.x, acc.y);
}
__device__ __forceinline__ double2 minus_conj(double2 w) { return make_double2(-w.x, w.y); }
__device__ __forceinline__ bool all_zero(double2 a, double2 b, double2 c, double2 d) {
  return a.x == 0.0 && a.y == 0.0 && b.x == 0.0 && b.y == 0.0 && c.x == 0.0 && c.y == 0.0 &&
         d.x == 0.0 && d.y == 0.0;
}

// ---------------------------------------------------------------------------
// Lexicographic Dslash: out(s) = m in(s) + sg * sum_mu [W_mu(s) in(s+mu) - conj(W_mu(s-mu)) in(s-mu)]
// sg = +1 for D, -1 for D^dag (D - m is anti-Hermitian, Sec. II).
// One thread per site; consecutive threads take consecutive x0, so every
// load of in and W is coalesced; neighbour values are re-read from L1/L2.
template <typename C2>
struct Hops {  // a site's neighbours and their links
  C2 xs, a, b, c, d, w0, w1, w0m, w1m;
  long s;
};
template <typename C2>
__device__ __forceinline__ Hops<C2> load_hops(const C2* __restrict__ in, const C2* __restrict__ W,
                                              int x0, int x1, int L0, int L1) {
  const long N = (long)L0 * L1, row = (long)x1 * L0;
  const long sm0 = row + (x0 == 0 ? L0 - 1 : x0 - 1);
  const long sm1 = (long)(x1 == 0 ? L1 - 1 : x1 - 1) * L0 + x0;
  Hops<C2> h;
  h.s = row + x0;
  h.xs = __ldg(in + h.s);
  h.a = __ldg(in + row + (x0 + 1 == L0 ? 0 : x0 + 1));
  h.b = __ldg(in + sm0);
  h.c = __ldg(in + (long)(x1 + 1 == L1 ? 0 : x1 + 1) * L0 + x0);
  h.d = __ldg(in + sm1);
  h.w0 = __ldg(W + h.s);
  h.w1 = __ldg(W + N + h.s);
  h.w0m = __ldg(W + sm0);
  h.w1m = __ldg(W + N + sm1);
  return h;
}
template <typename C2, typename R, bool DAG>
__device__ __forceinline__ C2 sum_hops(const Hops<C2>& h, R mass) {
  R hx = mass * h.xs.x, hy = mass * h.xs.y;
  auto fwd = [&](C2 w, C2 v) {  // +- w v
    if (DAG) { w.x = -w.x; w.y = -w.y; }
    hx = fma(w.x, v.x, hx); hx = fma(-w.y, v.y, hx);
    hy = fma(w.x, v.y, hy); hy = fma(w.y, v.x, hy);
  };
  auto bwd = [&](C2 w, C2 v) {  // -+ conj(w) v
    if (DAG) { w.x = -w.x; w.y = -w.y; }
    hx = fma(-w.x, v.x, hx); hx = fma(-w.y, v.y, hx);
    hy = fma(-w.x, v.y, hy); hy = fma(w.y, v.x, hy);
  };
  fwd(h.w0, h.a);
  fwd(h.w1, h.c);
  bwd(h.w0m, h.b);
  bwd(h.w1m, h.d);
  C2 o;
  o.x = hx;
  o.y = hy;
  return o;
}
// FP32: bound by HBM.
template <bool DAG>
__global__ void __launch_bounds__(256) k_dslash_lex32(const float2* __restrict__ in,
                                                      float2* __restrict__ out,
                                                      const float2* __restrict__ W, float mass,
                                                      int L0, int L1) {
  const int x0 = blockIdx.x * blockDim.x + threadIdx.x;
  if (x0 >= L0) return;
  const Hops<float2> h = load_hops(in, W, x0, blockIdx.y, L0, L1);
  out[h.s] = sum_hops<float2, float, DAG>(h, mass);
}
// FP64: of the eight warps of a CTA two belong to each quarter of the SM; one of the two
// works in FP64 (18 operations per site, two per clock and SM) and the other forms its hops in
// integers (intmul.cuh) with one FMA per component for the mass term, so that both
// pipes are busy.  The warps change places from row to row, for lattices that fill half a
// CTA.  2044 x 2052, of 39.6 us at the HBM rate: all in FP64 132.2 us, all in integers 114.9
// (about 350 integer operations per site, 64 per clock and SM), split 88.1.  32 x 32 is one
// launch either way (6.5 us).  Relative error 1.3e-16 against 1.5e-16 in FP64 alone.
template <bool DAG>
__global__ void __launch_bounds__(256) k_dslash_lex(const double2* __restrict__ in,
                                                    double2* __restrict__ out,
                                                    const double2* __restrict__ W, double mass,
                                                    int L0, int L1) {
  using namespace swint;
  const int x0 = blockIdx.x * blockDim.x + threadIdx.x;
  if (x0 >= L0) return;
  const Hops<double2> h = load_hops(in, W, x0, blockIdx.y, L0, L1);
  const unsigned mv = max(max(magnitude(h.a), magnitude(h.b)), max(magnitude(h.c), magnitude(h.d)));
  const unsigned mw =
      max(max(magnitude(h.w0), magnitude(h.w1)), max(magnitude(h.w0m), magnitude(h.w1m)));
  const int e = (int)(mv >> 20);
  const bool ints = (((threadIdx.x >> 7) ^ blockIdx.y) & 1) && link_usable(mw);
  if (ints && usable(e)) {
    Csum t;
    t.add(num(h.w0, kLinkExp), num(h.a, e));
    t.add(num(h.w1, kLinkExp), num(h.c, e));
    t.add(num(minus_conj(h.w0m), kLinkExp), num(h.b, e));
    t.add(num(minus_conj(h.w1m), kLinkExp), num(h.d, e));
    const double2 v = t.value(kLinkExp, e);
    out[h.s] = make_double2(fma(mass, h.xs.x, DAG ? -v.x : v.x), fma(mass, h.xs.y, DAG ? -v.y : v.y));
  } else if (ints && mv == 0 && all_zero(h.a, h.b, h.c, h.d)) {
    out[h.s] = make_double2(mass * h.xs.x, mass * h.xs.y);  // a sparse source
  } else {
    out[h.s] = sum_hops<double2, double, DAG>(h, mass);
  }
}

// ---------------------------------------------------------------------------
__global__ void k_pack(const double2* __restrict__ lex, double2* __restrict__ ps, int L0, int L1) {
  int N = L0 * L1;
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= N) return;
  int x0 = s % L0, x1 = s / L0;
  ps[ps_index(x0, x1, L0, N)] = lex[s];
}
__global__ void k_unpack(const double2* __restrict__ ps, double2* __restrict__ lex, int L0, int L1) {
  int N = L0 * L1;
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= N) return;
  int x0 = s % L0, x1 = s / L0;
  lex[s] = ps[ps_index(x0, x1, L0, N)];
}

// ---------------------------------------------------------------------------
// B^-1 per KD block.  B is D restricted to the 2x2 block with corner at even
// coordinates, mass included (Sec. II.A).  Site k of the block sits at
// (2X0 + (k & 1), 2X1 + (k >> 1)).  For direction mu the partner inside the
// block of site k is k ^ (1 << mu): a forward hop (coefficient W_mu(s)) when
// x_mu is even, a backward hop (coefficient -conj(W_mu(s - mu))) when odd.
// Inverted by Gauss-Jordan elimination with partial pivoting in FP64.
__global__ void k_binv_build(const double2* __restrict__ Wps, double mass, double hop_scale,
                             double2* __restrict__ binv, int L0, int L1) {
  int N = L0 * L1;
  int nb = N >> 2;
  int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nb) return;
  double2 M[4][4], I[4][4];
  for (int i = 0; i < 4; ++i)
    for (int j = 0; j < 4; ++j) {
      M[i][j] = make_double2(i == j ? mass : 0.0, 0.0);
      I[i][j] = make_double2(i == j ? 1.0 : 0.0, 0.0);
    }
  int x0b, x1b;
  ps_coords(4 * b, L0, N, x0b, x1b);  // site k = 0 of the block
  for (int k = 0; k < 4; ++k) {
    int x0 = x0b + (k & 1), x1 = x1b + (k >> 1);
    for (int mu = 0; mu < 2; ++mu) {
      int kp = k ^ (1 << mu);
      int xm = mu == 0 ? x0 : x1;
      if ((xm & 1) == 0) {
        double2 w = Wps[mu * N + 4 * b + k];
        M[k][kp] = make_double2(hop_scale * w.x, hop_scale * w.y);
      } else {
        double2 w = Wps[mu * N + 4 * b + kp];  // W_mu(s - mu), s - mu is site kp
        M[k][kp] = make_double2(-hop_scale * w.x, hop_scale * w.y);
      }
    }
  }
  for (int c = 0; c < 4; ++c) {
    int p = c;
    double best = hypot(M[c][c].x, M[c][c].y);
    for (int r = c + 1; r < 4; ++r) {
      double v = hypot(M[r][c].x, M[r][c].y);
      if (v > best) { best = v; p = r; }
    }
    if (p != c)
      for (int j = 0; j < 4; ++j) {
        double2 t = M[c][j]; M[c][j] = M[p][j]; M[p][j] = t;
        t = I[c][j]; I[c][j] = I[p][j]; I[p][j] = t;
      }
    double2 piv = M[c][c];
    double den = piv.x * piv.x + piv.y * piv.y;
    double2 inv = make_double2(piv.x / den, -piv.y / den);
    for (int j = 0; j < 4; ++j) { M[c][j] = cmul(M[c][j], inv); I[c][j] = cmul(I[c][j], inv); }
    for (int r = 0; r < 4; ++r) {
      if (r == c) continue;
      double2 f = M[r][c];
      for (int j = 0; j < 4; ++j) {
        double2 a = cmul(f, M[c][j]), e = cmul(f, I[c][j]);
        M[r][j].x -= a.x; M[r][j].y -= a.y;
        I[r][j].x -= e.x; I[r][j].y -= e.y;
      }
    }
  }
  for (int i = 0; i < 4; ++i)
    for (int j = 0; j < 4; ++j) binv[16 * b + 4 * i + j] = I[i][j];
}

// Row i of a block's B^-1 (dagger: of its adjoint) times its vector.  Four neighbouring lanes
// hold a block, lane i its site i: with a thread per block a 64^2 lattice was 16 warps,
// each of which waited for 56 FMAs of 64 clocks, and every load of the table touched 32 lines.
// The diagonal is real: B - m is anti-Hermitian and couples the two site parities only.
__device__ __forceinline__ double2 block_row(const double2* __restrict__ m, int i, double2 u,
                                             bool dagger) {
  const unsigned quad = 0xfu << (threadIdx.x & 28);
  const double d = m[5 * i].x;
  double2 acc = make_double2(d * u.x, d * u.y);
#pragma unroll
  for (int k = 1; k < 4; ++k) {
    const int j = i ^ k;
    const double2 v = make_double2(__shfl_xor_sync(quad, u.x, k), __shfl_xor_sync(quad, u.y, k));
    double2 a = m[dagger ? 4 * j + i : 4 * i + j];
    if (dagger) a.y = -a.y;
    cfma(acc, a, v);
  }
  return acc;
}
// The same with all four products added in the order of the columns, the diagonal as a complex
// number.  The kernels on parity-split fields use this one: they relax the null vectors, whose
// values depend on every rounding (mg_setup), so their order of operations is fixed.
__device__ __forceinline__ double2 block_row_ordered(const double2* __restrict__ m, int i,
                                                     double2 u, bool dagger) {
  const unsigned quad = 0xfu << (threadIdx.x & 28);
  double2 acc = make_double2(0.0, 0.0);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const double2 v = make_double2(__shfl_sync(quad, u.x, j, 4), __shfl_sync(quad, u.y, j, 4));
    double2 a = m[dagger ? 4 * j + i : 4 * i + j];
    if (dagger) a.y = -a.y;
    cfma(acc, a, v);
  }
  return acc;
}
// out = M in (or M^dag in) on nblk KD blocks, a thread per site; one member of a batch per
// blockIdx.y.
template <int W>
__global__ void k_block_apply(const double2* __restrict__ M, Pack<2, W> io, int nblk, int dagger,
                              const int* ctl) {
  after_previous();
  if (ctl && ctl[4 * blockIdx.y]) return;
  const double2* in = io.v[0][blockIdx.y];
  double2* out = io.v[1][blockIdx.y];
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 4 * nblk) return;
  out[t] = block_row_ordered(M + 16 * (long)(t >> 2), t & 3, in[t], dagger);
}

// (C in)(s) for a site s of parity half par: the two hops of s that leave its
// KD block.  in is the opposite parity half.
__device__ __forceinline__ double2 hop_out(const double2* __restrict__ Wps,
                                           const double2* in, int f, int L0, int L1,
                                           int N) {
  int x0, x1;
  ps_coords(f, L0, N, x0, x1);
  int half = N >> 1;
  double2 acc = make_double2(0.0, 0.0);
  // direction 0
  if (x0 & 1) {  // forward neighbour is in the next block
    int t = ps_index(x0 + 1 == L0 ? 0 : x0 + 1, x1, L0, N);
    cfma(acc, Wps[f], in[t < half ? t : t - half]);
  } else {
    int t = ps_index(x0 == 0 ? L0 - 1 : x0 - 1, x1, L0, N);
    double2 w = Wps[t];
    double2 v = in[t < half ? t : t - half];
    acc.x -= w.x * v.x + w.y * v.y;
    acc.y -= w.x * v.y - w.y * v.x;
  }
  // direction 1
  if (x1 & 1) {
    int t = ps_index(x0, x1 + 1 == L1 ? 0 : x1 + 1, L0, N);
    cfma(acc, Wps[N + f], in[t < half ? t : t - half]);
  } else {
    int t = ps_index(x0, x1 == 0 ? L1 - 1 : x1 - 1, L0, N);
    double2 w = Wps[N + t];
    double2 v = in[t < half ? t : t - half];
    acc.x -= w.x * v.x + w.y * v.y;
    acc.y -= w.x * v.y - w.y * v.x;
  }
  return acc;
}

// out_p = src_p + sign C in_{1-p} on parity half p = par, or (par < 0) on both halves of
// full vectors; operands (src or null, in, out) of one member of a batch per blockIdx.y.
template <int W>
__global__ void k_hop(const double2* __restrict__ Wps, int par, double sign, Pack<3, W> io, int L0,
                      int L1, const int* ctl) {
  after_previous();
  if (ctl && ctl[4 * blockIdx.y]) return;
  const double2* src = io.v[0][blockIdx.y];
  const double2* in = io.v[1][blockIdx.y];
  double2* out = io.v[2][blockIdx.y];
  int N = L0 * L1, half = N >> 1;
  int h = blockIdx.x * blockDim.x + threadIdx.x;
  if (h >= (par < 0 ? N : half)) return;
  if (par < 0 && h < half) in += half;
  double2 c = hop_out(Wps, in, par < 0 ? h : par * half + h, L0, L1, N);
  double2 o = src ? src[h] : make_double2(0.0, 0.0);
  o.x = fma(sign, c.x, o.x);
  o.y = fma(sign, c.y, o.y);
  out[h] = o;
}

// out_p = src_p + sign M C in_{1-p} (M^dag: dagger), as above.  M: B^-1 of all blocks.
template <int W>
__global__ void k_hop_block(const double2* __restrict__ Wps, const double2* __restrict__ M,
                            int par, int dagger, double sign, Pack<3, W> io, int L0, int L1,
                            const int* ctl) {
  after_previous();
  if (ctl && ctl[4 * blockIdx.y]) return;
  const double2* src = io.v[0][blockIdx.y];
  const double2* in = io.v[1][blockIdx.y];
  double2* out = io.v[2][blockIdx.y];
  const int N = L0 * L1, half = N >> 1;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (par < 0 ? N : half)) return;
  if (par < 0 && t < half) in += half;
  const int f = par < 0 ? t : par * half + t;
  const double2 u = hop_out(Wps, in, f, L0, L1, N);
  const double2 acc = block_row_ordered(M + 16 * (long)(f >> 2), f & 3, u, dagger);
  double2 o = src ? src[t] : make_double2(0.0, 0.0);
  o.x = fma(sign, acc.x, o.x);
  o.y = fma(sign, acc.y, o.y);
  out[t] = o;
}

// Long links of the Naik term (Sec. II.A, Eq. freehisq, gauged with the
// product of the three links of the path): W3_mu(s) = c3 eta_mu(s) / 2 *
// U_mu(s) U_mu(s+mu) U_mu(s+2mu), from W_mu = eta_mu U_mu / 2 (lexicographic).
__global__ void k_long_links(const double2* __restrict__ W, double c3, double2* __restrict__ W3,
                             int L0, int L1) {
  long N = (long)L0 * L1;
  long s = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= N) return;
  int x0 = (int)(s % L0), x1 = (int)(s / L0);
  for (int mu = 0; mu < 2; ++mu) {
    long s1 = mu == 0 ? (long)x1 * L0 + (x0 + 1) % L0 : (long)((x1 + 1) % L1) * L0 + x0;
    long s2 = mu == 0 ? (long)x1 * L0 + (x0 + 2) % L0 : (long)((x1 + 2) % L1) * L0 + x0;
    double2 a = W[mu * N + s], b = W[mu * N + s1], c = W[mu * N + s2];
    // each W carries eta / 2 with the same eta along the path (eta_1 depends
    // on x0 only): U U U = 8 a b c / eta^3 = 8 a b c eta, so
    // W3 = c3 (eta / 2) U U U = 4 c3 a b c
    double2 abc = cmul(cmul(a, b), c);
    W3[mu * N + s] = make_double2(4.0 * c3 * abc.x, 4.0 * c3 * abc.y);
  }
}

// Naik-improved D: out(s) = m in(s) + sum_mu [c1 (W in(s+mu) - W(s-mu)^* in(s-mu))
//                                            + W3 in(s+3mu) - W3(s-3mu)^* in(s-3mu)]
__global__ void k_dslash_naik_lex(const double2* __restrict__ in, double2* __restrict__ out,
                                  const double2* __restrict__ W, const double2* __restrict__ W3,
                                  double mass, double c1, int L0, int L1) {
  int x0 = blockIdx.x * blockDim.x + threadIdx.x;
  int x1 = blockIdx.y;
  if (x0 >= L0) return;
  long N = (long)L0 * L1;
  long s = (long)x1 * L0 + x0;
  double2 h1 = make_double2(0.0, 0.0), h3 = make_double2(0.0, 0.0);
  for (int mu = 0; mu < 2; ++mu) {
    auto site = [&](int k) {
      return mu == 0 ? (long)x1 * L0 + ((x0 + k) % L0 + L0) % L0
                     : (long)(((x1 + k) % L1 + L1) % L1) * L0 + x0;
    };
    long f1 = site(1), b1 = site(-1), f3 = site(3), b3 = site(-3);
    cfma(h1, W[mu * N + s], in[f1]);
    double2 w = W[mu * N + b1], v = in[b1];
    h1.x -= w.x * v.x + w.y * v.y;
    h1.y -= w.x * v.y - w.y * v.x;
    cfma(h3, W3[mu * N + s], in[f3]);
    w = W3[mu * N + b3];
    v = in[b3];
    h3.x -= w.x * v.x + w.y * v.y;
    h3.y -= w.x * v.y - w.y * v.x;
  }
  double2 xs = in[s];
  out[s] = make_double2(mass * xs.x + c1 * h1.x + h3.x, mass * xs.y + c1 * h1.y + h3.y);
}

// D (sg = +1) or D^dag (sg = -1) on a full parity-split vector:
// out(f) = m in(f) + sg sum_mu [W_mu(s) in(s+mu) - conj(W_mu(s-mu)) in(s-mu)].
__global__ void k_dslash_ps(const double2* __restrict__ Wps, double mass, double sg,
                            const double2* __restrict__ in, double2* __restrict__ out, int L0,
                            int L1) {
  int N = L0 * L1;
  int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= N) return;
  int x0, x1;
  ps_coords(f, L0, N, x0, x1);
  int xp0 = x0 + 1 == L0 ? 0 : x0 + 1, xm0 = x0 == 0 ? L0 - 1 : x0 - 1;
  int xp1 = x1 + 1 == L1 ? 0 : x1 + 1, xm1 = x1 == 0 ? L1 - 1 : x1 - 1;
  int fp0 = ps_index(xp0, x1, L0, N), fm0 = ps_index(xm0, x1, L0, N);
  int fp1 = ps_index(x0, xp1, L0, N), fm1 = ps_index(x0, xm1, L0, N);
  double2 h = make_double2(0.0, 0.0);
  cfma(h, Wps[f], in[fp0]);
  cfma(h, Wps[N + f], in[fp1]);
  double2 w = Wps[fm0], v = in[fm0];
  h.x -= w.x * v.x + w.y * v.y;
  h.y -= w.x * v.y - w.y * v.x;
  w = Wps[N + fm1];
  v = in[fm1];
  h.x -= w.x * v.x + w.y * v.y;
  h.y -= w.x * v.y - w.y * v.x;
  double2 xs = in[f];
  out[f] = make_double2(fma(sg, h.x, mass * xs.x), fma(sg, h.y, mass * xs.y));
}

// ---------------------------------------------------------------------------
// KD operators on lexicographic fields, for callers that hand over fields in
// that order: no packing passes, and no division in an index (row of KD blocks
// = blockIdx.y).  One thread per site, a block in four neighbouring lanes; its
// sites are 32-byte pieces of two rows, whole sectors.  Bound by the FP64 pipe
// (S: 176 FMAs per pair of blocks, 37 us at 1036 x 1012).  S there: 63.5 us (a thread
// per block: 72.1, whose one wave of warps first waited for all loads and then for the FP64
// pipe; packing passes and operators on halves: 97.8).
struct KdSite {
  int x0, x1;  // of the site
  int j;       // its place in the block
  long b;      // the block's index in the B^-1 table (parity-split)
  long s;      // x0 + L0 x1
};
// Sites of the blocks of parity `par`, or (par < 0) of all, in row X1 of blocks.
__device__ __forceinline__ bool kd_site(int L0, int L1, int par, int X1, KdSite& k) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x, i = t >> 2;
  const int X0 = par < 0 ? i : 2 * i + ((X1 + par) & 1);
  if (X0 >= L0 / 2) return false;
  k.j = t & 3;
  k.x0 = 2 * X0 + (k.j & 1);
  k.x1 = 2 * X1 + (k.j >> 1);
  k.b = (long)((X0 + X1) & 1) * ((long)L0 * L1 / 8) + (long)X1 * (L0 >> 2) + (X0 >> 1);
  k.s = (long)k.x1 * L0 + k.x0;
  return true;
}
// C in at a site: the two hops that leave its block, forward from an odd coordinate.
__device__ __forceinline__ double2 kd_hop(const double2* __restrict__ W, const double2* in,
                                          const KdSite& k, int L0, int L1) {
  const long N = (long)L0 * L1;
  const bool f0 = k.j & 1, f1 = k.j >> 1;
  const long t0 = (long)k.x1 * L0 + (f0 ? (k.x0 + 1 == L0 ? 0 : k.x0 + 1) : (k.x0 == 0 ? L0 - 1 : k.x0 - 1));
  const long t1 = (long)(f1 ? (k.x1 + 1 == L1 ? 0 : k.x1 + 1) : (k.x1 == 0 ? L1 - 1 : k.x1 - 1)) * L0 + k.x0;
  const double2 w = W[f0 ? k.s : t0], z = W[N + (f1 ? k.s : t1)];
  double2 acc = make_double2(0.0, 0.0);
  cfma(acc, f0 ? w : minus_conj(w), in[t0]);
  cfma(acc, f1 ? z : minus_conj(z), in[t1]);
  return acc;
}
// out = B^-1 in on the blocks of parity par (all: par < 0).
__global__ void __launch_bounds__(128) k_kd_block(const double2* __restrict__ binv, int par,
                                                  const double2* __restrict__ in,
                                                  double2* __restrict__ out, int L0, int L1) {
  KdSite k;
  for (int X1 = blockIdx.y; X1 < L1 / 2; X1 += gridDim.y) {
    if (!kd_site(L0, L1, par, X1, k)) return;
    out[k.s] = block_row(binv + 16 * k.b, k.j, in[k.s], false);
  }
}
// out = M C in (DAG: in - M^dag C in) on the blocks of parity par (all: par < 0), M = B^-1.
// in and out may be one field where their blocks differ.
template <bool DAG>
__global__ void __launch_bounds__(128) k_kd_hop_block(const double2* __restrict__ W,
                                                      const double2* __restrict__ binv, int par,
                                                      const double2* in, double2* out, int L0,
                                                      int L1) {
  KdSite k;
  for (int X1 = blockIdx.y; X1 < L1 / 2; X1 += gridDim.y) {
    if (!kd_site(L0, L1, par, X1, k)) return;
    const double2 v = block_row(binv + 16 * k.b, k.j, kd_hop(W, in, k, L0, L1), DAG);
    if (DAG) {
      const double2 o = in[k.s];
      out[k.s] = make_double2(o.x - v.x, o.y - v.y);
    } else {
      out[k.s] = v;
    }
  }
}
// out = src + sign C in; EVEN: on the even blocks, and 0 on the odd block beside each (a
// warp of alternating blocks would spend its FP64 issue on idle lanes).
template <bool EVEN>
__global__ void __launch_bounds__(128) k_kd_hop(const double2* __restrict__ W, double sign,
                                                const double2* __restrict__ src,
                                                const double2* __restrict__ in,
                                                double2* __restrict__ out, int L0, int L1) {
  KdSite k;
  for (int X1 = blockIdx.y; X1 < L1 / 2; X1 += gridDim.y) {
    if (!kd_site(L0, L1, EVEN ? 0 : -1, X1, k)) return;
    const double2 c = kd_hop(W, in, k, L0, L1);
    double2 o = src[k.s];
    o.x = fma(sign, c.x, o.x);
    o.y = fma(sign, c.y, o.y);
    out[k.s] = o;
    if (EVEN) out[k.s + ((k.x0 & 2) ? -2 : 2)] = make_double2(0.0, 0.0);
  }
}

inline int nblocks(long n, int t) { return (int)((n + t - 1) / t); }

}  // namespace

void launch_long_links(const sw_gauge* g, double c3, double2* W3, cudaStream_t s) {
  k_long_links<<<nblocks(g->N, 256), 256, 0, s>>>(g->W_lex, c3, W3, g->L0, g->L1);
  SW_LAUNCH_CHECK();
}
void launch_dslash_naik_lex(const sw_gauge* g, const double2* W3, double mass, double c1,
                            const double2* in, double2* out, cudaStream_t s) {
  dim3 grid(nblocks(g->L0, 256), g->L1);
  k_dslash_naik_lex<<<grid, 256, 0, s>>>(in, out, g->W_lex, W3, mass, c1, g->L0, g->L1);
  SW_LAUNCH_CHECK();
}
void launch_dslash_ps(const sw_gauge* g, double mass, int dagger, const double2* in, double2* out,
                      cudaStream_t s) {
  k_dslash_ps<<<nblocks(g->N, 256), 256, 0, s>>>(g->W_ps, mass, dagger ? -1.0 : 1.0, in, out,
                                                 g->L0, g->L1);
  SW_LAUNCH_CHECK();
}

void launch_dslash_lex(const sw_gauge* g, double mass, int dagger, const double2* in, double2* out,
                       cudaStream_t s) {
  dim3 grid(nblocks(g->L0, 256), g->L1);
  auto k = dagger ? k_dslash_lex<true> : k_dslash_lex<false>;
  k<<<grid, 256, 0, s>>>(in, out, g->W_lex, mass, g->L0, g->L1);
  SW_LAUNCH_CHECK();
}
void launch_dslash_lex32(const sw_gauge* g, float mass, int dagger, const float2* in, float2* out,
                         cudaStream_t s) {
  dim3 grid(nblocks(g->L0, 256), g->L1);
  auto k = dagger ? k_dslash_lex32<true> : k_dslash_lex32<false>;
  k<<<grid, 256, 0, s>>>(in, out, g->W_lex32, mass, g->L0, g->L1);
  SW_LAUNCH_CHECK();
}
void launch_pack(const sw_gauge* g, const double2* lex, double2* ps, cudaStream_t s) {
  k_pack<<<nblocks(g->N, 256), 256, 0, s>>>(lex, ps, g->L0, g->L1);
  SW_LAUNCH_CHECK();
}
void launch_unpack(const sw_gauge* g, const double2* ps, double2* lex, cudaStream_t s) {
  k_unpack<<<nblocks(g->N, 256), 256, 0, s>>>(ps, lex, g->L0, g->L1);
  SW_LAUNCH_CHECK();
}
void launch_binv_build(const sw_gauge* g, double mass, double2* binv, cudaStream_t s,
                       double hop_scale) {
  k_binv_build<<<nblocks(g->N / 4, 128), 128, 0, s>>>(g->W_ps, mass, hop_scale, binv, g->L0,
                                                      g->L1);
  SW_LAUNCH_CHECK();
}
void many_block_apply(const sw_gauge* g, const double2* binv, int par, int dagger,
                      const Many<2>& io, cudaStream_t s, const int* ctl) {
  const int half = g->N / 8, nblk = par < 0 ? 2 * half : half;
  with_width(io.n, [&](auto w) {
    constexpr int W = decltype(w)::value;
    launch_early(k_block_apply<W>, dim3(nblocks(4L * nblk, 128), io.n), 128, 0, s,
                 binv + (par > 0 ? (long)half * 16 : 0), Pack<2, W>(io), nblk, dagger, ctl);
  });
}
void many_hop(const sw_gauge* g, int par, double sign, const Many<3>& io, cudaStream_t s,
              const int* ctl) {
  with_width(io.n, [&](auto w) {
    constexpr int W = decltype(w)::value;
    launch_early(k_hop<W>, dim3(nblocks(par < 0 ? g->N : g->N / 2, 256), io.n), 256, 0, s, g->W_ps,
                 par, sign, Pack<3, W>(io), g->L0, g->L1, ctl);
  });
}
void many_hop_block(const sw_gauge* g, const double2* binv, int par, int dagger, double sign,
                    const Many<3>& io, cudaStream_t s, const int* ctl) {
  with_width(io.n, [&](auto w) {
    constexpr int W = decltype(w)::value;
    launch_early(k_hop_block<W>, dim3(nblocks(par < 0 ? g->N : g->N / 2, 128), io.n), 128, 0, s,
                 g->W_ps, binv, par, dagger, sign, Pack<3, W>(io), g->L0, g->L1, ctl);
  });
}
void launch_block_apply(const sw_gauge* g, const double2* binv, int par, int dagger,
                        const double2* in, double2* out, cudaStream_t s) {
  many_block_apply(g, binv, par, dagger, Many<2>(0, in, out), s);
}
void launch_hop(const sw_gauge* g, int par, double sign, const double2* src, const double2* in,
                double2* out, cudaStream_t s) {
  many_hop(g, par, sign, Many<3>(0, src, in, out), s);
}

// Member-wise Many of operands k... of another.
template <int K, typename... I>
static Many<sizeof...(I)> pick(const Many<K>& a, I... k) {
  Many<sizeof...(I)> o;
  for (int m = 0; m < a.n; ++m) o.add(a.slot[m], a.v[k][m]...);
  return o;
}
// A A^dag x with A^dag x = x + B^-dag C^dag x = x - B^-dag C x (C is anti-Hermitian) and
// A t = t + C B^-1 t.
void many_normal_A(const sw_gauge* g, const double2* binv, const Many<4>& v, cudaStream_t s,
                   const int* ctl) {
  many_hop_block(g, binv, -1, 1, -1.0, pick(v, 0, 0, 2), s, ctl);
  many_block_apply(g, binv, -1, 0, pick(v, 2, 3), s, ctl);
  many_hop(g, -1, 1.0, pick(v, 2, 3, 1), s, ctl);
}
// S x_e = x_e - A_eo A_oe x_e with A_oe = C_oe B_e^-1 and A_eo = C_eo B_o^-1
// (A_ee = A_oo = I on KD-block parity):
//   t_e = B_e^-1 x_e;  v_o = B_o^-1 C_oe t_e;  y_e = x_e - C_eo v_o.
void many_S(const sw_gauge* g, const double2* binv, const Many<3>& v, cudaStream_t s) {
  Many<3> hb;
  for (int m = 0; m < v.n; ++m) hb.add(0, (const double2*)nullptr, v.v[1][m], v.v[2][m]);
  many_block_apply(g, binv, 0, 0, pick(v, 0, 1), s);
  many_hop_block(g, binv, 1, 0, 1.0, hb, s);
  many_hop(g, 0, -1.0, pick(v, 0, 2, 1), s);
}

static dim3 kd_grid(const sw_gauge* g, bool half) {
  const int rows = g->L1 / 2;
  return dim3(nblocks(g->L0 * (half ? 1L : 2L), 128), rows < 32768 ? rows : 32768);
}
// The same operators on lexicographic fields; tmp must hold N complex, out may be neither in
// nor tmp.
void fine_lex_A(const sw_gauge* g, const double2* binv, const double2* in, double2* out,
                double2* tmp, cudaStream_t s) {
  k_kd_block<<<kd_grid(g, false), 128, 0, s>>>(binv, -1, in, tmp, g->L0, g->L1);
  SW_LAUNCH_CHECK();
  k_kd_hop<false><<<kd_grid(g, false), 128, 0, s>>>(g->W_lex, 1.0, in, tmp, out, g->L0, g->L1);
  SW_LAUNCH_CHECK();
}
void fine_lex_Adag(const sw_gauge* g, const double2* binv, const double2* in, double2* out,
                   cudaStream_t s) {
  k_kd_hop_block<true><<<kd_grid(g, false), 128, 0, s>>>(g->W_lex, binv, -1, in, out, g->L0, g->L1);
  SW_LAUNCH_CHECK();
}
void fine_lex_S(const sw_gauge* g, const double2* binv, const double2* in, double2* out,
                double2* tmp, cudaStream_t s) {
  k_kd_block<<<kd_grid(g, true), 128, 0, s>>>(binv, 0, in, tmp, g->L0, g->L1);
  SW_LAUNCH_CHECK();
  k_kd_hop_block<false><<<kd_grid(g, true), 128, 0, s>>>(g->W_lex, binv, 1, tmp, tmp, g->L0, g->L1);
  SW_LAUNCH_CHECK();
  k_kd_hop<true><<<kd_grid(g, true), 128, 0, s>>>(g->W_lex, -1.0, in, tmp, out, g->L0, g->L1);
  SW_LAUNCH_CHECK();
}
