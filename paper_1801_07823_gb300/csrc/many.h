// Vector operations and level operators over the members of a batch (right-hand
// sides of a batched solve, null vectors of a setup; a single solve is a batch of
// one) with one launch for all of them.
#pragma once
#include <type_traits>

#include "sw_internal.h"

// Operands of up to kMaxBatch members: v[k][m] is operand k of member m; slot[m] the
// member's first scalar slot.
template <int K>
struct Many {
  int n = 0;
  double2* v[K][kMaxBatch];
  int slot[kMaxBatch];
  Many() = default;
  template <typename... P>
  Many(int first_slot, P... p) {
    add(first_slot, p...);
  }
  template <typename... P>
  void add(int first_slot, P... p) {
    static_assert(sizeof...(P) == K, "one pointer per operand");
    double2* q[K] = {const_cast<double2*>((const double2*)p)...};
    for (int k = 0; k < K; ++k) v[k][n] = q[k];
    slot[n++] = first_slot;
  }
};
// The same as a kernel parameter, W >= n members wide.
template <int K, int W>
struct Pack {
  double2* v[K][W];
  int slot[W];
  explicit Pack(const Many<K>& m) {
    for (int i = 0; i < W; ++i) {
      const bool in = i < m.n;
      for (int k = 0; k < K; ++k) v[k][i] = in ? m.v[k][i] : nullptr;
      slot[i] = in ? m.slot[i] : 0;
    }
  }
};
// Calls f with the narrowest of the compiled widths that holds n members: a
// launch's parameters are copied to the device, so one member should not
// carry the pointers of 64.
template <typename F>
void with_width(int n, F&& f) {
  if (n <= 1)
    f(std::integral_constant<int, 1>{});
  else if (n <= 16)
    f(std::integral_constant<int, 16>{});
  else
    f(std::integral_constant<int, kMaxBatch>{});
}

// Slots are relative to each member's first; sums go to slots, coefficients come from
// them.  host: also the first component of each member's sum, to host[m] (pinned memory).
// ctl: member m does nothing when ctl[4 m] is set.  Operands are named in their order.
void many_init(sw_ctx* c, long n, const Many<3>& xrb, int s_rr, double* host);  // x = 0, r = b, |r|^2
void many_dot_norm(sw_ctx* c, long n, const Many<2>& qr, int s);  // <q, r>, |q|^2 in s, s + 1
// MR step with a = om S[s] / S[s + 1].  First: x = a b, r = b - a q; then x += a r, r -= a q;
// last of the post-smoother: o = (x1 + e) + (x + a r).
void many_mr_first(sw_ctx* c, long n, const Many<4>& xrbq, int s, double om);
void many_mr(sw_ctx* c, long n, const Many<3>& xrq, int s, double om);
void many_mr_last(sw_ctx* c, long n, const Many<5>& oxrab, int s, double om, bool first);
void many_sub(sw_ctx* c, long n, const Many<3>& oab);                       // o = a - b
void many_sub_norm(sw_ctx* c, long n, const Many<3>& oab, int s, double* host);
void many_dot(sw_ctx* c, long n, const Many<2>& ab, int s);
void many_norm(sw_ctx* c, long n, const Many<1>& a, int s, double* host = nullptr);
// q -= S[s] qj, p -= S[s] pj; then <qn, q> in s, or |q|^2 in s_qq for a member without qn
void many_mgs(sw_ctx* c, long n, const Many<5>& q_p_qj_pj_qn, int s, int s_qq);
void many_scale_dot(sw_ctx* c, long n, const Many<3>& qpr, int s_qq, int s_a);  // q, p /= |q|; <q, r>
// x += S[s_a] p, r -= S[s_a] q; |r|^2
void many_update(sw_ctx* c, long n, const Many<4>& xrpq, int s_a, int s_rr, double* host);
// <a, b> and |a|^2 of the setup, like many_cg_start and many_cg_step with plain FP64 trees over
// fixed slices (see mg_setup).
void many_setup_dot(sw_ctx* c, long n, const Many<2>& ab, int s, const int* ctl = nullptr);
void many_setup_norm(sw_ctx* c, long n, const Many<1>& a, int s, double* host = nullptr);
void many_copy(sw_ctx* c, long n, const Many<2>& ob);                       // o = b
void many_add(sw_ctx* c, long n, const Many<2>& ob);                        // o += b
void many_project(sw_ctx* c, long n, const Many<2>& vu, int s);             // v -= S[s] u
void many_normalise(sw_ctx* c, long n, const Many<1>& v, int s);            // v /= sqrt(S[s])
// CG with stopping tests on the device, in ctl per member: [0] done, [1] iterations,
// [2] non-finite residual.  Start: x = 0, r = p = -b; step: x += a p, r -= a q with
// a = S[s_rr] / S[s_pq], |r|^2 in s_new; S[s_stop] is the norm to reach.
void many_cg_start(sw_ctx* c, long n, const Many<4>& xrpb, int s_rr, int s_stop, double tol,
                   int maxit, int* ctl);
void many_cg_step(sw_ctx* c, long n, const Many<4>& xrpq, int s_rr, int s_pq, int s_new, int s_stop,
                  int maxit, int* ctl);
void many_xpay(sw_ctx* c, long n, const Many<2>& pr, int s_new, int s_old, const int* ctl);

// Operators on the members.  par < 0: both halves of full parity-split vectors.
void many_block_apply(const sw_gauge* g, const double2* binv, int par, int dagger,
                      const Many<2>& in_out, cudaStream_t s, const int* ctl = nullptr);
void many_hop(const sw_gauge* g, int par, double sign, const Many<3>& src_in_out, cudaStream_t s,
              const int* ctl = nullptr);
void many_hop_block(const sw_gauge* g, const double2* binv, int par, int dagger, double sign,
                    const Many<3>& src_in_out, cudaStream_t s, const int* ctl = nullptr);
// S on even halves; tmp: N / 2 per member.  out serves as scratch: neither in nor tmp.
void many_S(const sw_gauge* g, const double2* binv, const Many<3>& in_out_tmp, cudaStream_t s);
void many_S32(const sw_gauge* g, const float2* W32, const float2* binv32, const Many<3>& in_out_tmp,
              cudaStream_t s);
// A A^dag on full vectors; t, u: N of scratch.
void many_normal_A(const sw_gauge* g, const double2* binv, const Many<4>& in_out_t_u,
                   cudaStream_t s, const int* ctl);
// FP64 stencil on the FP64 pipe, its sums in a fixed order.
void many_coarse(const CoarseGeom& g, const double2* Y, int dagger, const Many<2>& in_out,
                 cudaStream_t s, const int* ctl = nullptr, unsigned long long* exec = nullptr);
void many_coarse_h(const CoarseGeom& g, const __half2* Yh, const float* scale, int dagger,
                   const Many<2>& in_out, cudaStream_t s);
void many_digit(const CoarseGeom& g, const DigitStencil& t, const double2* Y, int dagger,
                const Many<2>& in_out, int device, cudaStream_t s, const int* ctl,
                unsigned long long* exec);
// Level-1 transfer on the even parity half.  P: [N][nv] parity-split rows.
// full = 1: full parity-split vectors (fine operator D) instead of the even half.
// lex: the fine vector is a whole lexicographic field (odd sites ignored, or written as 0).
void many_restrict_fine(const sw_gauge* g, int a0, int a1, int nv, const double2* P,
                        const Many<2>& in_out, cudaStream_t s, int full = 0, bool lex = false);
void many_prolong_fine(const sw_gauge* g, int a0, int a1, int nv, const double2* P,
                       const Many<2>& in_out, cudaStream_t s, int full = 0, bool lex = false);
// Level >= 2 transfer.  P: [sites][nc][nv].
void many_restrict_coarse(const CoarseGeom& g, int b0, int b1, int nv, const double2* P,
                          const Many<2>& in_out, cudaStream_t s);
void many_prolong_coarse(const CoarseGeom& g, int b0, int b1, int nv, const double2* P,
                         const Many<2>& in_out, cudaStream_t s);
