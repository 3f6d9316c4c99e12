// split2d.cuh -- the FP64 block recursion of the 2D Euler step (Eqs. 4.5-4.6)
// on the FP32 pipes: the method of split1d.cuh (float-float pairs on flux
// increments, one Jacobian product per order, precision by magnitude) on the
// 2p x 2p block. Node j of the block anchored at cell a carries f(u_j) - f(u_a)
// and g(u_j) - g(u_a); with (v, w) the velocity, d = (a, b1, b2, e),
//   W1 = b1 - v a, W2 = b2 - w a, L = dH' - h a, (dv, dw) = (W1, W2) / (rho + a),
//   Q11 = W1 dv, Q12 = W1 dw, Q22 = W2 dw, T = (dv, dw) (L - kappa (Q11 + Q22)),
// the remainder of f is (0, Q11 - kappa Q, Q12, T1 - v kappa Q), Q = Q11 + Q22,
// and of g (0, Q12, Q22 - kappa Q, T2 - w kappa Q).
#pragma once

#include "split1d.cuh"

namespace {

// Per-cell record: u as three floats per component, (v, w) and h as pairs, the
// velocity scale s = sqrt(h) (NaN outside the range the pairs carry).
struct Split2Rec {
  float4 uh, um, ul;  // high, middle and low parts of rho, m_x, m_y, E
  float4 vw;          // v, w as pairs
  float4 hs;          // h as a pair, s
};

__device__ __forceinline__ void split2_record(Split2Rec &r, const double *u, double gm1) {
  const double ri = recip(u[0]);
  const double v = __dmul_rn(u[1], ri), w = __dmul_rn(u[2], ri);
  const double p = __dmul_rn(gm1, fma(-0.5, fma(u[2], w, __dmul_rn(u[1], v)), u[3]));
  const double h = __dmul_rn(__dadd_rn(u[3], p), ri);
  const F3 a = f3_from(u[0]), b = f3_from(u[1]), c = f3_from(u[2]), e = f3_from(u[3]);
  const FF V = ff_bits(v), W = ff_bits(w), H = ff_bits(h);
  r.uh = make_float4(a.h, b.h, c.h, e.h);
  r.um = make_float4(a.m, b.m, c.m, e.m);
  r.ul = make_float4(a.l, b.l, c.l, e.l);
  r.vw = make_float4(V.h, V.l, W.h, W.l);
  const float s0 = __fsqrt_rn(H.h), m0 = __fmul_rn(a.h, s0), m1 = __fmul_rn(a.h, H.h), m2 = __fmul_rn(m1, s0);
  const bool fine = split_range(a.h) && split_range(H.h) && split_range(m0) && split_range(m1) && split_range(m2);
  r.hs = make_float4(H.h, H.l, fine ? s0 : __int_as_float(0x7fffffff), 0.0f);
}

struct Split2Const {
  FF gam, kap, gm1;
};
__device__ __forceinline__ Split2Const split2_const(const Step2DArgs &a) {
  return Split2Const{ff_of(a.sgam), ff_of(a.skap), ff_of(a.sgm1)};
}

// The linear parts at a node (rho, v, w, h) for d = (u[0], u[1], u[2], u[3]):
// F[0..3], G[1..3] of the Jacobian products (G[0] = u[2], F[0] = u[1]), and W1,
// W2, L.
struct Split2Lin {
  FF F1, F2, F3, G2, G3, W1, W2, L;
};
__device__ __forceinline__ Split2Lin split2_lin(const Split2Const &C, FF v, FF w, FF h, const FF *u) {
  Split2Lin o;
  o.W1 = ff_add(u[1], ff_neg(ff_mul(v, u[0])));
  o.W2 = ff_add(u[2], ff_neg(ff_mul(w, u[0])));
  const FF m1 = ff_mul(v, ff_add(u[1], o.W1)), m2 = ff_mul(w, ff_add(u[2], o.W2));
  const FF dp = ff_add(ff_mul(C.gm1, u[3]), ff_neg(ff_mul(C.kap, ff_add(m1, m2))));
  const FF Lp = ff_add(u[3], dp);
  o.L = ff_add(Lp, ff_neg(ff_mul(h, u[0])));
  o.F1 = ff_add(m1, dp);
  o.G2 = ff_add(m2, dp);
  o.F2 = ff_add(ff_mul(w, u[1]), ff_mul(v, o.W2));
  o.F3 = ff_add(ff_mul(h, o.W1), ff_mul(v, Lp));
  o.G3 = ff_add(ff_mul(h, o.W2), ff_mul(w, Lp));
  return o;
}
// Adds the remainder sums (Q11, Q12, Q22, T1, T2) of pairs / of floats.
__device__ __forceinline__ void split2_rem(const Split2Const &C, FF v, FF w, const FF *u, const Split2Lin &o,
                                           const FF *q, FF *F, FF *G) {
  const FF kq = ff_mul(C.kap, ff_add(q[0], q[2]));
  F[0] = u[1];
  F[1] = ff_add(o.F1, ff_add(q[0], ff_neg(kq)));
  F[2] = ff_add(o.F2, q[1]);
  F[3] = ff_add(o.F3, ff_add(q[3], ff_neg(ff_mul(v, kq))));
  G[0] = u[2];
  G[1] = F[2];
  G[2] = ff_add(o.G2, ff_add(q[2], ff_neg(kq)));
  G[3] = ff_add(o.G3, ff_add(q[4], ff_neg(ff_mul(w, kq))));
}
__device__ __forceinline__ void split2_remf(const Split2Const &C, FF v, FF w, const FF *u, const Split2Lin &o,
                                            const float *q, FF *F, FF *G) {
  const float kq = __fmul_rn(C.kap.h, __fadd_rn(q[0], q[2]));
  F[0] = u[1];
  F[1] = ff_addf(o.F1, __fsub_rn(q[0], kq));
  F[2] = ff_addf(o.F2, q[1]);
  F[3] = ff_addf(o.F3, fmaf(-v.h, kq, q[3]));
  G[0] = u[2];
  G[1] = F[2];
  G[2] = ff_addf(o.G2, __fsub_rn(q[2], kq));
  G[3] = ff_addf(o.G3, fmaf(-w.h, kq, q[4]));
}
// The nonlinear terms at Taylor sums (D, W1, W2, L), D = rho + a.
__device__ __forceinline__ void split2_terms(FF kap, FF D, FF W1, FF W2, FF L, FF *q) {
  const float r0 = recip(D.h);
  const FF dv = ff_quot(W1, D, r0), dw = ff_quot(W2, D, r0);
  q[0] = ff_mul(W1, dv);
  q[1] = ff_mul(W1, dw);
  q[2] = ff_mul(W2, dw);
  const FF t = ff_add(L, ff_neg(ff_mul(kap, ff_add(q[0], q[2]))));
  q[3] = ff_mul(dv, t);
  q[4] = ff_mul(dw, t);
}
__device__ __forceinline__ void split2_termsf(float kap, float D, float W1, float W2, float L, float *q) {
  const float r = recip(D), dv = __fmul_rn(W1, r), dw = __fmul_rn(W2, r);
  q[0] = __fmul_rn(W1, dv);
  q[1] = __fmul_rn(W1, dw);
  q[2] = __fmul_rn(W2, dw);
  const float t = fmaf(-kap, __fadd_rn(q[0], q[2]), L);
  q[3] = __fmul_rn(dv, t);
  q[4] = __fmul_rn(dw, t);
}

// Exchange slots of the nodes' F^(k)/k! and G^(k)/k!: high and low parts.
struct Split2Slots {
  float4 *Fh, *Fl, *Gh, *Gl;
};
__device__ __forceinline__ void split2_put(const Split2Slots &x, int i, const FF *F, const FF *G) {
  x.Fh[i] = make_float4(F[0].h, F[1].h, F[2].h, F[3].h);
  x.Fl[i] = make_float4(F[0].l, F[1].l, F[2].l, F[3].l);
  x.Gh[i] = make_float4(G[0].h, G[1].h, G[2].h, G[3].h);
  x.Gl[i] = make_float4(G[0].l, G[1].l, G[2].l, G[3].l);
}

// One node of a 2p x 2p block: its state over the orders.
template <int p>
struct Split2Node {
  static constexpr int n = 2 * p, NL = n - 1;
  FF rho, v, w, h;
  float rs, rh, rhs;  // scales of rho v, of pressure and of energy flux
  FF A[NL], W1[NL], W2[NL], L[NL];
  float Ba, Bw, Bl;   // bounds of the Taylor sums
  int form;           // of the remainders (split1d.cuh): 0, 1 or 2, the same for all nodes of a vote
  FF w1, w2, l1;      // form 1: the first-order terms,
  float q1[5];        // their products over rho (float),
  float Pw, Pl;       // and their bounds p |W1|, p |L1|
};

// Loads node `r` of the block anchored at record `ra`; returns
// F = f(u_j) - f(u_a), G likewise, and whether they are below TAU of the scales.
template <int p>
__device__ __forceinline__ bool split2_start(const Split2Const &C, const Split2Rec &r, const Split2Rec &ra,
                                             Split2Node<p> &N, FF *F, FF *G) {
  const float4 uh = r.uh, um = r.um, ul = r.ul, ah = ra.uh, am = ra.um, al = ra.ul, avw = ra.vw, ahs = ra.hs;
  FF d[4];
  d[0] = f3_diff(F3{uh.x, um.x, ul.x}, F3{ah.x, am.x, al.x});
  d[1] = f3_diff(F3{uh.y, um.y, ul.y}, F3{ah.y, am.y, al.y});
  d[2] = f3_diff(F3{uh.z, um.z, ul.z}, F3{ah.z, am.z, al.z});
  d[3] = f3_diff(F3{uh.w, um.w, ul.w}, F3{ah.w, am.w, al.w});
  {
    const FF va{avw.x, avw.y}, wa{avw.z, avw.w}, ha{ahs.x, ahs.y};
    const Split2Lin o = split2_lin(C, va, wa, ha, d);
    FF q[5];
    split2_terms(C.kap, ff_add(FF{ah.x, am.x}, d[0]), o.W1, o.W2, o.L, q);
    split2_rem(C, va, wa, d, o, q, F, G);
  }
  N.rho = FF{uh.x, um.x};
  N.v = FF{r.vw.x, r.vw.y};
  N.w = FF{r.vw.z, r.vw.w};
  N.h = FF{r.hs.x, r.hs.y};
  N.rs = __fmul_rn(uh.x, r.hs.z);
  N.rh = __fmul_rn(uh.x, r.hs.x);
  N.rhs = __fmul_rn(N.rh, r.hs.z);
  N.Ba = N.Bw = N.Bl = N.Pw = N.Pl = 0.0f;
  N.w1 = N.w2 = N.l1 = FF{0.0f, 0.0f};
#pragma unroll
  for (int q = 0; q < 5; q++) N.q1[q] = 0.0f;
#pragma unroll
  for (int q = 0; q < Split2Node<p>::NL; q++) {
    N.A[q] = N.rho;
    N.W1[q] = N.W2[q] = N.L[q] = FF{0.0f, 0.0f};
  }
  // the anchor's scales too: its state is the base of the increments
  return fabsf(F[0].h) <= SPLIT_TAU * N.rs && fabsf(G[0].h) <= SPLIT_TAU * N.rs &&
         fabsf(F[1].h) <= SPLIT_TAU * N.rh && fabsf(F[2].h) <= SPLIT_TAU * N.rh &&
         fabsf(G[2].h) <= SPLIT_TAU * N.rh && fabsf(F[3].h) <= SPLIT_TAU * N.rhs &&
         fabsf(G[3].h) <= SPLIT_TAU * N.rhs && fabsf(d[0].h) <= SPLIT_TAU * uh.x && ahs.z > 0.0f;
}

// Whether the node's F, G are below SPLIT_TAIL of the scales.
template <int p>
__device__ __forceinline__ bool split2_small(const Split2Node<p> &N, const FF *F, const FF *G) {
  return fmaxf(fabsf(F[0].h), fabsf(G[0].h)) <= SPLIT_TAIL * N.rs &&
         fmaxf(fmaxf(fabsf(F[1].h), fabsf(F[2].h)), fabsf(G[2].h)) <= SPLIT_TAIL * N.rh &&
         fmaxf(fabsf(F[3].h), fabsf(G[3].h)) <= SPLIT_TAIL * N.rhs;
}
// After the last order: whether the pairs held, and whether float remainders did.
template <int p>
__device__ __forceinline__ bool split2_held(const Split2Node<p> &N) {
  return N.Ba <= SPLIT_TAU * N.rho.h && N.Bw <= SPLIT_TAU * N.rs && N.Bl <= SPLIT_TAU * N.rh;
}
template <int p>
__device__ __forceinline__ bool split2_quad(const Split2Node<p> &N, float m) {
  const float bw = m * N.Bw, bl = m * N.Bl;
  return bw * bw <= SPLIT_QUAD * N.rs * N.rs && bw * bl <= SPLIT_QUAD * N.rs * N.rh;
}
template <int p>
__device__ __forceinline__ bool split2_cubic(const Split2Node<p> &N, float m) {
  return split_cubic(m * N.Ba, m * N.Bw, m * N.Bl, N.rho.h, N.rs, N.rh);
}
// After the last order: whether the form of the remainders held.
template <int p>
__device__ __forceinline__ bool split2_form(const Split2Node<p> &N) {
  if (N.form == 0) return split2_quad(N, 1.0f);
  if (N.form == 2) return true;
  const float dw = N.Bw - N.Pw, dl = N.Bl - N.Pl;
  return split2_cubic(N, 1.0f) && dw * N.Bw <= SPLIT_MIX * N.rs * N.rs && dw * N.Bl <= SPLIT_MIX * N.rs * N.rh &&
         dl * N.Bw <= SPLIT_MIX * N.rs * N.rh;
}
// The bounds after an order's U (float parts), and at k = 2 the terms of form 1.
template <int p>
__device__ __forceinline__ void split2_bounds(Split2Node<p> &N, const float2 *lv, float a, float w1, float w2, float l) {
  const float pk = lv[Split2Node<p>::NL - 1].x;  // p^(k-1)
  N.Ba = fmaf(pk, fabsf(a), N.Ba);
  N.Bw = fmaf(pk, fmaxf(fabsf(w1), fabsf(w2)), N.Bw);
  N.Bl = fmaf(pk, fabsf(l), N.Bl);
}
template <int p>
__device__ __forceinline__ void split2_first(Split2Node<p> &N, const Split2Lin &o) {
  N.w1 = o.W1;
  N.w2 = o.W2;
  N.l1 = o.L;
  N.Pw = N.Bw;
  N.Pl = N.Bl;
  const float ri = recip(N.rho.h), v = __fmul_rn(o.W1.h, ri), w = __fmul_rn(o.W2.h, ri);
  N.q1[0] = __fmul_rn(o.W1.h, v);
  N.q1[1] = __fmul_rn(o.W1.h, w);
  N.q1[2] = __fmul_rn(o.W2.h, w);
  N.q1[3] = __fmul_rn(o.L.h, v);
  N.q1[4] = __fmul_rn(o.L.h, w);
}
// The weighted sums of an order's remainders in forms 0 and 1 (without the leading
// terms of form 1).
template <int p>
__device__ __forceinline__ void split2_levels(Split2Node<p> &N, float kap, int k, const float2 *lv, float a,
                                              float w1, float w2, float l, float *q) {
  constexpr int NL = Split2Node<p>::NL;
#pragma unroll
  for (int e = 0; e < 5; e++) q[e] = 0.0f;
  if (N.form == 0) {
#pragma unroll
    for (int i = 0; i < NL; i++) {
      const float c = lv[i].x, wt = lv[i].y;
      N.A[i].h = fmaf(c, a, N.A[i].h);
      N.W1[i].h = fmaf(c, w1, N.W1[i].h);
      N.W2[i].h = fmaf(c, w2, N.W2[i].h);
      N.L[i].h = fmaf(c, l, N.L[i].h);
      float t[5];
      split2_termsf(kap, N.A[i].h, N.W1[i].h, N.W2[i].h, N.L[i].h, t);
#pragma unroll
      for (int e = 0; e < 5; e++) q[e] = fmaf(wt, t[e], q[e]);
    }
  } else {
    if (k == 2) {  // A without rho, the others without their first-order terms
#pragma unroll
      for (int i = 0; i < NL; i++) N.A[i].h = 0.0f;
      w1 = w2 = l = 0.0f;
    }
#pragma unroll
    for (int i = 0; i < NL; i++) {
      const float r = (float)(i < p - 1 ? i - p + 1 : i - p + 2), c = lv[i].x, wt = lv[i].y;
      N.A[i].h = fmaf(c, a, N.A[i].h);
      N.W1[i].h = fmaf(c, w1, N.W1[i].h);
      N.W2[i].h = fmaf(c, w2, N.W2[i].h);
      N.L[i].h = fmaf(c, l, N.L[i].h);
      const float R = recip(__fadd_rn(N.rho.h, N.A[i].h)), ra = __fmul_rn(-(r * r), N.A[i].h);
      const float x1 = __fmul_rn(r, N.w1.h), x2 = __fmul_rn(r, N.w2.h);
      const float y1 = __fadd_rn(x1, N.W1[i].h), y2 = __fadd_rn(x2, N.W2[i].h), yl = fmaf(r, N.l1.h, N.L[i].h);
      // products of the sums less their leading part, r^2 q1 (1 + a / rho)
      const float n0 = fmaf(ra, N.q1[0], __fmul_rn(N.W1[i].h, __fadd_rn(x1, y1)));
      const float n1 = fmaf(ra, N.q1[1], fmaf(N.W1[i].h, y2, __fmul_rn(x1, N.W2[i].h)));
      const float n2 = fmaf(ra, N.q1[2], __fmul_rn(N.W2[i].h, __fadd_rn(x2, y2)));
      const float n3 = fmaf(ra, N.q1[3], fmaf(N.W1[i].h, yl, __fmul_rn(x1, N.L[i].h)));
      const float n4 = fmaf(ra, N.q1[4], fmaf(N.W2[i].h, yl, __fmul_rn(x2, N.L[i].h)));
      const float t0 = __fmul_rn(n0, R), t2 = __fmul_rn(n2, R);
      const float kq = __fmul_rn(-kap, fmaf(r * r, __fadd_rn(N.q1[0], N.q1[2]), __fadd_rn(t0, t2)));
      q[0] = fmaf(wt, t0, q[0]);
      q[1] = fmaf(wt, __fmul_rn(n1, R), q[1]);
      q[2] = fmaf(wt, t2, q[2]);
      q[3] = fmaf(wt, __fmul_rn(R, fmaf(y1, kq, n3)), q[3]);
      q[4] = fmaf(wt, __fmul_rn(R, fmaf(y2, kq, n4)), q[4]);
    }
  }
#pragma unroll
  for (int e = 0; e < 5; e++) q[e] = __fmul_rn(q[e], 1.0f / split_lq(p));
}

// U^(k-1)/(k-1)! of a node from the slots of its row (i0 + r) and its column
// (j0 + r n), with integer weights gx, gy; lx, ly = -lambda / ((k-1) LC).
template <int p>
__device__ __forceinline__ void split2_sums(const Split2Slots &x, int i0, int j0, int js, const float *gx,
                                            const float *gy, FF lx, FF ly, FF *u) {
  constexpr int n = 2 * p;
  FF a[4], b[4];
#pragma unroll
  for (int c = 0; c < 4; c++) a[c] = b[c] = FF{0.0f, 0.0f};
#pragma unroll
  for (int r = 0; r < n; r++) {
    const float4 yh = x.Fh[i0 + r], yl = x.Fl[i0 + r];
    ff_acc(a[0], FF{yh.x, yl.x}, gx[r]);
    ff_acc(a[1], FF{yh.y, yl.y}, gx[r]);
    ff_acc(a[2], FF{yh.z, yl.z}, gx[r]);
    ff_acc(a[3], FF{yh.w, yl.w}, gx[r]);
  }
#pragma unroll
  for (int r = 0; r < n; r++) {
    const float4 yh = x.Gh[j0 + r * js], yl = x.Gl[j0 + r * js];
    ff_acc(b[0], FF{yh.x, yl.x}, gy[r]);
    ff_acc(b[1], FF{yh.y, yl.y}, gy[r]);
    ff_acc(b[2], FF{yh.z, yl.z}, gy[r]);
    ff_acc(b[3], FF{yh.w, yl.w}, gy[r]);
  }
#pragma unroll
  for (int c = 0; c < 4; c++) u[c] = ff_add(ff_mul(ff_norm(a[c]), lx), ff_mul(ff_norm(b[c]), ly));
}

// Order k of a node in pairs, the remainders in the node's form. u: from
// split2_sums, o: from split2_lin.
template <int p>
__device__ __forceinline__ void split2_order(const Split2Const &C, Split2Node<p> &N, int k, const float2 *lv,
                                             const FF *u, const Split2Lin &o, FF *F, FF *G) {
  constexpr int NL = 2 * p - 1;
  if (N.form < 2) {
    float q[5];
    split2_levels(N, C.kap.h, k, lv, u[0].h, o.W1.h, o.W2.h, o.L.h, q);
    split2_remf(C, N.v, N.w, u, o, q, F, G);
    if (k == 3 && N.form == 1) {  // the leading terms
      const float ri = recip(N.rho.h);
      const FF dv = ff_quot(N.w1, N.rho, ri), dw = ff_quot(N.w2, N.rho, ri);
      const FF q0 = ff_mul(N.w1, dv), q2 = ff_mul(N.w2, dw), kq = ff_mul(C.kap, ff_add(q0, q2));
      F[1] = ff_add(F[1], ff_add(q0, ff_neg(kq)));
      F[2] = ff_add(F[2], ff_mul(N.w1, dw));
      F[3] = ff_add(F[3], ff_add(ff_mul(dv, N.l1), ff_neg(ff_mul(N.v, kq))));
      G[1] = F[2];
      G[2] = ff_add(G[2], ff_add(q2, ff_neg(kq)));
      G[3] = ff_add(G[3], ff_add(ff_mul(dw, N.l1), ff_neg(ff_mul(N.w, kq))));
    }
  } else {
    FF q[5];
#pragma unroll
    for (int e = 0; e < 5; e++) q[e] = FF{0.0f, 0.0f};
#pragma unroll
    for (int i = 0; i < NL; i++) {
      const float c = lv[i].x, wt = lv[i].y;
      ff_acc(N.A[i], u[0], c);
      ff_acc(N.W1[i], o.W1, c);
      ff_acc(N.W2[i], o.W2, c);
      ff_acc(N.L[i], o.L, c);
      FF t[5];
      split2_terms(C.kap, N.A[i], N.W1[i], N.W2[i], N.L[i], t);
#pragma unroll
      for (int e = 0; e < 5; e++) ff_acc(q[e], t[e], wt);
    }
    constexpr FF iq = split_ilq(p);
#pragma unroll
    for (int e = 0; e < 5; e++) q[e] = ff_mul(ff_norm(q[e]), iq);
    split2_rem(C, N.v, N.w, u, o, q, F, G);
  }
}

// Order k of a node in float (F, G high parts only).
template <int p>
__device__ __forceinline__ void split2_tail(const Split2Const &C, Split2Node<p> &N, int k, const float2 *lv, const Split2Slots &x,
                                            int i0, int j0, int js, const float *gx, const float *gy, float lx,
                                            float ly, FF *F, FF *G) {
  constexpr int n = 2 * p;
  float a[4] = {0.0f, 0.0f, 0.0f, 0.0f}, b[4] = {0.0f, 0.0f, 0.0f, 0.0f}, u[4];
#pragma unroll
  for (int r = 0; r < n; r++) {
    const float4 f = x.Fh[i0 + r], g = x.Gh[j0 + r * js];
    a[0] = fmaf(gx[r], f.x, a[0]);
    a[1] = fmaf(gx[r], f.y, a[1]);
    a[2] = fmaf(gx[r], f.z, a[2]);
    a[3] = fmaf(gx[r], f.w, a[3]);
    b[0] = fmaf(gy[r], g.x, b[0]);
    b[1] = fmaf(gy[r], g.y, b[1]);
    b[2] = fmaf(gy[r], g.z, b[2]);
    b[3] = fmaf(gy[r], g.w, b[3]);
  }
#pragma unroll
  for (int c = 0; c < 4; c++) u[c] = fmaf(ly, b[c], __fmul_rn(lx, a[c]));
  const float v = N.v.h, w = N.w.h, h = N.h.h, kap = C.kap.h, gm1 = C.gm1.h;
  const float W1 = fmaf(-v, u[0], u[1]), W2 = fmaf(-w, u[0], u[2]);
  const float m1 = __fmul_rn(v, __fadd_rn(u[1], W1)), m2 = __fmul_rn(w, __fadd_rn(u[2], W2));
  const float dp = fmaf(gm1, u[3], __fmul_rn(-kap, __fadd_rn(m1, m2)));
  const float Lp = __fadd_rn(u[3], dp), L1 = fmaf(-h, u[0], Lp);
  split2_bounds(N, lv, u[0], W1, W2, L1);
  float q[5];
  split2_levels(N, kap, k, lv, u[0], W1, W2, L1, q);
  if (k == 3) {  // the leading terms (0 in form 0)
#pragma unroll
    for (int e = 0; e < 5; e++) q[e] = __fadd_rn(q[e], N.q1[e]);
  }
  const float kq = __fmul_rn(kap, __fadd_rn(q[0], q[2]));
  F[0].h = u[1];
  F[1].h = __fadd_rn(__fadd_rn(m1, dp), __fsub_rn(q[0], kq));
  F[2].h = __fadd_rn(fmaf(w, u[1], __fmul_rn(v, W2)), q[1]);
  F[3].h = __fadd_rn(fmaf(h, W1, __fmul_rn(v, Lp)), fmaf(-v, kq, q[3]));
  G[0].h = u[2];
  G[1].h = F[2].h;
  G[2].h = __fadd_rn(__fadd_rn(m2, dp), __fsub_rn(q[2], kq));
  G[3].h = __fadd_rn(fmaf(h, W2, __fmul_rn(w, Lp)), fmaf(-w, kq, q[4]));
#pragma unroll
  for (int c = 0; c < 4; c++) F[c].l = G[c].l = 0.0f;
}

// The flux sums: one thread per (direction, component) of a block adds
// (840 / k) sum_r gh_r F^(k-1)_r/(k-1)! over the row j2 = 0 (direction 0) or the
// column j1 = 0 from the slots; i0, st: first slot and stride.
template <int p>
__device__ __forceinline__ void split2_flux(const Split2Slots &x, const SplitTab &tab, int dir, int c, int i0,
                                            int st, float ck, FF &S) {
  const float *H = reinterpret_cast<const float *>(dir ? x.Gh : x.Fh);
  const float *Lo = reinterpret_cast<const float *>(dir ? x.Gl : x.Fl);
  FF t{0.0f, 0.0f};
#pragma unroll
  for (int r = 0; r < 2 * p; r++) {
    const int i = (i0 + r * st) * 4 + c;
    ff_acc(t, FF{H[i], Lo[i]}, tab.gh[p - 2][r]);
  }
  ff_acc(S, ff_norm(t), ck);
}

}  // namespace
