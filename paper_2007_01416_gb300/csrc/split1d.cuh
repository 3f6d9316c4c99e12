// split1d.cuh -- the FP64 CAT2p flux of the nonlinear 1D laws on the FP32 pipes.
//
// The FP64 pipe of sm_103a issues two fused multiply-adds per SM and cycle, the
// FP32 pipes 128. The CAT2p recursion (Sec. 2.2) costs some 1000 FP64
// instructions per node at p = 4, so an FP64 step is bound by that pipe alone.
// Here the recursion runs in float-float pairs (an unevaluated sum of two
// floats, about 2^-46 relative) on flux increments, which reaches FP64 accuracy
// because the increments are small against the flux itself:
//
//  1. F = f(u_i) + G, and every term of G is built from increments (as the FP32
//     path does): f(u_j) - f(u_i), and f(u_j + d) - f(u_j) at the time levels.
//  2. f(u + d) - f(u) = A(u) d + q(u; d), with A the flux Jacobian and q the
//     remainder in closed form, quadratic in d. The time-derivative weights
//     gamma^{k-1,0}_r are exact on polynomials of degree <= 2p-1 in r, and the
//     Taylor sum d_r = sum_l r^l/l! U^(l) of order k has degree k-1, so
//         sum_r gamma^{k-1,0}_r A d_r = A U^(k-1):
//     one Jacobian product per order replaces the linear part of all 2p-1 time
//     levels, and only q is evaluated level by level. For Euler, with
//     W = b - v a, L = dH' - h a (d = (a, b, e), v = m/rho, h = H/rho):
//         dv = W / (rho + a),  Q = W dv,  T = dv (L - kappa Q),
//         q = (0, (1 - kappa) Q, T - kappa v Q),  kappa = (gamma - 1)/2.
//  3. The rational weights are used as integers (exact in float) with one
//     common denominator per sum: g1 x LC, gamma^{k}/k! x LQ, gh x LH.
//  4. Precision by magnitude. With all increments below TAU = 2^-5 of the local
//     flux scales the float-float error is below the FP64 kernel's own rounding
//     (CPU experiments against 64-bit-mantissa arithmetic, rms error in units of
//     2^-53 of the flux scale at increments of 2^-5: 0.25 against 0.40 of the FP64
//     recursion at p = 4, 0.19 against 0.32 at p = 2; equal at 2^-3.5). Above TAU
//     the caller evaluates the recursion in FP64. The remainders take one of
//     three forms, by the size of the Taylor sums (time increments):
//       0  in float, where the quadratic terms are below 2^-23 of the scales (Burgers:
//          2^-25 of u^2);
//       1  (2D blocks; in 1D it was slower than form 2: P = 4 at N = 262144
//          261 -> 280 us a step) their leading term exactly, the rest in float: with d_r = r d_1 + d'_r,
//          the products r^2 d_1 d_1 / rho are polynomials of degree 2 in r, so
//          their weighted sum is d_1 d_1 / rho at k = 3 and 0 otherwise (one pair);
//          what is left is cubic, or carries the small d', and is formed without
//          cancellation. For cubic terms below 2^-27 and d' d_1 below 2^-25;
//       2  in pairs.
//     From the order on at which F^(k-2) is below 2^-28 of the scales the sums
//     are float too (forms 0 and 1). All leave the measured error unchanged
//     (0.19-0.22). Each decision is taken per interface (2D: per block), by a vote of
//     its lanes, against scales of its own nodes, and checked against bounds of all
//     Taylor sums at the end.
//
// What bounds it: instruction issue and the latency of dependent FP32 operations (a
// pair operation is a chain of 4 to 11), at 14 warps per SM 0.6 instructions per
// cycle and scheduler. P = 4, N = 16384, Euler: 283 us a step in FP64, 25.7 here
// (P = 3 144 -> 22.0, P = 2 43.7 -> 17.1).
#pragma once

#include "phys1d.cuh"

static __device__ SplitTab g_split;  // uploaded beside c_tab

namespace {

// The table to shared memory by the first threads of a CTA (at least 64).
__device__ __forceinline__ void split_tab(SplitTab &t, int tid, int nthreads) {
  const float4 *src = reinterpret_cast<const float4 *>(&g_split);
  float4 *dst = reinterpret_cast<float4 *>(&t);
  for (int q = tid; q < (int)(sizeof(SplitTab) / 16); q += nthreads) dst[q] = __ldg(&src[q]);
}

// ---- float-float arithmetic (Knuth's TwoSum, Dekker's Fast2Sum, TwoProd by FMA) ----
__device__ __forceinline__ FF ff_two(float a, float b) {
  const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
  return FF{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ FF ff_fast(float a, float b) {  // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return FF{s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ FF ff_norm(FF a) { return ff_fast(a.h, a.l); }
__device__ __forceinline__ FF ff_neg(FF a) { return FF{-a.h, -a.l}; }
__device__ __forceinline__ FF ff_add(FF a, FF b) {
  const FF s = ff_two(a.h, b.h);
  return ff_fast(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ FF ff_addf(FF a, float b) {
  const FF s = ff_two(a.h, b);
  return ff_fast(s.h, __fadd_rn(s.l, a.l));
}
// Products and running sums leave their low part unnormalised (a few units of the
// high part's last place), which the operations below allow for; ff_add
// normalises, as its operands may cancel.
__device__ __forceinline__ FF ff_mul(FF a, FF b) {
  const float p = __fmul_rn(a.h, b.h);
  return FF{p, fmaf(a.l, b.h, fmaf(a.h, b.l, fmaf(a.h, b.h, -p)))};
}
__device__ __forceinline__ FF ff_mulf(FF a, float g) {
  const float p = __fmul_rn(a.h, g);
  return FF{p, fmaf(a.l, g, fmaf(a.h, g, -p))};
}
// s += x g
__device__ __forceinline__ void ff_acc(FF &s, FF x, float g) {
  const float p = __fmul_rn(x.h, g);
  const float e = fmaf(x.h, g, -p);
  const FF t = ff_two(s.h, p);
  s.h = t.h;
  s.l = __fadd_rn(fmaf(x.l, g, __fadd_rn(s.l, t.l)), e);
}
// w / d with d's approximate reciprocal r
__device__ __forceinline__ FF ff_quot(FF w, FF d, float r) {
  const float q = __fmul_rn(w.h, r);
  return FF{q, __fmul_rn(__fadd_rn(fmaf(-q, d.h, w.h), fmaf(-q, d.l, w.l)), r)};
}
__device__ __forceinline__ FF ff_bits(double x) {
  const Bits64 b = bits_of(x);
  return FF{__uint_as_float(b.hi), __fmul_rn(small_float((b.lo + 32u) >> 6), __fmul_rn(64.0f, b.ulp))};
}
__device__ __forceinline__ FF ff_of(float2 a) { return FF{a.x, a.y}; }

// An FP64 value as three floats h + m + l (exact for values in float's range),
// and the difference of two such values as a pair.
struct F3 {
  float h, m, l;
};
__device__ __forceinline__ F3 f3_from(double x) {
  const Bits64 b = bits_of(x);
  return F3{__uint_as_float(b.hi), __fmul_rn(small_float(b.lo >> 14), __fmul_rn(16384.0f, b.ulp)),
            __fmul_rn(small_float(b.lo & 0x3fffu), b.ulp)};
}
__device__ __forceinline__ FF f3_diff(F3 a, F3 b) {
  const FF s = ff_two(a.h, -b.h), t = ff_two(a.m, -b.m), w = ff_two(s.h, t.h);
  return ff_fast(w.h, __fadd_rn(w.l, __fadd_rn(s.l, __fadd_rn(t.l, __fsub_rn(a.l, b.l)))));
}

// Common denominators of the integer weights (index p).
__device__ __forceinline__ constexpr float split_lq(int p) { return p == 4 ? 5040.0f : p == 3 ? 120.0f : 6.0f; }
__device__ __forceinline__ constexpr FF split_ilq(int p) {  // 1 / LQ
  return FF{(float)(1.0 / (double)split_lq(p)),
            (float)(1.0 / (double)split_lq(p) - (double)(float)(1.0 / (double)split_lq(p)))};
}
// 1 / (840 LH): the flux sums carry 840 / k and gh x LH
__device__ __forceinline__ double split_ginv(int p) {
  return p == 4 ? 1.0 / (840.0 * 840.0) : p == 3 ? 1.0 / (840.0 * 60.0) : 1.0 / (840.0 * 12.0);
}

constexpr float SPLIT_TAU = 0x1p-5f;    // increments, of the local scales
constexpr float SPLIT_QUAD = 0x1p-23f;  // quadratic terms that float carries
constexpr float SPLIT_QUADB = 0x1p-25f;  // the same for Burgers, against u^2 (the flux is half of it)
constexpr float SPLIT_CUB = 0x1p-27f;   // form 1: cubic terms that float carries,
constexpr float SPLIT_MIX = 0x1p-25f;   // and products of the first-order and the further terms
constexpr float SPLIT_ADJ = 0x1p-8f;    // increments at which the adjoint takes its Jacobians from pairs
constexpr float SPLIT_ADJ_H = 0x1p40f;  // and the largest h whose products with a cotangent they carry
constexpr float SPLIT_TAIL = 0x1p-28f;  // F^(k-2) from which on float suffices

// Whether the cubic terms W W max(a, W) and W L max(a, W) are below SPLIT_CUB of
// the scales (a of rho, w of rs, l of rh).
__device__ __forceinline__ bool split_cubic(float a, float w, float l, float rho, float rs, float rh) {
  const float x = __fmul_rn(a, recip(rho)), y = __fmul_rn(w, recip(rs)), z = __fmul_rn(l, recip(rh));
  return __fmul_rn(__fmul_rn(y, fmaxf(y, z)), fmaxf(x, y)) <= SPLIT_CUB;
}

// A scale that the pairs carry: their low parts (2^-53 of it) stay normal floats
// and so do products of two scales.
__device__ __forceinline__ bool split_range(float x) { return x > 0x1p-42f && x < 0x1p60f; }

// Per-cell records of a staged tile of TW cells (what a stencil node needs,
// computed once per cell instead of once per interface and node).
template <int FLUX, int TW>
struct SplitRec {};
template <int TW>
struct SplitRec<ACAT_FLUX_BURGERS, TW> {
  float2 u[TW];  // u as a pair
  float4 f[TW];  // f as three floats
};
template <int TW>
struct SplitRec<ACAT_FLUX_EULER1D, TW> {
  double fd[3][TW];  // f(u)
  // [0] rho, v; [1] h, s, f_0 low; [2] f high, f_1 low; [3] f middle, f_2 low.
  // s = sqrt(h) is the velocity scale (NaN outside the range float-float
  // carries with margin: the recursion is then evaluated in FP64)
  float4 q[4][TW];
};

template <int FLUX, int TW>
__device__ __forceinline__ void split_record(SplitRec<FLUX, TW> &r, int k, const double *u, double gm1,
                                             double *v_out = nullptr, double *h_out = nullptr) {
  if constexpr (FLUX == ACAT_FLUX_BURGERS) {
    const FF w = ff_bits(u[0]);
    const F3 f = f3_from(__dmul_rn(__dmul_rn(0.5, u[0]), u[0]));
    r.u[k] = make_float2(w.h, w.l);
    r.f[k] = make_float4(f.h, f.m, f.l, 0.0f);
  } else if constexpr (FLUX == ACAT_FLUX_EULER1D) {
    const double ri = recip(u[0]);
    const double v = __dmul_rn(u[1], ri);
    const double p = __dmul_rn(gm1, fma(__dmul_rn(-0.5, u[1]), v, u[2]));
    const double H = __dadd_rn(u[2], p), h = __dmul_rn(H, ri);
    const double f1 = fma(u[1], v, p), f2 = __dmul_rn(v, H);
    if (v_out) *v_out = v;
    if (h_out) *h_out = h;
    r.fd[0][k] = u[1];
    r.fd[1][k] = f1;
    r.fd[2][k] = f2;
    const FF R = ff_bits(u[0]), V = ff_bits(v), Hh = ff_bits(h);
    const F3 a = f3_from(u[1]), b = f3_from(f1), c = f3_from(f2);
    const float s0 = __fsqrt_rn(Hh.h), m0 = __fmul_rn(R.h, s0), m1 = __fmul_rn(R.h, Hh.h), m2 = __fmul_rn(m1, s0);
    const bool fine = split_range(R.h) && split_range(Hh.h) && split_range(m0) && split_range(m1) && split_range(m2);
    const float s = fine ? s0 : __int_as_float(0x7fffffff);
    r.q[0][k] = make_float4(R.h, R.l, V.h, V.l);
    r.q[1][k] = make_float4(Hh.h, Hh.l, s, a.l);
    r.q[2][k] = make_float4(a.h, b.h, c.h, b.l);
    r.q[3][k] = make_float4(a.m, b.m, c.m, c.l);
  }
}

// -lambda / ((k-1) LC) as pairs, k = 2..2p, for p = 2..P: entry [p-2][k-2].
struct SplitLam {
  float2 v[3][7];
};
__device__ __forceinline__ void split_lam(SplitLam &s, double lam, int t) {
  if (t < 21) {
    const int p = 2 + t / 7, k1 = t - (p - 2) * 7 + 1;
    const FF x = ff_bits(__dmul_rn(-lam, c_tab.ilc[p][k1]));
    s.v[p - 2][k1 - 1] = make_float2(x.h, x.l);
  }
}

// Sum of a pair over the n lanes of a group (lane l, first lane base); lane
// `base` holds the result (every lane at n = 4, 8).
template <int n>
__device__ __forceinline__ FF split_sum(unsigned mask, int base, int l, FF t) {
  if constexpr (n == 6) {
    const int o = base + (l < 3 ? l + 3 : l - 3);
    t = ff_add(t, FF{__shfl_sync(mask, t.h, o), __shfl_sync(mask, t.l, o)});
    const int o1 = base + (l + 1) % 6, o2 = base + (l + 2) % 6;
    const FF a{__shfl_sync(mask, t.h, o1), __shfl_sync(mask, t.l, o1)};
    const FF b{__shfl_sync(mask, t.h, o2), __shfl_sync(mask, t.l, o2)};
    return ff_add(ff_add(t, a), b);
  } else {
#pragma unroll
    for (int w = 1; w < n; w <<= 1)
      t = ff_add(t, FF{__shfl_sync(mask, t.h, base + (l ^ w)), __shfl_sync(mask, t.l, base + (l ^ w))});
    return t;
  }
}

// G x (840 LH) of one Euler interface by a group of 2p lanes (lane l <-> node
// l - p + 1); ic: tile index of cell i. xa, xb: the group's exchange slots (two
// sets XSET apart). Returns whether the float-float recursion holds (uniform in
// the group); G is in lane `base`. ADJ: keeps the node's U^(k-1)/(k-1)! as
// (a, W, L) in xst, pair e of order k at xst[((k - 2) 6 + e) 32], and takes the
// tighter bound SPLIT_ADJ; no flux.
template <int p, int TW, bool ADJ = false>
__device__ __forceinline__ bool cat_split_euler(const SplitRec<ACAT_FLUX_EULER1D, TW> &rec, const Step1DArgs &a,
                                                const SplitTab &tab, const float2 *lamk, int ic, int l, int base,
                                                float4 *xa, float2 *xb, FF *G, float *xst = nullptr) {
  constexpr int n = 2 * p, NL = n - 1;
  const unsigned mask = ((1u << n) - 1u) << base;
  const FF gam = ff_of(a.sgam), kap = ff_of(a.skap), omk = ff_of(a.somk), gm = ff_of(a.sgm1);
  float g1r[n];
#pragma unroll
  for (int r = 0; r < n; r++) g1r[r] = tab.g1[p - 2][l][r];
  const int jc = ic + l - p + 1;
  const float4 q0 = rec.q[0][jc], q1 = rec.q[1][jc];
  const FF rho{q0.x, q0.y}, v{q0.z, q0.w}, h{q1.x, q1.y};
  const float rs = __fmul_rn(rho.h, q1.z), rh = __fmul_rn(rho.h, h.h), rhs = __fmul_rn(rh, q1.z);
  FF Y[3], S[3];
  {
    const float4 q2 = rec.q[2][jc], q3 = rec.q[3][jc], a1 = rec.q[1][ic], a2 = rec.q[2][ic], a3 = rec.q[3][ic];
    Y[0] = f3_diff(F3{q2.x, q3.x, q1.w}, F3{a2.x, a3.x, a1.w});
    Y[1] = f3_diff(F3{q2.y, q3.y, q2.w}, F3{a2.y, a3.y, a2.w});
    Y[2] = f3_diff(F3{q2.z, q3.z, q3.w}, F3{a2.z, a3.z, a3.w});
  }
  if (!__all_sync(mask, fabsf(Y[0].h) <= SPLIT_TAU * rs && fabsf(Y[1].h) <= SPLIT_TAU * rh &&
                            fabsf(Y[2].h) <= SPLIT_TAU * rhs))
    return false;
  const FF kv = ff_mul(kap, v);
  const FF Y0[3] = {Y[0], Y[1], Y[2]};
  bool allow = true;  // float remainders not yet ruled out
#pragma unroll 1
  for (;;) {
    FF A[NL], W[NL], L[NL];
#pragma unroll
    for (int q = 0; q < NL; q++) {
      A[q] = rho;
      W[q] = FF{0.0f, 0.0f};
      L[q] = FF{0.0f, 0.0f};
    }
#pragma unroll
    for (int c = 0; c < 3; c++) {
      Y[c] = Y0[c];
      S[c] = FF{0.0f, 0.0f};
      ff_acc(S[c], Y[c], 840.0f);
    }
    bool flt = allow, tail = false;
    float Ba = 0.0f, Bw = 0.0f, Bl = 0.0f;  // bounds of the Taylor sums
#pragma unroll 1
    for (int k = 2; k <= n; k++) {
      const float2 lk = lamk[k - 2];
      const float2 *lv = tab.lv[p - 2][k - 2];
      const float pk = lv[NL - 1].x, ck = tab.k840[k - 1];  // p^(k-1), 840 / k
      float4 *xs = xa + (k & 1) * XSET;
      if (!tail && flt)
        tail = __all_sync(mask, fabsf(Y[0].h) <= SPLIT_TAIL * rs && fabsf(Y[1].h) <= SPLIT_TAIL * rh &&
                                    fabsf(Y[2].h) <= SPLIT_TAIL * rhs);
      if (tail) {
        xs[l] = make_float4(Y[0].h, Y[1].h, Y[2].h, 0.0f);
        __syncwarp(mask);
        float u0 = 0.0f, u1 = 0.0f, u2 = 0.0f;
#pragma unroll
        for (int r = 0; r < n; r++) {
          const float4 y = xs[r];
          u0 = fmaf(g1r[r], y.x, u0);
          u1 = fmaf(g1r[r], y.y, u1);
          u2 = fmaf(g1r[r], y.z, u2);
        }
        u0 = __fmul_rn(u0, lk.x);
        u1 = __fmul_rn(u1, lk.x);
        u2 = __fmul_rn(u2, lk.x);
        const float w = fmaf(-v.h, u0, u1), s = __fmul_rn(v.h, __fadd_rn(u1, w));
        const float Lp = fmaf(gam.h, u2, __fmul_rn(-kap.h, s)), L1 = fmaf(-h.h, u0, Lp);
        Ba = fmaf(pk, fabsf(u0), Ba);
        Bw = fmaf(pk, fabsf(w), Bw);
        Bl = fmaf(pk, fabsf(L1), Bl);
        if constexpr (ADJ) {
          float *q = xst + (k - 2) * 6 * 32;
          q[0] = u0;
          q[64] = w;
          q[128] = L1;
          q[32] = q[96] = q[160] = 0.0f;
        }
        float sq = 0.0f, st = 0.0f;
#pragma unroll
        for (int q = 0; q < NL; q++) {
          const float c = lv[q].x, wt = lv[q].y;
          A[q].h = fmaf(c, u0, A[q].h);
          W[q].h = fmaf(c, w, W[q].h);
          L[q].h = fmaf(c, L1, L[q].h);
          const float dv = __fmul_rn(W[q].h, recip(A[q].h)), Q = __fmul_rn(W[q].h, dv);
          sq = fmaf(wt, Q, sq);
          st = fmaf(wt, __fmul_rn(dv, fmaf(-kap.h, Q, L[q].h)), st);
        }
        sq = __fmul_rn(sq, 1.0f / split_lq(p));
        st = __fmul_rn(st, 1.0f / split_lq(p));
        Y[0].h = u1;
        Y[1].h = fmaf(omk.h, __fadd_rn(s, sq), __fmul_rn(gm.h, u2));
        Y[2].h = __fadd_rn(fmaf(v.h, Lp, __fmul_rn(h.h, w)), fmaf(-kv.h, sq, st));
#pragma unroll
        for (int c = 0; c < 3; c++) S[c].l = fmaf(ck, Y[c].h, S[c].l);
        continue;
      }
      float2 *xt = xb + (k & 1) * XSET;
      xs[l] = make_float4(Y[0].h, Y[1].h, Y[2].h, Y[0].l);
      xt[l] = make_float2(Y[1].l, Y[2].l);
      __syncwarp(mask);
      FF u[3] = {FF{0.0f, 0.0f}, FF{0.0f, 0.0f}, FF{0.0f, 0.0f}};
#pragma unroll
      for (int r = 0; r < n; r++) {
        const float4 y = xs[r];
        const float2 z = xt[r];
        ff_acc(u[0], FF{y.x, y.w}, g1r[r]);
        ff_acc(u[1], FF{y.y, z.x}, g1r[r]);
        ff_acc(u[2], FF{y.z, z.y}, g1r[r]);
      }
#pragma unroll
      for (int c = 0; c < 3; c++) u[c] = ff_mul(ff_norm(u[c]), FF{lk.x, lk.y});
      const FF w = ff_add(u[1], ff_neg(ff_mul(v, u[0])));
      const FF s = ff_mul(v, ff_add(u[1], w));
      const FF Lp = ff_add(ff_mul(gam, u[2]), ff_neg(ff_mul(kap, s)));
      const FF L1 = ff_add(Lp, ff_neg(ff_mul(h, u[0])));
      Ba = fmaf(pk, fabsf(u[0].h), Ba);
      Bw = fmaf(pk, fabsf(w.h), Bw);
      Bl = fmaf(pk, fabsf(L1.h), Bl);
      if constexpr (ADJ) {
        float *q = xst + (k - 2) * 6 * 32;
        q[0] = u[0].h;
        q[32] = u[0].l;
        q[64] = w.h;
        q[96] = w.l;
        q[128] = L1.h;
        q[160] = L1.l;
        // the bounds only grow: a coarse grid leaves for the FP64 sweep before the recursion
        // (at p = 2 the vote cost what it saved)
        if (p >= 3 && k == 2 && !__all_sync(mask, Ba <= SPLIT_ADJ * rho.h && Bw <= SPLIT_ADJ * rs && Bl <= SPLIT_ADJ * rh))
          return false;
      }
      if (k == 2 && flt) {  // float remainders, by the first-order increments with a margin of 4
        const float bw = 2.0f * Bw, bl = 2.0f * Bl;
        flt = __all_sync(mask, bw * bw <= SPLIT_QUAD * rs * rs && bw * bl <= SPLIT_QUAD * rs * rh);
      }
      FF y1 = ff_add(ff_mul(omk, s), ff_mul(gm, u[2])), y2 = ff_add(ff_mul(h, w), ff_mul(v, Lp));
      if (flt) {
        float sq = 0.0f, st = 0.0f;
#pragma unroll
        for (int q = 0; q < NL; q++) {
          const float c = lv[q].x, wt = lv[q].y;
          A[q].h = fmaf(c, u[0].h, A[q].h);
          W[q].h = fmaf(c, w.h, W[q].h);
          L[q].h = fmaf(c, L1.h, L[q].h);
          const float dv = __fmul_rn(W[q].h, recip(A[q].h)), Q = __fmul_rn(W[q].h, dv);
          sq = fmaf(wt, Q, sq);
          st = fmaf(wt, __fmul_rn(dv, fmaf(-kap.h, Q, L[q].h)), st);
        }
        sq = __fmul_rn(sq, 1.0f / split_lq(p));
        st = __fmul_rn(st, 1.0f / split_lq(p));
        y1 = ff_addf(y1, __fmul_rn(omk.h, sq));
        y2 = ff_addf(y2, fmaf(-kv.h, sq, st));
      } else {
        FF sq{0.0f, 0.0f}, st{0.0f, 0.0f};
#pragma unroll
        for (int q = 0; q < NL; q++) {
          const float c = lv[q].x, wt = lv[q].y;
          ff_acc(A[q], u[0], c);
          ff_acc(W[q], w, c);
          ff_acc(L[q], L1, c);
          const FF dv = ff_quot(W[q], A[q], recip(A[q].h));
          const FF Q = ff_mul(W[q], dv);
          const FF T = ff_mul(dv, ff_add(L[q], ff_neg(ff_mul(kap, Q))));
          ff_acc(sq, Q, wt);
          ff_acc(st, T, wt);
        }
        constexpr FF iq = split_ilq(p);
        sq = ff_mul(ff_norm(sq), iq);
        st = ff_mul(ff_norm(st), iq);
        y1 = ff_add(y1, ff_mul(omk, sq));
        y2 = ff_add(y2, ff_add(st, ff_neg(ff_mul(kv, sq))));
      }
      Y[0] = u[1];
      Y[1] = y1;
      Y[2] = y2;
#pragma unroll
      for (int c = 0; c < 3; c++) ff_acc(S[c], Y[c], ck);
    }
    constexpr float tau = ADJ ? SPLIT_ADJ : SPLIT_TAU;
    const bool small = Ba <= tau * rho.h && Bw <= tau * rs && Bl <= tau * rh;
    if (!__all_sync(mask, small && (!ADJ || h.h < SPLIT_ADJ_H))) return false;
    if (!flt || __all_sync(mask, Bw * Bw <= SPLIT_QUAD * rs * rs && Bw * Bl <= SPLIT_QUAD * rs * rh)) break;
    allow = false;  // the remainders grew past float: once more with pairs
  }
  if constexpr (ADJ) return true;
  const float gw = tab.gh[p - 2][l];
#pragma unroll
  for (int c = 0; c < 3; c++) G[c] = split_sum<n>(mask, base, l, ff_mulf(ff_norm(S[c]), gw));
  return true;
}

// The same for Burgers, f = u^2 / 2: A = u, q = d^2 / 2. The velocity scale is the
// largest |u| of the stencil itself. (Taken from dt, as cfl / lambda, it is the largest
// |u| of the grid, or more where dt is imposed: then regions of small |u| pass with
// increments of their own size, and lambda F is off by 20 x 2^-53 of the |u| there.)
// Error of F in 2^-53 of the scale u^2 / 2, over waves a + b sin with 60 to 40000 cells
// a period, dt of CFL / 1000 to CFL and local scales of 1 to 1/64 of the largest |u|,
// CPU experiments against 64-bit mantissas: rms 0.6-0.7 (FP64 recursion 1.3-1.8), largest 3.7
// (8.6).
template <int p, int TW>
__device__ __forceinline__ bool cat_split_burgers(const SplitRec<ACAT_FLUX_BURGERS, TW> &rec, const SplitTab &tab,
                                                  const float2 *lamk, int ic, int l, int base, FF *G) {
  constexpr int n = 2 * p, NL = n - 1;
  const unsigned mask = ((1u << n) - 1u) << base;
  float g1r[n], vs = 0.0f;
#pragma unroll
  for (int r = 0; r < n; r++) {
    g1r[r] = tab.g1[p - 2][l][r];
    vs = fmaxf(vs, fabsf(rec.u[ic - p + 1 + r].x));  // a NaN fails the vote on its Y0
  }
  const int jc = ic + l - p + 1;
  const FF uj = ff_of(rec.u[jc]);
  const float4 fj = rec.f[jc], fi = rec.f[ic];
  const FF Y0 = f3_diff(F3{fj.x, fj.y, fj.z}, F3{fi.x, fi.y, fi.z});
  const float v2 = __fmul_rn(vs, vs);
  if (!__all_sync(mask, split_range(vs) && split_range(v2) && fabsf(Y0.h) <= SPLIT_TAU * v2)) return false;
  FF S;
  bool allow = true;
#pragma unroll 1
  for (;;) {
    FF D[NL], Y = Y0;
#pragma unroll
    for (int q = 0; q < NL; q++) D[q] = FF{0.0f, 0.0f};
    S = FF{0.0f, 0.0f};
    ff_acc(S, Y, 840.0f);
    bool flt = allow;
    float B = 0.0f;
#pragma unroll 1
    for (int k = 2; k <= n; k++) {
      const float2 lk = lamk[k - 2], *lv = tab.lv[p - 2][k - 2];
      FF u{0.0f, 0.0f};
#pragma unroll
      for (int r = 0; r < n; r++)
        ff_acc(u, FF{__shfl_sync(mask, Y.h, base + r), __shfl_sync(mask, Y.l, base + r)}, g1r[r]);
      u = ff_mul(ff_norm(u), FF{lk.x, lk.y});
      B = fmaf(lv[NL - 1].x, fabsf(u.h), B);
      if (k == 2) {
        if (!__all_sync(mask, B <= SPLIT_TAU * vs)) return false;  // as at the end
        if (flt) flt = __all_sync(mask, 4.0f * B * B <= SPLIT_QUADB * v2);
      }
      Y = ff_mul(uj, u);
      if (flt) {
        float sq = 0.0f;
#pragma unroll
        for (int q = 0; q < NL; q++) {
          D[q].h = fmaf(lv[q].x, u.h, D[q].h);
          sq = fmaf(lv[q].y, __fmul_rn(D[q].h, D[q].h), sq);
        }
        Y = ff_addf(Y, __fmul_rn(sq, 0.5f / split_lq(p)));
      } else {
        FF sq{0.0f, 0.0f};
#pragma unroll
        for (int q = 0; q < NL; q++) {
          ff_acc(D[q], u, lv[q].x);
          ff_acc(sq, ff_mul(D[q], D[q]), lv[q].y);
        }
        constexpr FF iq = split_ilq(p);
        sq = ff_mul(ff_norm(sq), iq);
        Y = ff_add(Y, FF{0.5f * sq.h, 0.5f * sq.l});
      }
      ff_acc(S, Y, tab.k840[k - 1]);
    }
    if (!__all_sync(mask, B <= SPLIT_TAU * vs)) return false;
    if (!flt || __all_sync(mask, B * B <= SPLIT_QUADB * v2)) break;
    allow = false;
  }
  G[0] = split_sum<n>(mask, base, l, ff_mulf(ff_norm(S), tab.gh[p - 2][l]));
  return true;
}

// Linear transport: f is linear, so F^(k-1)_j = a U^(k-1)_j with no time
// levels; the recursion is 2p FMAs per order and stays in FP64.
template <int p>
__device__ __forceinline__ double cat_linear(const double *q, int l, int base, double lam, double adv) {
  constexpr int n = 2 * p;
  const unsigned mask = ((1u << n) - 1u) << base;
  double g1r[n];
  const double m = __dmul_rn(-lam, adv);
#pragma unroll
  for (int r = 0; r < n; r++) g1r[r] = __dmul_rn(c_tab.g1[p][l][r], m);
  double Y = __dmul_rn(adv, q[l - p + 1]), S = Y;
#pragma unroll
  for (int k = 2; k <= n; k++) {
    double u = 0.0;
#pragma unroll
    for (int r = 0; r < n; r++) u = fma(g1r[r], __shfl_sync(mask, Y, base + r), u);
    Y = u;
    S = fma(c_tab.invfact[k], Y, S);
  }
  const double w = __dmul_rn(c_tab.gh[p][l], S);
  double t = __shfl_sync(mask, w, base);
#pragma unroll
  for (int r = 1; r < n; r++) t = __dadd_rn(t, __shfl_sync(mask, w, base + r));
  return t;
}

}  // namespace
