// The double-float evaluator of the source-plane chi2 and of the image search's
// Newton steps: dPIE, SIS and point mass at one image, or at two side by side.
//
// Its roundings are fixed.  A set with an image next to a critical curve
// divides by det ~ 1e-5 and smaller, which turns an evaluator's last bits
// (~2e-14) into 1e-9 of the chi2 (mu-weighted, 4096 sets x 372 images), so
// this one keeps three-term divisions and renormalises every operation, and
// every shortcut below gives the same bits: FastTwoSum where the larger
// operand is known, differences that are exact by Sterbenz' lemma, sums with
// an exact zero left out, constants of a record formed once per record.
// Newton started next to a fold wanders, so that there too the last bits decide
// whether a borderline image is found (1 of 10^5 images).
// (lens_device.cuh's dpie_df takes 40 % fewer operations, with other bits.)
//
// F is float (one image) or float2 (two: the paired FP32 instructions round
// each component as the scalar ones do).  What bounds the chi2 kernels is
// the latency of one long dependent chain per image on 16 warps per SM: two
// images per thread give two chains, and a potential's record is read once
// for both.
#pragma once

#include "lens_device.cuh"

namespace lens {

// ------------------------------------------------------ float / float2 arithmetic
// (explicit roundings: a product and a sum must not be fused differently in
// the two forms)
__device__ __forceinline__ float f_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float f_sub(float a, float b) { return __fadd_rn(a, -b); }
__device__ __forceinline__ float f_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float f_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float f_neg(float a) { return -a; }
__device__ __forceinline__ float f_rcp(float a) { return rcp_a(a); }
__device__ __forceinline__ float f_rsqrt(float a) { return rsqrt_a(a); }
__device__ __forceinline__ float2 f_add(float2 a, float2 b) { return add2(a, b); }
__device__ __forceinline__ float2 f_sub(float2 a, float2 b) { return sub2(a, b); }
__device__ __forceinline__ float2 f_mul(float2 a, float2 b) { return mul2(a, b); }
__device__ __forceinline__ float2 f_fma(float2 a, float2 b, float2 c) { return fma2(a, b, c); }
__device__ __forceinline__ float2 f_neg(float2 a) { return neg2(a); }
__device__ __forceinline__ float2 f_rcp(float2 a) { return rcp2(a); }
__device__ __forceinline__ float2 f_rsqrt(float2 a) { return rsqrt2(a); }
template <class F>
__device__ __forceinline__ F f_dup(float a);
template <>
__device__ __forceinline__ float f_dup<float>(float a) { return a; }
template <>
__device__ __forceinline__ float2 f_dup<float2>(float a) { return dup2(a); }
// component h of F (h < f_lanes<F>)
template <class F>
constexpr int f_lanes = 1;
template <>
constexpr int f_lanes<float2> = 2;
__device__ __forceinline__ float f_part(float a, int) { return a; }
__device__ __forceinline__ float f_part(float2 a, int h) { return h ? a.y : a.x; }
__device__ __forceinline__ void f_put(float &a, int, float v) { a = v; }
__device__ __forceinline__ void f_put(float2 &a, int h, float v) { part2(a, h) = v; }

template <class F>
struct Df {
  F hi, lo;
};
template <class F>
__device__ __forceinline__ Df<F> d_dup(float hi, float lo) { return {f_dup<F>(hi), f_dup<F>(lo)}; }
// a where m's bit of the component is set, else b
template <class F>
__device__ __forceinline__ Df<F> d_sel(unsigned m, const Df<F> &a, const Df<F> &b) {
  Df<F> r;
#pragma unroll
  for (int h = 0; h < f_lanes<F>; ++h) {
    f_put(r.hi, h, m >> h & 1u ? f_part(a.hi, h) : f_part(b.hi, h));
    f_put(r.lo, h, m >> h & 1u ? f_part(a.lo, h) : f_part(b.lo, h));
  }
  return r;
}
template <class F>
constexpr unsigned f_all = (1u << f_lanes<F>) - 1u;
template <class F>
__device__ __forceinline__ unsigned f_above(F a, float x) {
  unsigned m = 0;
#pragma unroll
  for (int h = 0; h < f_lanes<F>; ++h) m |= (f_part(a, h) > x ? 1u : 0u) << h;
  return m;
}

template <class F>
__device__ __forceinline__ Df<F> d_two(F a, F b) {  // TwoSum
  const F s = f_add(a, b), bb = f_sub(s, a);
  return {s, f_add(f_sub(a, f_sub(s, bb)), f_sub(b, bb))};
}
template <class F>
__device__ __forceinline__ Df<F> d_fast(F a, F b) {  // FastTwoSum
  const F s = f_add(a, b);
  return {s, f_sub(b, f_sub(s, a))};
}
template <class F>
__device__ __forceinline__ Df<F> d_neg(Df<F> a) { return {f_neg(a.hi), f_neg(a.lo)}; }
// the rest of an accurate addition whose high parts' TwoSum is s
template <class F>
__device__ __forceinline__ Df<F> d_add_tail(Df<F> s, F alo, F blo) {
  const Df<F> t = d_two(alo, blo);
  s = d_fast(s.hi, f_add(s.lo, t.hi));
  return d_fast(s.hi, f_add(s.lo, t.lo));
}
template <class F>
__device__ __forceinline__ Df<F> d_add(Df<F> a, Df<F> b) { return d_add_tail(d_two(a.hi, b.hi), a.lo, b.lo); }
template <class F>
__device__ __forceinline__ Df<F> d_sub(Df<F> a, Df<F> b) { return d_add(a, d_neg(b)); }
// a + b with |a| >= |b| or a = 0
template <class F>
__device__ __forceinline__ Df<F> d_add_big(Df<F> a, Df<F> b) { return d_add_tail(d_fast(a.hi, b.hi), a.lo, b.lo); }
// a - b where a.hi - b.hi is exact (b.hi within a factor of two of a.hi)
template <class F>
__device__ __forceinline__ Df<F> d_sub_near(Df<F> a, Df<F> b) {
  const F s = f_sub(a.hi, b.hi);
  const Df<F> t = d_two(a.lo, f_neg(b.lo));
  const Df<F> r = d_fast(s, t.hi);
  return d_fast(r.hi, f_add(r.lo, t.lo));
}
// one-TwoSum addition (df_add_ss); _big: |a| >= |b|
template <class F>
__device__ __forceinline__ Df<F> d_ss(Df<F> a, Df<F> b) {
  const Df<F> s = d_two(a.hi, b.hi);
  return d_fast(s.hi, f_add(s.lo, f_add(a.lo, b.lo)));
}
template <class F>
__device__ __forceinline__ Df<F> d_ss_big(Df<F> a, Df<F> b) {
  const Df<F> s = d_fast(a.hi, b.hi);
  return d_fast(s.hi, f_add(s.lo, f_add(a.lo, b.lo)));
}
template <class F>
__device__ __forceinline__ Df<F> d_mul(Df<F> a, Df<F> b) {
  const F p = f_mul(a.hi, b.hi);
  F e = f_fma(a.hi, b.hi, f_neg(p));
  e = f_fma(a.hi, b.lo, e);
  e = f_fma(a.lo, b.hi, e);
  return d_fast(p, e);
}
template <class F>
__device__ __forceinline__ Df<F> d_mulf(Df<F> a, F b) {
  const F p = f_mul(a.hi, b);
  return d_fast(p, f_fma(a.lo, b, f_fma(a.hi, b, f_neg(p))));
}
// a / b: MUFU reciprocal of b.hi, then two remainders a - b q correct the
// quotient (its first term may be off by a few 2^-24).  Division and the
// polynomial are called, not inlined: the evaluator's code then fits the
// instruction caches (stalls on instruction fetch were 2.3 of 7 per issue;
// 1000 scaled sets 29.2 -> 25.1 -> 21.6 ms with each, 4096 sets x 372 images
// 0.327 -> 0.310 ms).
template <class F>
__device__ __noinline__ Df<F> d_div(Df<F> a, Df<F> b) {
  const F ib = f_rcp(b.hi);
  const F q1 = f_mul(a.hi, ib);
  Df<F> r = d_sub_near(a, d_mulf(b, q1));
  const F q2 = f_mul(r.hi, ib);
  r = d_sub_near(r, d_mulf(b, q2));
  const Df<F> q = d_fast(q1, q2), s = d_two(q.hi, f_mul(r.hi, ib));
  return d_fast(s.hi, f_add(s.lo, q.lo));
}
template <class F>
__device__ __forceinline__ Df<F> d_sqrt(Df<F> a) {  // a > 0 (0 for the components that are not)
  const F y = f_rsqrt(a.hi), s = f_mul(a.hi, y), half = f_mul(f_dup<F>(0.5f), y);
  const F e = f_add(f_fma(f_neg(s), s, a.hi), a.lo), t = f_add(s, f_mul(e, half));
  return d_sel(f_above(a.hi, 0.f), Df<F>{t, f_fma(e, half, f_sub(s, t))}, d_dup<F>(0.f, 0.f));
}
template <class F>
__device__ __noinline__ Df<F> d_poly(Df<F> t, const float (*c)[2]) {
  F tail = f_dup<F>(c[11][0]);
#pragma unroll
  for (int k = 10; k >= 7; --k) tail = f_fma(tail, t.hi, f_dup<F>(c[k][0]));
  Df<F> p = d_ss_big(d_dup<F>(c[6][0], c[6][1]), d_mulf(t, tail));
#pragma unroll
  for (int k = 5; k >= 0; --k) p = d_ss_big(d_dup<F>(c[k][0], c[k][1]), d_mul(p, t));  // |p t| < |c| / 6
  return p;
}
template <class F>
__device__ __forceinline__ unsigned d_abs(Df<F> &a) {  // the components that were negative
  unsigned neg = 0;
#pragma unroll
  for (int h = 0; h < f_lanes<F>; ++h) neg |= (f_part(a.hi, h) < 0.f ? 1u : 0u) << h;
  a = d_sel(neg, d_neg(a), a);
  return neg;
}
// atan(w) and atanh(w) for any argument (|w| < 1 for atanh), by the reductions
// of atan64 / atanh64; atanh is NaN within ~1e-15 of 1.
template <class F>
__device__ __forceinline__ Df<F> d_atan(Df<F> w) {
  const unsigned neg = d_abs(w), inv = f_above(w.hi, 1.f);
  Df<F> v = w, base = d_dup<F>(0.f, 0.f);
  if (inv) v = d_sel(inv, d_div(d_dup<F>(1.f, 0.f), w), w);
  const unsigned shift = f_above(v.hi, 0.4f);
  if (shift) {
    const Df<F> c = d_dup<F>(0.6875f, 0.f);
    v = d_sel(shift, d_div(d_sub(v, c), d_ss_big(d_dup<F>(1.f, 0.f), d_mulf(v, c.hi))), v);
    base = d_sel(shift, d_dup<F>(ATAN_11_16_DF[0], ATAN_11_16_DF[1]), base);
  }
  Df<F> r = d_add_big(base, d_mul(v, d_poly(d_mul(v, v), C_ATAN_DF)));
  if (inv) r = d_sel(inv, d_add_big(d_dup<F>(PI_2_DF[0], PI_2_DF[1]), d_neg(r)), r);
  return d_sel(neg, d_neg(r), r);
}
template <class F>
__device__ __forceinline__ Df<F> d_atanh(Df<F> w) {
  const unsigned neg = d_abs(w), big = f_all<F> & ~[&] {
    unsigned m = 0;
#pragma unroll
    for (int h = 0; h < f_lanes<F>; ++h) m |= (f_part(w.hi, h) <= 0.4f ? 1u : 0u) << h;
    return m;
  }();
  Df<F> v = w, base = d_dup<F>(0.f, 0.f);
  unsigned bad = 0;
  if (big) {
    const Df<F> one = d_dup<F>(1.f, 0.f), om = d_sub(one, w);  // 1 - w, exact enough to pick the centre
    Df<F> c = base, A = base;
#pragma unroll
    for (int h = 0; h < f_lanes<F>; ++h) {
      const float o = f_part(om.hi, h), est = 0.5f * (__logf(1.f + f_part(w.hi, h)) - __logf(o));
      const int k = __float2int_rn(est * 1.25f);
      const bool out = (big >> h & 1u) && (!(o > 0.f) || k > 22);
      bad |= (out ? 1u : 0u) << h;
      const int kk = k < 1 || k > 22 ? 1 : k;
      f_put(c.hi, h, ATANH_C_DF[kk][0]);
      f_put(c.lo, h, ATANH_C_DF[kk][1]);
      f_put(A.hi, h, ATANH_A_DF[kk][0]);
      f_put(A.lo, h, ATANH_A_DF[kk][1]);
    }
    v = d_sel(big, d_div(d_sub(w, c), d_sub(one, d_mul(w, c))), w);
    base = d_sel(big, A, base);
  }
  Df<F> r = d_add_big(base, d_mul(v, d_poly(d_mul(v, v), C_ATANH_DF)));
  if (bad) r = d_sel(bad, d_dup<F>(__int_as_float(0x7fc00000), 0.f), r);
  return d_sel(neg, d_neg(r), r);
}

// The record's constants that this evaluator forms itself: s_t - s_c, b q / 2
// times q^2 (s_t^2 - s_c^2) and, if UW, u and b q / u.
template <bool UW>
__device__ __forceinline__ void record_consts(float2 *r) {
  if (r[F_U2].x < 0.f) return;  // SIS, point mass
  auto D = [&](int k) { return Df<float>{r[k].x, r[k].y}; };
  auto put = [&](int k, Df<float> d) { r[k] = make_float2(d.hi, d.lo); };
  put(F_DS, d_ss(D(F_ST), d_neg(D(F_SC))));
  put(F_KTC, d_mul(D(F_HB), D(F_KTC)));
  if (!UW) return;
  const Df<float> u = d_sqrt(D(F_U2));
  put(F_U, u);
  if (u.hi > 0.f) put(F_BU, d_div(D(F_BQ), u));  // (never used for a circular one)
}

// One dPIE potential (record r after record_consts<UW>, or as it is (RAW, with
// UW = false); shared by the images):
// deflection and, if HESS, kappa, gamma1, gamma2 into h[0..2].  Returns the
// components whose result is finite.
template <bool HESS, bool UW, class F, bool RAW = false>
__device__ __forceinline__ unsigned dpie_fixed(const float2 *__restrict__ r, Df<F> X, Df<F> Y, Df<F> &ax, Df<F> &ay,
                                               Df<F> *h) {
  auto ld = [&](int k) {
    const float2 v = r[k];
    return d_dup<F>(v.x, v.y);
  };
  const Df<F> c = ld(F_C), s = ld(F_S);
  const Df<F> dX = d_sub(X, ld(F_X0)), dY = d_sub(Y, ld(F_Y0));
  const Df<F> x = d_ss(d_mul(c, dX), d_mul(s, dY)), y = d_ss(d_mul(c, dY), d_neg(d_mul(s, dX)));
  const Df<F> u2 = ld(F_U2), x2 = d_mul(x, x), y2 = d_mul(y, y);
  const Df<F> R = d_ss(d_mul(ld(F_Q2), x2), y2);
  const Df<F> psc = d_sqrt(d_ss(R, ld(F_KC))), pst = d_sqrt(d_ss(R, ld(F_KT)));
  const Df<F> Sp = d_ss_big(pst, psc);
  const Df<F> sc = ld(F_SC), st = ld(F_ST);
  const Df<F> dS = RAW ? d_ss(st, d_neg(sc)) : ld(F_DS);
  const Df<F> numx = d_mul(d_mul(x, dS), d_ss(Sp, ld(F_Q2SS)));
  const Df<F> denx = d_mul(Sp, d_ss(d_mul(d_ss(psc, sc), d_ss(pst, st)), d_mul(u2, x2)));
  const Df<F> Zx = d_div(numx, denx);
  const Df<F> numy = d_mul(d_mul(y, ld(F_Q2DS)), d_ss(Sp, ld(F_SS)));
  const Df<F> deny = d_mul(Sp, d_sub(d_mul(d_ss(psc, ld(F_Q2SC)), d_ss(pst, ld(F_Q2ST))), d_mul(u2, y2)));
  const Df<F> Zy = d_div(numy, deny);
  const Df<F> tx = d_mul(u2, d_mul(Zx, Zx)), ty = d_mul(u2, d_mul(Zy, Zy));
  const Df<F> bq = ld(F_BQ);
  unsigned poly = 0, ok = f_all<F>;
#pragma unroll
  for (int k = 0; k < f_lanes<F>; ++k)
    poly |= (f_part(tx.hi, k) < (float)T_SERIES64 && f_part(ty.hi, k) < (float)T_SERIES64 ? 1u : 0u) << k;
  Df<F> axp, ayp;
  if (poly) {  // bq Z atan(w)/w, w = u Z
    axp = d_mul(d_mul(bq, Zx), d_poly(tx, C_ATAN_DF));
    ayp = d_mul(d_mul(bq, Zy), d_poly(ty, C_ATANH_DF));
  }
  if (poly != f_all<F>) {
    Df<float> us = {r[F_U].x, r[F_U].y}, bus = {r[F_BU].x, r[F_BU].y};  // (bq / u) atan(u Z)
    if (!UW) {
      us = d_sqrt(Df<float>{r[F_U2].x, r[F_U2].y});
      bus = d_div(Df<float>{r[F_BQ].x, r[F_BQ].y}, us);
    }
    const Df<F> u = d_dup<F>(us.hi, us.lo), bu = d_dup<F>(bus.hi, bus.lo);
    const Df<F> gx = d_mul(bu, d_atan(d_mul(u, Zx))), gy = d_mul(bu, d_atanh(d_mul(u, Zy)));
#pragma unroll
    for (int k = 0; k < f_lanes<F>; ++k)
      if (!(poly >> k & 1u) && !(fabsf(f_part(gx.hi, k)) < INFINITY && fabsf(f_part(gy.hi, k)) < INFINITY))
        ok &= ~(1u << k);
    axp = poly ? d_sel(poly, axp, gx) : gx;
    ayp = poly ? d_sel(poly, ayp, gy) : gy;
  }
  ax = d_ss(d_mul(c, axp), d_neg(d_mul(s, ayp)));
  ay = d_ss(d_mul(s, axp), d_mul(c, ayp));
  if (HESS) {
    const Df<F> r2 = d_ss(x2, y2), ymx = d_sub(y2, x2), one = d_dup<F>(1.f, 0.f);
    const Df<F> two_sc = {f_add(sc.hi, sc.hi), f_add(sc.lo, sc.lo)}, two_st = {f_add(st.hi, st.hi), f_add(st.lo, st.lo)};
    const Df<F> Dc = d_ss(d_ss(ld(F_DC0), d_mul(two_sc, psc)), r2), Dt = d_ss(d_ss(ld(F_DT0), d_mul(two_st, pst)), r2);
    const Df<F> fc = d_div(one, d_mul(psc, Dc)), ft = d_div(one, d_mul(pst, Dt));
    const Df<F> g1p = d_mul(ld(F_HB), d_sub(d_mul(fc, d_sub(ymx, ld(F_U2SC2))), d_mul(ft, d_sub(ymx, ld(F_U2ST2)))));
    const Df<F> g2p = d_neg(d_mul(d_mul(bq, d_sub(fc, ft)), d_mul(x, y)));
    h[0] = d_div(RAW ? d_mul(ld(F_HB), ld(F_KTC)) : ld(F_KTC), d_mul(d_mul(Sp, psc), pst));
    const Df<F> c2 = ld(F_C2), s2 = ld(F_S2);
    h[1] = d_sub(d_mul(c2, g1p), d_mul(s2, g2p));
    h[2] = d_add(d_mul(s2, g1p), d_mul(c2, g2p));
  }
  return ok;
}

// SIS or point mass (circ_df), strength b; zero at the centre.
template <bool HESS, class F>
__device__ __noinline__ void circ_fixed(float2 x0, float2 y0, float2 bb, bool point, Df<F> X, Df<F> Y, Df<F> &ax,
                                        Df<F> &ay, Df<F> *h) {
  const Df<F> b = d_dup<F>(bb.x, bb.y), zero = d_dup<F>(0.f, 0.f);
  const Df<F> dX = d_sub(X, d_dup<F>(x0.x, x0.y)), dY = d_sub(Y, d_dup<F>(y0.x, y0.y));
  const Df<F> r2 = d_ss(d_mul(dX, dX), d_mul(dY, dY));
  const unsigned in = f_above(r2.hi, 0.f);
  const F half = f_dup<F>(0.5f);
  const Df<F> ir2 = d_div(d_dup<F>(1.f, 0.f), r2);
  const Df<F> f = point ? d_mul(b, ir2) : d_mul(b, d_sqrt(ir2));  // b/r^2 or b/r
  ax = d_sel(in, d_mul(f, dX), zero);
  ay = d_sel(in, d_mul(f, dY), zero);
  if (HESS) {
    const Df<F> g = point ? d_mul(f, ir2) : d_mul(d_mulf(f, half), ir2);
    h[0] = point ? zero : d_sel(in, d_mulf(f, half), zero);
    h[1] = d_sel(in, d_mul(g, d_sub(d_mul(dY, dY), d_mul(dX, dX))), zero);
    h[2] = d_sel(in, d_neg(d_mulf(d_mul(g, d_mul(dX, dY)), f_dup<F>(2.f))), zero);
  }
}

// Any potential: the components whose result holds (the others take FP64).
template <bool HESS, bool UW, class F, bool RAW = false>
__device__ __forceinline__ unsigned any_fixed(const float2 *__restrict__ r, Df<F> X, Df<F> Y, Df<F> &ax, Df<F> &ay,
                                              Df<F> *h) {
  if (r[F_U2].x < 0.f) {
    circ_fixed<HESS>(r[F_X0], r[F_Y0], r[F_BQ], r[F_U2].x < -1.5f, X, Y, ax, ay, h);
    return f_all<F>;
  }
  return dpie_fixed<HESS, UW, F, RAW>(r, X, Y, ax, ay, h);
}

}  // namespace lens
