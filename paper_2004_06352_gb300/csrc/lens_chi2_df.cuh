// The double-float evaluator of the source-plane chi2's varying potentials:
// the forms of lens_device.cuh's dpie_df with three-term divisions and every
// operation renormalised.  A set with an image next to a critical curve
// divides by det ~ 1e-5 and smaller, which turns the evaluator's last bits
// (~2e-14) into 1e-9 of its chi2, so this kernel keeps the roundings its
// results have always had; dpie_df, 1.7 times fewer operations at the same
// accuracy, moves mu-weighted chi2 by up to 1e-9 (4096 sets x 372 images).
#pragma once

#include "lens_device.cuh"

namespace lens {
// a / b: MUFU reciprocal of b.hi, then two remainders a - b q correct the
// quotient (its first term may be off by a few 2^-24).  Called, not inlined:
// at each of its ~10 call sites it would make the kernel outgrow the
// instruction cache (4096 sets: 0.373 -> 0.359 ms).
static __device__ __noinline__ df df_div3(df a, df b) {
  const float ib = rcp_a(b.hi);
  const float q1 = a.hi * ib;
  df r = df_sub(a, df_mulf(b, q1));
  const float q2 = r.hi * ib;
  r = df_sub(r, df_mulf(b, q2));
  const float q3 = r.hi * ib;
  return df_add_ss(fast_two_sum(q1, q2), df{q3, 0.f});
}

__device__ __forceinline__ df df_poly3(df t, const float (*c)[2]) {
  float tail = c[11][0];
#pragma unroll
  for (int k = 10; k >= 7; --k) tail = fmaf(tail, t.hi, c[k][0]);
  df p = df_add_ss(df{c[6][0], c[6][1]}, df_mulf(t, tail));
#pragma unroll
  for (int k = 5; k >= 0; --k) p = df_add_ss(df{c[k][0], c[k][1]}, df_mul(p, t));  // |p t| < 0.16 |p|: no cancellation
  return p;
}

// atan(w) and atanh(w) for any argument (|w| < 1 for atanh), by the reductions
// of atan64 / atanh64; atanh returns NaN within ~1e-15 of 1.
__device__ __forceinline__ df df_atan3(df w) {
  const bool neg = w.hi < 0.f;
  const df a = neg ? df_neg(w) : w;
  const bool inv = a.hi > 1.f;
  df v = inv ? df_div3(df{1.f, 0.f}, a) : a;
  df base = {0.f, 0.f};
  if (v.hi > 0.4f) {
    v = df_div3(df_sub(v, df{0.6875f, 0.f}), df_add_ss(df{1.f, 0.f}, df_mulf(v, 0.6875f)));
    base = df{ATAN_11_16_DF[0], ATAN_11_16_DF[1]};
  }
  df r = df_add(base, df_mul(v, df_poly3(df_mul(v, v), C_ATAN_DF)));
  if (inv) r = df_sub(df{PI_2_DF[0], PI_2_DF[1]}, r);
  return neg ? df_neg(r) : r;
}
__device__ __forceinline__ df df_atanh3(df w) {
  const bool neg = w.hi < 0.f;
  const df a = neg ? df_neg(w) : w;
  df r;
  if (a.hi <= 0.4f) {
    r = df_mul(a, df_poly3(df_mul(a, a), C_ATANH_DF));
  } else {
    const df om = df_sub(df{1.f, 0.f}, a);  // 1 - a, exact enough to pick the centre
    const float est = 0.5f * (__logf(1.f + a.hi) - __logf(om.hi));
    const int k = __float2int_rn(est * 1.25f);
    if (!(om.hi > 0.f) || k > 22) return df{__int_as_float(0x7fc00000), 0.f};
    const int kk = k < 1 ? 1 : k;
    const df c = {ATANH_C_DF[kk][0], ATANH_C_DF[kk][1]};
    const df v = df_div3(df_sub(a, c), df_sub(df{1.f, 0.f}, df_mul(a, c)));
    r = df_add(df{ATANH_A_DF[kk][0], ATANH_A_DF[kk][1]}, df_mul(v, df_poly3(df_mul(v, v), C_ATANH_DF)));
  }
  return neg ? df_neg(r) : r;
}

// One dPIE potential (record r): deflection and, if HESS, kappa, gamma1,
// gamma2 into h[0..2]; false for a non-finite result.  UW: u and b q / u from
// the record (record_uw), else formed where they are needed.
template <bool HESS, bool UW>
__device__ __forceinline__ bool dpie_df3(const float2 *__restrict__ r, df X, df Y, df &ax, df &ay,
                                        df *h) {
  auto ld = [&](int k) {
    const float2 v = r[k];
    return df{v.x, v.y};
  };
  const df c = ld(F_C), s = ld(F_S);
  const df dX = df_sub(X, ld(F_X0)), dY = df_sub(Y, ld(F_Y0));
  // rotations: the one-TwoSum add's error is bounded by 2^-47 |(dX, dY)|
  const df x = df_add_ss(df_mul(c, dX), df_mul(s, dY)), y = df_add_ss(df_mul(c, dY), df_neg(df_mul(s, dX)));
  const df q2 = ld(F_Q2), u2 = ld(F_U2);
  const df x2 = df_mul(x, x), y2 = df_mul(y, y);
  // every sum below adds non-negative terms except dS and the y denominator
  const df R = df_add_ss(df_mul(q2, x2), y2);
  const df psc = df_sqrt(df_add_ss(R, ld(F_KC)));
  const df pst = df_sqrt(df_add_ss(R, ld(F_KT)));
  const df Sp = df_add_ss(psc, pst);
  const df sc = ld(F_SC), st = ld(F_ST);
  const df Ec = df_add_ss(psc, sc), Et = df_add_ss(pst, st);
  const df dS = df_add_ss(st, df_neg(sc));  // st > sc > 0: error 2^-47 (st + sc) < 2^-46 dS
  const df numx = df_mul(df_mul(x, dS), df_add_ss(Sp, ld(F_Q2SS)));
  const df denx = df_mul(Sp, df_add_ss(df_mul(Ec, Et), df_mul(u2, x2)));
  const df Zx = df_div3(numx, denx);
  const df Fc = df_add_ss(psc, ld(F_Q2SC)), Ft = df_add_ss(pst, ld(F_Q2ST));
  const df numy = df_mul(df_mul(y, ld(F_Q2DS)), df_add_ss(Sp, ld(F_SS)));
  const df deny = df_mul(Sp, df_sub(df_mul(Fc, Ft), df_mul(u2, y2)));
  const df Zy = df_div3(numy, deny);
  const df tx = df_mul(u2, df_mul(Zx, Zx)), ty = df_mul(u2, df_mul(Zy, Zy));
  const df bq = ld(F_BQ);
  df axp, ayp;
  if (tx.hi < (float)T_SERIES64 && ty.hi < (float)T_SERIES64) {  // bq Z atan(w)/w, w = u Z
    axp = df_mul(df_mul(bq, Zx), df_poly3(tx, C_ATAN_DF));
    ayp = df_mul(df_mul(bq, Zy), df_poly3(ty, C_ATANH_DF));
  } else {
    const df u = UW ? ld(F_U) : df_sqrt(u2), bu = UW ? ld(F_BU) : df_div3(bq, u);  // (bq / u) atan(u Z)
    axp = df_mul(bu, df_atan3(df_mul(u, Zx)));
    ayp = df_mul(bu, df_atanh3(df_mul(u, Zy)));
    if (!(fabsf(axp.hi) < INFINITY && fabsf(ayp.hi) < INFINITY)) return false;
  }
  ax = df_add_ss(df_mul(c, axp), df_neg(df_mul(s, ayp)));  // rotation back: error 2^-47 |(axp, ayp)|
  ay = df_add_ss(df_mul(s, axp), df_mul(c, ayp));
  if (HESS) {
    const df r2 = df_add_ss(x2, y2), ymx = df_sub(y2, x2);
    const df Dc = df_add_ss(df_add_ss(ld(F_DC0), df_mul(df_mulf(sc, 2.f), psc)), r2);
    const df Dt = df_add_ss(df_add_ss(ld(F_DT0), df_mul(df_mulf(st, 2.f), pst)), r2);
    const df fc = df_div3(df{1.f, 0.f}, df_mul(psc, Dc)), ft = df_div3(df{1.f, 0.f}, df_mul(pst, Dt));
    const df hb = ld(F_HB);
    const df g1p = df_mul(hb, df_sub(df_mul(fc, df_sub(ymx, ld(F_U2SC2))), df_mul(ft, df_sub(ymx, ld(F_U2ST2)))));
    const df g2p = df_neg(df_mul(df_mul(bq, df_sub(fc, ft)), df_mul(x, y)));
    h[0] = df_div3(df_mul(hb, ld(F_KTC)), df_mul(df_mul(Sp, psc), pst));
    const df c2 = ld(F_C2), s2 = ld(F_S2);
    h[1] = df_sub(df_mul(c2, g1p), df_mul(s2, g2p));
    h[2] = df_add(df_mul(s2, g1p), df_mul(c2, g2p));
  }
  return true;
}

// SIS or point mass, as circ_df.
template <bool HESS>
__device__ __forceinline__ void circ_df3(const float2 *__restrict__ r, df X, df Y, df &ax, df &ay,
                                        df *h) {
  const float2 x0 = r[F_X0], y0 = r[F_Y0], b2 = r[F_BQ];
  const df b = {b2.x, b2.y};
  const df dX = df_sub(X, df{x0.x, x0.y}), dY = df_sub(Y, df{y0.x, y0.y});
  const df r2 = df_add_ss(df_mul(dX, dX), df_mul(dY, dY));
  if (!(r2.hi > 0.f)) {
    ax = ay = df{0.f, 0.f};
    if (HESS) h[0] = h[1] = h[2] = df{0.f, 0.f};
    return;
  }
  const bool point = r[F_U2].x < -1.5f;
  const df ir2 = df_div3(df{1.f, 0.f}, r2);
  const df f = point ? df_mul(b, ir2) : df_mul(b, df_sqrt(ir2));  // b/r^2 or b/r
  ax = df_mul(f, dX);
  ay = df_mul(f, dY);
  if (HESS) {
    // SIS: kappa = b/(2r), gamma = b/(2r^3) (y^2-x^2, -2xy); point: kappa = 0,
    // gamma = b/r^4 (y^2-x^2, -2xy)
    const df g = point ? df_mul(f, ir2) : df_mul(df_mulf(f, 0.5f), ir2);
    h[0] = point ? df{0.f, 0.f} : df_mulf(f, 0.5f);
    h[1] = df_mul(g, df_sub(df_mul(dY, dY), df_mul(dX, dX)));
    h[2] = df_neg(df_mulf(df_mul(g, df_mul(dX, dY)), 2.f));
  }
}

// u and b q / u of a dPIE record as this evaluator forms them, once per record
__device__ __forceinline__ void record_uw(float2 *r) {
  if (!(r[F_U2].x > 0.f)) return;  // circular (never used), SIS, point mass
  const df u = df_sqrt(df{r[F_U2].x, r[F_U2].y}), bu = df_div3(df{r[F_BQ].x, r[F_BQ].y}, u);
  r[F_U] = make_float2(u.hi, u.lo);
  r[F_BU] = make_float2(bu.hi, bu.lo);
}

}  // namespace lens
