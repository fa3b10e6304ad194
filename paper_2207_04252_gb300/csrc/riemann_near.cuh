// Exact Riemann solution on the face (Sect. 2.6) where the star pressure is
// close to both side pressures, |x_K| <= 1/64 (float) or 1/128 (double) with
// x_K = p*/p_K - 1: every face of a smooth flow, and all but a few cells
// around a strong shock.
//
// There the pressure function of a side is f_K = x p_K / (rho_K c_K) S(x),
// its derivative T(x) / (rho_K c_K) with T = (x S)', and the star density
// rho_K (1 + x D(x)); S, D are the Taylor series of the rarefaction branch
// (x <= 0) or of the shock branch, which agree to first order, so that one
// straight line of code with selected coefficients serves both and the lanes
// of a warp do not diverge.  With beta = (gamma - 1)/(2 gamma):
//   rarefaction  S_k = C(beta, k+1)/beta,   D_k = C(1/gamma, k+1),
//   shock        S_k = C(-1/2, k) ((gamma+1)/(2 gamma))^k,  D_k = (-beta)^k / gamma.
// The differences that enter (p_R - p_L, u_R - u_L) are the caller's, so the
// perturbation forms pass theirs exactly.
//
// In double the Newton iteration runs in float and its result is corrected by
// FP64 residuals: step = -F/F' with F in FP64 and the quotient in float.  A
// step has a relative error of about 2^-22, so the iteration ends once it is
// below 2^-31 p (one evaluation of F for |x| up to about 2^-9, two beyond).
// What the caller does with the solution sets how far it is taken:
//   NEAR_STATE       the star state.  1/(rho c) and 1/p to about 2^-42, one Newton
//                    step from the float values (five and two FP64 operations
//                    instead of seven and three): they multiply p* - p_K, so p* is
//                    within 2^-53 p + 2^-42 |p* - p_K| (2^-49 p at |x| = 1/128);
//   NEAR_INVERSES    the same with 1/(rho c) and 1/p to their last bits (the adjoint);
//   NEAR_DEPARTURES  p* - p_K, u* - u_K and rho* - rho_K to their own last bits (the
//                    perturbation forms, whose result they are): the linear
//                    solution is taken in FP64, the float iteration gives only
//                    what S - 1 adds to it (|x| of it and less, and nothing that
//                    float's range could lose), and the residuals go on to 2^-31
//                    of the larger |p* - p_K|: one evaluation for |x| up to about
//                    2^-10.  Twelve FP64 operations a face more than NEAR_STATE, 1.7 %
//                    of a step of 93 x 131 x 37 bi-fluid cells (2.64 -> 2.69 ms); a
//                    second evaluation in place of the linear solution took 4.8 %.
// The series are summed in double to x^3, the rest (below 2^-30 of the sum at
// |x| = 1/128) in float: 1/128 is where float's rounding of the tail reaches
// 2^-54 of the sum; each power of two more takes another FP64 term per sum.
//
// What bounds the callers: in FP64 the two-lane FP64 pipe, which sees about
// 55 operations here against 250 to 300 of the FP64 Newton iteration with its
// two branches; in float the issue slots.  A step of the gas disc, 128 x 256 x 32
// cells in double, went from 10.8 to 3.8 ms with this and the parabola of
// stage_full.cuh; the bi-fluid one in float, 512 x 1024 x 128, from 28.9 to 19.6.
#pragma once
#include <cstring>

#include "narrow.cuh"

namespace rossbi {

constexpr int NEAR_N = 4;  // FP64 terms of a series
constexpr int NEAR_T = 5;  // float terms of its tail
constexpr float NEAR_XF = 0.015625f, NEAR_XD = 0.0078125f;

// Series coefficients of one gamma, [0] rarefaction, [1] shock (built on the host).
struct NearCoef {
  double s[2][NEAR_N], d[2][NEAR_N];
  float st[2][NEAR_T], dt[2][NEAR_T];  // tails: the terms x^4 ... x^8
  double t[2][NEAR_N], h[2][NEAR_N];   // (x S)' and (x D)', for the adjoint
  float tt[2][NEAR_T], ht[2][NEAR_T];
  float sf[2][5], tf[2][5], df[2][4];  // S, T, D in float
  f32x2 g2, t22, t12, s12;             // twice gamma, the mean of the branches' T_2, T_1 and S_1
  double gamma, g_gm1;  // gamma, gamma / (gamma - 1)
  float gammaf;
};

// Builds the coefficients of gamma (host).
inline NearCoef near_coef(double gamma) {
  NearCoef c{};
  const double beta = (gamma - 1.0) / (2.0 * gamma), alpha = (gamma + 1.0) / (2.0 * gamma), ig = 1.0 / gamma;
  double bb = beta, bg = ig, bh = 1.0, al = 1.0, be = ig;  // C(beta, k+1), C(1/gamma, k+1), C(-1/2, k), alpha^k, (-beta)^k / gamma
  for (int k = 0; k < NEAR_N + NEAR_T; ++k) {
    const double s[2] = {bb / beta, bh * al}, d[2] = {bg, be};
    for (int q = 0; q < 2; ++q) {
      if (k < NEAR_N) {
        c.s[q][k] = s[q];
        c.d[q][k] = d[q];
        c.t[q][k] = (k + 1) * s[q];
        c.h[q][k] = (k + 1) * d[q];
      } else {
        c.st[q][k - NEAR_N] = (float)s[q];
        c.dt[q][k - NEAR_N] = (float)d[q];
        c.tt[q][k - NEAR_N] = (float)((k + 1) * s[q]);
        c.ht[q][k - NEAR_N] = (float)((k + 1) * d[q]);
      }
      if (k < 5) {
        c.sf[q][k] = (float)s[q];
        c.tf[q][k] = (float)((k + 1) * s[q]);
        if (k < 4) c.df[q][k] = (float)d[q];
      }
    }
    bb *= (beta - (k + 1)) / (k + 2);
    bg *= (ig - (k + 1)) / (k + 2);
    bh *= (-0.5 - k) / (k + 1);
    al *= alpha;
    be *= -beta;
  }
  c.gamma = gamma;
  c.g_gm1 = gamma / (gamma - 1.0);
  c.gammaf = (float)gamma;
  auto twice = [](float v) {
    f32x2 r;
    const float two[2] = {v, v};
    std::memcpy(&r, two, sizeof(r));
    return r;
  };
  c.g2 = twice(c.gammaf);
  c.t22 = twice(0.5f * (c.tf[0][2] + c.tf[1][2]));
  c.t12 = twice(c.tf[0][1]);
  c.s12 = twice(c.sf[0][1]);
  return c;
}

// Float series to x^4, less its constant and over x; the branches share the
// first two coefficients.
__device__ __forceinline__ float near_slope_f(const float (&c)[2][5], bool shock, float x) {
  float t = shock ? c[1][4] : c[0][4];
#pragma unroll
  for (int k = 3; k >= 2; --k) t = fmaf(t, x, shock ? c[1][k] : c[0][k]);
  return fmaf(t, x, c[0][1]);
}
__device__ __forceinline__ float near_sum_f(const float (&c)[2][5], bool shock, float x) {
  return fmaf(near_slope_f(c, shock, x), x, c[0][0]);
}
// The same to x^3 (truncation below 2^-26 at |x| = 1/64).
template <int N>
__device__ __forceinline__ float near_cubic(const float (&c)[2][N], bool shock, float x) {
  const float t = fmaf(shock ? c[1][3] : c[0][3], x, shock ? c[1][2] : c[0][2]);
  return fmaf(fmaf(t, x, c[0][1]), x, c[0][0]);
}
// In double: NEAR_N terms in double, the tail in float.
__device__ __forceinline__ double near_sum(const double (&c)[2][NEAR_N], const float (&ct)[2][NEAR_T], bool shock,
                                           double x) {
  const float xf = narrow(x);
  float t = shock ? ct[1][NEAR_T - 1] : ct[0][NEAR_T - 1];
#pragma unroll
  for (int k = NEAR_T - 2; k >= 0; --k) t = fmaf(t, xf, shock ? ct[1][k] : ct[0][k]);
  double v = widen(t);
#pragma unroll
  for (int k = NEAR_N - 1; k >= 2; --k) v = fma(v, x, shock ? c[1][k] : c[0][k]);
  return fma(fma(v, x, c[0][1]), x, c[0][0]);
}

enum { NEAR_GENERAL = 0, NEAR_LEFT = 1, NEAR_RIGHT = 2, NEAR_STAR_L = 3, NEAR_STAR_R = 4 };

enum { NEAR_STATE, NEAR_INVERSES, NEAR_DEPARTURES };  // what the solution is for, see above

// What the solution needs beyond the face state (the adjoint reads it).
template <class T>
struct NearStar {
  T d;          // p* - p_L
  T us;         // u* about the base velocity of ul, ur
  T drho;       // rho* - rho_K of the side K that the face lies on
  T fl, fr;     // pressure functions at p*
  T ircl, ircr, ipl, ipr;
};

// Which state is on the face: NEAR_LEFT / NEAR_RIGHT (the side's own, the
// flow being supersonic), NEAR_STAR_L / NEAR_STAR_R (the star state of that
// side; s is set), or NEAR_GENERAL: not near, or within the sonic band where
// a fan or a shock may sit on the face; the caller then takes the general
// solver.  (rl, pl), (rr, pr): densities and pressures (a float state that is
// not positive comes back as NEAR_GENERAL; a double one is the caller's to sort
// out); dP = p_R - p_L, ul, ur velocities about u0, dU = u_R - u_L; vl, vr the
// full velocities; WHAT: one of the three above (the float solution has one way).
template <int WHAT>
__device__ __forceinline__ int near_riemann(const NearCoef& C, double rl, double ul, double pl, double rr, double ur,
                                            double pr, double dP, double dU, double u0, bool has_u0, double vl,
                                            double vr, NearStar<double>& s) {
  using T = double;
  // The float work is in units in which p_L and the sound speed are of order
  // one: pressures by 2^k (bias bp), velocities by 2^m (bias bu), densities by
  // 2^(k - 2m).  In the caller's units the small steps of a small pressure would
  // be below float's range.  p and rho beyond 2^500, whose product may leave
  // the range of double, and densities 2^80 apart go to the general solver.
  const int ep = exponent(pl), er = exponent(rl);
  if ((unsigned)(ep - 523) > 1000u || (unsigned)(er - 523) > 1000u) return NEAR_GENERAL;
  const int m = (ep - er) >> 1, bp = ep - 127, bu = FLOAT_BIAS + m, br = bp - 2 * m;
  const float plf = narrow(pl, bp), prf = narrow(pr, bp), rlf = narrow(rl, br), rrf = narrow(rr, br);
  if (!(rrf > 0x1p-80f && rrf < 0x1p80f)) return NEAR_GENERAL;
  const float ulf = narrow(vl, bu), urf = narrow(vr, bu);
  const float gl = C.gammaf * plf, gr = C.gammaf * prf;
  const float il = recip_sqrt(gl) * recip_sqrt(rlf), ir = recip_sqrt(gr) * recip_sqrt(rrf);  // 1 / (rho c)
  const float cl = gl * il, cr = gr * ir;
  const float ipl = recip_normal(plf), ipr = recip_normal(prf);
  const float dPf = narrow(dP, bp), dUf = narrow(dU, bu);
  // linear (acoustic) star pressure d = p* - p_L
  float d = (dPf * ir - dUf) * recip_normal(il + ir);
  float xl = d * ipl, xr = (d - dPf) * ipr;
  float X = fabsf(xl) + fabsf(xr);
  if (!(X <= 2.0f * NEAR_XF)) return NEAR_GENERAL;  // NaN too
  // supersonic by a margin that covers every wave speed at |x| <= 1/32
  if (ulf >= 1.1f * cl) return NEAR_LEFT;
  if (-urf >= 1.1f * cr) return NEAR_RIGHT;
  if (!(X <= NEAR_XD)) return NEAR_GENERAL;
  if (WHAT == NEAR_STATE) {
    const int bq = 2 * FLOAT_BIAS - bp, bi = bq + m;  // of 1/p, 1/(rho c)
    s.ircl = refine_recip_sqrt(C.gamma * (pl * rl), widen(il, bi));
    s.ircr = refine_recip_sqrt(C.gamma * (pr * rr), widen(ir, bi));
    s.ipl = refine_recip(pl, widen(ipl, bq));
    s.ipr = refine_recip(pr, widen(ipr, bq));
  } else {
    s.ircl = recip_sqrt(C.gamma * (pl * rl));
    s.ircr = recip_sqrt(C.gamma * (pr * rr));
    s.ipl = recip(pl);
    s.ipr = recip(pr);
  }
  {
    float tl = 0.0f, tr = 0.0f;
#pragma unroll
    for (int it = 0; it < 2; ++it) {
      const bool sl = d > 0.0f, sr = d > dPf;
      xl = d * ipl;
      xr = (d - dPf) * ipr;
      tl = il * near_sum_f(C.tf, sl, xl);
      tr = ir * near_sum_f(C.tf, sr, xr);
      d -= (d * il * near_sum_f(C.sf, sl, xl) + (d - dPf) * ir * near_sum_f(C.sf, sr, xr) + dUf) * recip_normal(tl + tr);
    }
    const float iD = recip_normal(tl + tr);
    const float small = 4.6e-10f * (WHAT == NEAR_DEPARTURES ? fmaxf(fabsf(d), fabsf(d - dPf)) : fminf(plf, prf));
    T dd, f1 = T(0), f2 = T(0);
    if (WHAT == NEAR_DEPARTURES) {
      xl = d * ipl;
      xr = (d - dPf) * ipr;
      const float ql = d * il * (xl * near_slope_f(C.sf, d > 0.0f, xl));
      const float qr = (d - dPf) * ir * (xr * near_slope_f(C.sf, d > dPf, xr));
      dd = fma(fma(dP, s.ircr, -dU), recip(s.ircl + s.ircr), widen(-(ql + qr) * recip_normal(il + ir), bp));
    } else {
      dd = widen(d, bp);
    }
    float step = 0.0f;
    bool more = true;
    for (int it = 0; it < 4 && more; ++it) {
      const T dr = dd - dP;
      const T yl = dd * s.ipl, yr = dr * s.ipr;
      const bool sl = !sign_bit(yl), sr = !sign_bit(yr);
      f1 = dd * s.ircl * near_sum(C.s, C.st, sl, yl);
      f2 = dr * s.ircr * near_sum(C.s, C.st, sr, yr);
      step = -narrow(f1 + f2 + dU, bu) * iD;
      dd += widen(step, bp);
      more = !(fabsf(step) <= small);
    }
    if (more) return NEAR_GENERAL;
    s.d = dd;
    s.fl = f1 + widen(tl * step, bu);
    s.fr = f2 + widen(tr * step, bu);
  }
  s.us = ul - s.fl;
  // u* = u_L - f_L = u_R + f_R: the side that the face lies on gives it
  const bool left = !sign_bit(has_u0 ? u0 + s.us : s.us);
  if (!left) s.us = ur + s.fr;
  // the head of side K is at u_K -/+ c_K, its shock or tail within |x| c_K of
  // it: the side's own state beyond that band, the star state before it
  const float v = left ? ulf : -urf, c = left ? cl : cr, band = c * fmaf(1.25f, X, 1e-5f);
  if (v - c >= band) return left ? NEAR_LEFT : NEAR_RIGHT;
  if (!(c - v > band)) return NEAR_GENERAL;
  const T x = left ? s.d * s.ipl : (s.d - dP) * s.ipr;
  s.drho = (left ? rl : rr) * (x * near_sum(C.d, C.dt, !sign_bit(x), x));
  return left ? NEAR_STAR_L : NEAR_STAR_R;
}

// The same in float, the two sides in the halves of packed values (they take
// the same operations).
template <int WHAT>
__device__ __forceinline__ int near_riemann(const NearCoef& C, float rl, float ul, float pl, float rr, float ur,
                                            float pr, float dP, float dU, float u0, bool has_u0, float ulf, float urf,
                                            NearStar<float>& s) {
  const f32x2 one = pack2(1.0f, 1.0f), g2 = mul2(C.g2, pack2(pl, pr));
  float gl, gr, il, ir, cl, cr, xl, xr, fl, fr, tl, tr;
  unpack2(g2, gl, gr);
  const f32x2 i2 = mul2(pack2(recip_sqrt(gl), recip_sqrt(gr)), pack2(recip_sqrt(rl), recip_sqrt(rr)));  // 1 / (rho c)
  unpack2(i2, il, ir);
  unpack2(mul2(g2, i2), cl, cr);
  s.ipl = recip_normal(pl);
  s.ipr = recip_normal(pr);
  const f32x2 ip2 = pack2(s.ipl, s.ipr);
  // linear (acoustic) star pressure d = p* - p_L
  const float sum = il + ir;
  float d = (dP * ir - dU) * recip_normal(sum);
  unpack2(mul2(pack2(d, d - dP), ip2), xl, xr);
  const float X = fabsf(xl) + fabsf(xr);
  // NaN too: a state that is not positive; a sum beyond 2^126: densities or
  // pressures so small (subnormal, too) that their inverses leave float's range
  if (!(X <= 2.0f * NEAR_XF) || !(sum < 0x1p126f)) return NEAR_GENERAL;
  if (ulf >= 1.1f * cl) return NEAR_LEFT;
  if (-urf >= 1.1f * cr) return NEAR_RIGHT;
  if (!(X <= NEAR_XF)) return NEAR_GENERAL;
  // One Newton step from the acoustic value, whose error is below 0.45 x^2 p:
  // what it leaves, below 0.1 x^4 p, is under the rounding of d for |x| <=
  // 1/128, and a second step's beyond.  The slope needs three digits only
  // (T to x^2 with the branches' mean T_2).
  auto newton = [&]() {
    const float dr = d - dP;
    const f32x2 d2 = pack2(d, dr), x2 = mul2(d2, ip2);
    const f32x2 t2 = mul2(i2, fma2(fma2(C.t22, x2, C.t12), x2, one));
    const bool sl = d > 0.0f, sr = dr > 0.0f;  // shock branches
    f32x2 S = fma2(pack2(sl ? C.sf[1][3] : C.sf[0][3], sr ? C.sf[1][3] : C.sf[0][3]), x2,
                   pack2(sl ? C.sf[1][2] : C.sf[0][2], sr ? C.sf[1][2] : C.sf[0][2]));
    S = fma2(fma2(S, x2, C.s12), x2, one);
    f32x2 f2 = mul2(mul2(d2, i2), S);
    unpack2(f2, fl, fr);
    unpack2(t2, tl, tr);
    const float step = -(fl + fr + dU) * recip_normal(tl + tr);
    d += step;
    unpack2(fma2(t2, pack2(step, step), f2), fl, fr);
  };
  newton();
  if (X > 0.0078125f) newton();
  s.d = d;
  s.fl = fl;
  s.fr = fr;
  s.us = ul - fl;
  const bool left = !sign_bit(has_u0 ? u0 + s.us : s.us);
  if (!left) s.us = ur + fr;
  const float v = left ? ulf : -urf, c = left ? cl : cr, band = c * fmaf(1.25f, X, 1e-5f);
  if (v - c >= band) return left ? NEAR_LEFT : NEAR_RIGHT;
  if (!(c - v > band)) return NEAR_GENERAL;
  const float x = left ? d * s.ipl : (d - dP) * s.ipr;
  s.drho = (left ? rl : rr) * (x * near_cubic(C.df, x > 0.0f, x));
  return left ? NEAR_STAR_L : NEAR_STAR_R;
}

}  // namespace rossbi
