// Discrete adjoint of the FP64 RK2 step (reverse stage kernels).
//
// The step map E^n -> E^{n+1} at a fixed dt is differentiated as written:
// limiter branches, the wave pattern and sampling of the exact Riemann
// solution, the dust upwinding and the positivity fallback are held at the
// branch the forward values take; the star pressure's derivative follows from
// the implicit function theorem at the converged p*.  Where rounding alone decides
// a branch, both sides' derivatives belong to the same forward value.  Conservative
// departures take the forward's own expressions there too.  With primitive ones
// such states are usual (the pressure departure of an isobaric one, the velocities
// of a wall's face beside an equilibrium ghost); their branches come from
// expressions of the adjoint's own, slope_branches and for contacts at rest
// riemann_vjp_general, which do not move when the forward is arranged for speed, so that
// the side taken there may be the other one than in the forward's rounding.  For
// one stage
//     Y = E_base + tau (G(E_in) - R0) / V,    E_out = D(Y)   (drag),
// a cotangent lambda_out on E_out gives mu = D'(Y)^T lambda_out on Y and on
// E_base, the weighted cotangent mu' = tau / V mu on G, and
// G'(E_in)^T mu' = sum over faces (flux part) + V S'(E_in)^T mu' (sources).
//
// Kernels:
//   adj_point_kernel  drag and source adjoints per cell, writes mu', the
//                     cotangent of E^n and the d/dSt block partials;
//   adj_flux_kernel   flux part of G'^T mu' along one axis, accumulated into
//                     the cotangent of the stage input.
// A line of L lanes along the axis owns T = L - 4 cells: lane p holds cell
// c = c0 - 2 + p, reconstructs it (gas: the conservative departures, or the
// primitive ones with RC = RECON_PRIM), solves the face below it (once per tile),
// back-propagates the face cotangent to both face states, passes the lower
// one down by a shuffle, back-propagates its own reconstruction and passes
// the neighbour contributions up and down by shuffles; every sum has a fixed
// order, so the result is deterministic.
//
// The FP64 pipe bounds the flux kernel.  With six tangents through the Riemann
// solution it took 255 registers, eight warps per SM and, for a gradient through
// two bi-fluid steps of 128 x 256 x 32 cells, most of 159 ms; with the closed
// reverse of the near solution, the gas before the dust (168 registers, twelve
// warps per SM) and lines by the axis (launch.cuh) the gradient takes 41 ms, a
// third of it in the flux kernels (1.40, 0.95 and 1.38 ms a stage along r, theta
// and z), the rest in forward stages and the point kernels.
#pragma once
#include "stage_full.cuh"

namespace rossbi {

// ------------------------------------------------------------------ face flux adjoints
struct FluxCot {  // cotangent of the flux in face order: mass, normal and transverse momenta, energy
  double m, n, t1, t2, e;
};
// Cotangents of the face state's own values, F = (m, m u + p, m ut1, m ut2,
// H u) with m = rho u, H = rho K + g / (g - 1) p, K = |v|^2 / 2.
__device__ __forceinline__ void flux_state_vjp(double g_gm1, double rho, double u, double p, double ut1, double ut2,
                                               const FluxCot& F, double& rb, double& ub, double& pb, double& ut1b,
                                               double& ut2b) {
  const double m = rho * u, K = 0.5 * fma(u, u, fma(ut1, ut1, ut2 * ut2));
  const double mb = fma(F.e, K, fma(F.n, u, fma(F.t1, ut1, fma(F.t2, ut2, F.m))));  // d/dm, with H u = m K + g/(g-1) p u
  const double Fm = F.e * m, Fp = F.e * g_gm1;
  rb = mb * u;
  ub = fma(F.n, m, fma(Fp, p, fma(Fm, u, mb * rho)));
  pb = fma(Fp, u, F.n);
  ut1b = fma(F.t1, m, Fm * ut1);
  ut2b = fma(F.t2, m, Fm * ut2);
}

// f_K and df_K/dp at the star pressure; for gamma = 7/5 zK = (p / p_K)^(1/7) is given.
template <bool G75>
__device__ __forceinline__ void pressure_fn_at(double g, const RSide& K, double p, double zK, double& f, double& fd) {
  if (p <= K.p) {
    const double prat = p / K.p;
    const double e = G75 ? zK : pow(prat, (g - 1.0) / (2.0 * g));
    f = 2.0 * K.c / (g - 1.0) * (e - 1.0);
    fd = e / (prat * K.rho * K.c);
  } else {
    const double A = 2.0 / ((g + 1.0) * K.rho);
    const double B = (g - 1.0) / (g + 1.0) * K.p;
    const double q = sqrt(A / (B + p));
    f = (p - K.p) * q;
    fd = (1.0 - 0.5 * (p - K.p) / (B + p)) * q;
  }
}

// The general Riemann solution of a face (riemann_face) with its reverse: the
// face's mass flux, the side whose transverse velocity it carries, and the
// cotangents b of (rho, u, p)_L and (rho, u, p)_R for the cotangent F of the flux;
// l1, l2, r1, r2 the transverse velocities.  The wave pattern picks one of four
// closed forms in the side K that the face lies on (its own state, a fan, the star
// state behind a rarefaction or a shock); f_K enters by df_K/drho_K = -f_K / (2
// rho_K) and p* f_K' + p_K df_K/dp_K = f_K / 2, as in gas_flux_vjp.  An adjoint step
// of 140 x 96 x 36 cells with jumps of 3 % at all faces takes 19.6 ms; six tangents
// carried through the solution took 26.9 (21.2 in a kernel of 255 registers without
// the near solution).
struct RFaceVjp {
  double m, b[6];
  int side;
  unsigned status;
};
template <bool G75>
__device__ __forceinline__ RFaceVjp riemann_vjp(double g, double g_gm1, const RSide& L, const RSide& R, double l1,
                                                double l2, double r1, double r2, const FluxCot& F) {
  enum { OWN, FAN, RAREFACTION, SHOCK };
  RFaceVjp o{};
  int what = OWN;
  double ps = 0.0, us = 0.0, fl = 0.0, fdl = 0.0, fr = 0.0, fdr = 0.0, zl = 0.0, zr = 0.0;
  const double pfloor = 1e-8 * fmin(L.p, R.p), t = 2.0 * (g_gm1 - 1.0);  // 2 / (gamma - 1)
  if (t * (L.c + R.c) <= R.u - L.u) {  // vacuum
    if (0.0 <= L.u + t * L.c) {
      o.side = -1;
      what = 0.0 <= L.u - L.c ? OWN : FAN;
    } else if (0.0 >= R.u - t * R.c) {
      o.side = 1;
      what = 0.0 >= R.u + R.c ? OWN : FAN;
    } else {
      return o;
    }
  } else {
    ps = fmax(pfloor, 0.5 * (L.p + R.p) - 0.125 * (R.u - L.u) * (L.rho + R.rho) * (L.c + R.c));
    bool conv = false;
    if (G75) {
      const double k = root7(L.p / R.p);
      double z = root7(ps / L.p), step;
      conv = newton_z_g75(L, R, R.u - L.u, pfloor, k, ps, z, fl, fdl, fr, fdr, step);  // the forward's iteration
      zl = z;
      zr = z * k;
    } else {
      for (int it = 0; it < 100; ++it) {
        pressure_fn(g, L, ps, fl, fdl);
        pressure_fn(g, R, ps, fr, fdr);
        const double pn = fmax(pfloor, ps - (fl + fr + R.u - L.u) / (fdl + fdr));
        const double change = 2.0 * fabs(pn - ps) / (pn + ps);
        ps = pn;
        if (change <= 1e-12) {
          conv = true;
          break;
        }
      }
    }
    if (!conv) o.status = STATUS_RIEMANN;
    pressure_fn_at<G75>(g, L, ps, zl, fl, fdl);
    pressure_fn_at<G75>(g, R, ps, zr, fr, fdr);
    us = 0.5 * (L.u + R.u) + 0.5 * (fr - fl);
    o.side = 0.0 <= us ? -1 : 1;
    // the same on either side with the axis turned round: v towards the face
    const RSide& K = o.side < 0 ? L : R;
    const double sgn = o.side < 0 ? 1.0 : -1.0, v = sgn * K.u, ratio = ps / K.p;
    if (ps > K.p) {
      what = 0.0 <= v - K.c * sqrt((g + 1.0) / (2.0 * g) * ratio + (g - 1.0) / (2.0 * g)) ? OWN : SHOCK;
    } else if (0.0 <= v - K.c) {
      what = OWN;
    } else {
      const double tail = sgn * us - K.c * (G75 ? (o.side < 0 ? zl : zr) : pow(ratio, (g - 1.0) / (2.0 * g)));
      what = (o.side < 0 ? 0.0 > tail : 0.0 >= tail) ? RAREFACTION : FAN;
    }
  }
  const bool left = o.side < 0;
  const RSide K = left ? L : R;
  const double sgn = left ? 1.0 : -1.0, ipk = recip(K.p);
  double rho = K.rho, u = K.u, p = K.p, h = 1.0, dh = 0.0, cf = 0.0;  // h(x) = rho* / rho_K, x = p* / p_K
  if (what == FAN) {
    cf = 2.0 / (g + 1.0) * (K.c + sgn * 0.5 * (g - 1.0) * K.u);
    const double r = cf / K.c;
    u = sgn * cf;
    rho *= G75 ? r * r * (r * r) * r : pow(r, 2.0 / (g - 1.0));
    p *= G75 ? r * r * (r * r) * (r * r * r) : pow(r, 2.0 * g / (g - 1.0));
  } else if (what != OWN) {
    const double x = ps * ipk, g6 = (g - 1.0) / (g + 1.0);
    u = us;
    p = ps;
    if (what == RAREFACTION) {
      const double z = left ? zl : zr;
      h = G75 ? z * z * (z * z) * z : pow(x, 1.0 / g);
      dh = h * recip(g * x);
    } else {
      const double i = recip(x * g6 + 1.0);
      h = (x + g6) * i;
      dh = (1.0 - g6 * g6) * i * i;
    }
    rho *= h;
  }
  double rb, ub, pb, t1b, t2b;
  flux_state_vjp(g_gm1, rho, u, p, left ? l1 : r1, left ? l2 : r2, F, rb, ub, pb, t1b, t2b);
  o.m = rho * u;
  double kr = rb, ku = ub, kp = pb;  // cotangents of K
  double* b = o.b;
  if (what == FAN) {
    const double q = 2.0 / (g - 1.0) * (rb * rho + g * (pb * p));  // cotangent of log(cf / c)
    const double cfb = sgn * ub + q / cf, cb = 2.0 / (g + 1.0) * cfb - q / K.c;
    ku = cfb * (sgn * (g - 1.0) / (g + 1.0));
    kr = (rb * rho - 0.5 * cb * K.c) / K.rho;
    kp = (pb * p + 0.5 * cb * K.c) * ipk;
  } else if (what != OWN) {
    const double hb = rb * K.rho * dh * ipk, gu = 0.5 * ub;
    const double psb = pb + hb + gu * (fdr - fdl);
    kr = rb * h;
    ku = 0.0;
    kp = -hb * (ps * ipk);
    const bool floor = ps == pfloor;
    const double lam = floor ? 0.0 : -psb * recip(fdl + fdr), pm = floor ? 1e-8 * psb : 0.0;
    const double flb = lam - gu, frb = lam + gu;
    b[0] = -0.5 * flb * fl * recip(L.rho);
    b[1] = gu - lam;
    b[2] = flb * (0.5 * fl - ps * fdl) * recip(L.p) + (L.p <= R.p ? pm : 0.0);
    b[3] = -0.5 * frb * fr * recip(R.rho);
    b[4] = gu + lam;
    b[5] = frb * (0.5 * fr - ps * fdr) * recip(R.p) + (L.p <= R.p ? 0.0 : pm);
  }
  b[0] += left ? kr : 0.0;
  b[1] += left ? ku : 0.0;
  b[2] += left ? kp : 0.0;
  b[3] += left ? 0.0 : kr;
  b[4] += left ? 0.0 : ku;
  b[5] += left ? 0.0 : kp;
  return o;
}
static __device__ __noinline__ RFaceVjp riemann_vjp_general(double g, double g_gm1, double rl, double ul, double pl,
                                                            double l1, double l2, double rr, double ur, double pr,
                                                            double r1, double r2, const FluxCot F) {
  const RSide L{rl, ul, pl, sqrt(g * pl / rl)}, R{rr, ur, pr, sqrt(g * pr / rr)};
  return g == 1.4 ? riemann_vjp<true>(g, g_gm1, L, R, l1, l2, r1, r2, F)
                  : riemann_vjp<false>(g, g_gm1, L, R, l1, l2, r1, r2, F);
}

// Cotangents of the primitive face states (u, v, w, P, rho in the field
// slots) for a cotangent Fb on the gas flux F(WL, WR) of gas_face_flux.
//
// Near p_K the reverse of the star state is closed: with f_K = x p_K irc_K
// S(x), df_K/drho_K = -f_K / (2 rho_K) at fixed p* and p_K (f ~ rho^-1/2) and
// p* f_K' + p_K df_K/dp_K = f_K / 2 (f has the dimension of (p/rho)^1/2), and
// the cotangent of p* passes to the side states through f_L + f_R + u_R - u_L
// = 0.  About 40 FP64 operations after the forward's 55, where six tangents
// carried through the solution took over a thousand.
template <int D, int RC>
__device__ __forceinline__ void gas_flux_vjp(const NearCoef& C, const double* WL, const double* WR, const double* Fb,
                                             double* WLb, double* WRb, unsigned& status) {
  constexpr int n = Axes<D>::n, t1 = Axes<D>::t1, t2 = Axes<D>::t2;
#pragma unroll
  for (int f = 0; f < 5; ++f) WLb[f] = WRb[f] = 0.0;
  const double rl = WL[RHO], rr = WR[RHO], pl = WL[EN], pr = WR[EN];
  if (!positive(rl) || !positive(rr) || !positive(pl) || !positive(pr)) return;  // zero flux
  const FluxCot F{Fb[RHO], Fb[n], Fb[t1], Fb[t2], Fb[EN]};
  const double dP = pr - pl;
  NearStar<double> s;
  int kind = near_riemann<NEAR_INVERSES>(C, rl, WL[n], pl, rr, WR[n], pr, dP, WR[n] - WL[n], 0.0, false, WL[n],
                                        WR[n], s);
  // A contact at rest (the wall face beside an equilibrium ghost, both of whose
  // states the limiter makes the equilibrium's) has its two sides' derivatives
  // to choose from by nothing but the rounding of u*.  With primitive departures
  // such faces are usual; the general solver, whose rounding does not depend on
  // how this one is arranged, decides them.
  if (RC == RECON_PRIM && kind >= NEAR_STAR_L &&
      fabsf(narrow(s.us)) <= 1e-14f * narrow(C.gamma * (pl * s.ircl)))
    kind = NEAR_GENERAL;
  if (kind == NEAR_GENERAL) {
    const RFaceVjp o =
        riemann_vjp_general(C.gamma, C.g_gm1, rl, WL[n], pl, WL[t1], WL[t2], rr, WR[n], pr, WR[t1], WR[t2], F);
    status |= o.status;
    WLb[RHO] = o.b[0];
    WLb[n] = o.b[1];
    WLb[EN] = o.b[2];
    WRb[RHO] = o.b[3];
    WRb[n] = o.b[4];
    WRb[EN] = o.b[5];
    const double m = o.m, Fm = F.e * m;
    if (o.side < 0) {
      WLb[t1] = F.t1 * m + Fm * WL[t1];
      WLb[t2] = F.t2 * m + Fm * WL[t2];
    } else if (o.side > 0) {
      WRb[t1] = F.t1 * m + Fm * WR[t1];
      WRb[t2] = F.t2 * m + Fm * WR[t2];
    }
    return;
  }
  const bool left = kind == NEAR_LEFT || kind == NEAR_STAR_L, star = kind >= NEAR_STAR_L;
  const double rk = left ? rl : rr;
  const double rho = star ? rk + s.drho : rk, u = star ? s.us : (left ? WL[n] : WR[n]);
  const double p = star ? pl + s.d : (left ? pl : pr);
  double rb, ub, pb, t1b, t2b;
  flux_state_vjp(C.g_gm1, rho, u, p, left ? WL[t1] : WR[t1], left ? WL[t2] : WR[t2], F, rb, ub, pb, t1b, t2b);
  double lr = 0.0, lu = 0.0, lp = 0.0, qr = 0.0, qu = 0.0, qp = 0.0;  // cotangents of (rho, u, p)_L and _R
  if (star) {
    const double yl = s.d * s.ipl, yr = (s.d - dP) * s.ipr;
    const bool sl = !sign_bit(yl), sr = !sign_bit(yr);
    const double tl = s.ircl * near_sum(C.t, C.tt, sl, yl), tr = s.ircr * near_sum(C.t, C.tt, sr, yr);
    // rho* = rho_K (1 + x D(x)), x = p*/p_K - 1
    const double x = left ? yl : yr, ipk = left ? s.ipl : s.ipr;
    const double hb = rb * rk * (near_sum(C.h, C.ht, left ? sl : sr, x) * ipk);
    const double rkb = rb * (rho * recip(rk)), pkb = -hb * (1.0 + x);
    const double gu = 0.5 * ub;
    const double psb = pb + hb + gu * (tr - tl);
    const double lam = -psb * recip(tl + tr);
    const double fl = lam - gu, fr = lam + gu;  // cotangents of f_L, f_R
    lu = gu - lam;
    qu = gu + lam;
    // 1 / (2 rho_K) = gamma p_K irc_K^2 / 2
    const double hg = -0.5 * C.gamma;
    lr = fl * s.fl * (hg * pl * (s.ircl * s.ircl)) + (left ? rkb : 0.0);
    qr = fr * s.fr * (hg * pr * (s.ircr * s.ircr)) + (left ? 0.0 : rkb);
    lp = fl * fma(-p, tl, 0.5 * s.fl) * s.ipl + (left ? pkb : 0.0);
    qp = fr * fma(-p, tr, 0.5 * s.fr) * s.ipr + (left ? 0.0 : pkb);
  } else {
    lr = left ? rb : 0.0;
    lu = left ? ub : 0.0;
    lp = left ? pb : 0.0;
    qr = left ? 0.0 : rb;
    qu = left ? 0.0 : ub;
    qp = left ? 0.0 : pb;
  }
  WLb[RHO] = lr;
  WLb[n] = lu;
  WLb[EN] = lp;
  WRb[RHO] = qr;
  WRb[n] = qu;
  WRb[EN] = qp;
  WLb[t1] = left ? t1b : 0.0;
  WLb[t2] = left ? t2b : 0.0;
  WRb[t1] = left ? 0.0 : t1b;
  WRb[t2] = left ? 0.0 : t2b;
}

// Cotangents of the dust face primitives (u, v, w, rho_d) for a cotangent Fb
// (dust order: momenta 0..2, mass 3) on dust_kinetic_flux<D>(WL, WR).
template <int D>
__device__ __forceinline__ void dust_flux_vjp(const double* WL, const double* WR, const double* Fb, double* WLb,
                                              double* WRb) {
  constexpr int n = Axes<D>::n, t1 = Axes<D>::t1, t2 = Axes<D>::t2;
  const double ml = WL[3] * pos_part(WL[n]);
  const double mr = WR[3] * neg_part(WR[n]);
  const double mlb = Fb[3] + Fb[n] * WL[n] + Fb[t1] * WL[t1] + Fb[t2] * WL[t2];
  const double mrb = Fb[3] + Fb[n] * WR[n] + Fb[t1] * WR[t1] + Fb[t2] * WR[t2];
  WLb[3] = 0.0;
  WRb[3] = 0.0;
  WLb[n] = Fb[n] * ml;
  WLb[t1] = Fb[t1] * ml;
  WLb[t2] = Fb[t2] * ml;
  WRb[n] = Fb[n] * mr;
  WRb[t1] = Fb[t1] * mr;
  WRb[t2] = Fb[t2] * mr;
  if (positive(WL[n])) {
    WLb[3] += mlb * WL[n];
    WLb[n] += mlb * WL[3];
  }
  if (positive(-WR[n])) {
    WRb[3] += mrb * WR[n];
    WRb[n] += mrb * WR[3];
  }
}

// ------------------------------------------------------------------ reconstruction adjoint
// Cotangents (bm, b0, bp) of the three cell deviations for cotangents gm, gp
// on the face values, at the branches br that parabola_branches took: each
// face value is e0 -/+ (alpha dm + beta dp) with the branch's two weights
// (lw = {w6 w0, w6 w1}, the upper limiter's).
template <bool UNI>
__device__ __forceinline__ void parabola_vjp(unsigned br, const double* w, const double* lw, double gm, double gp,
                                             double& bm, double& b0, double& bp) {
  const bool live = br & 1, first = br & 2, A = br & 4, B = br & 8;
  const double am = !live ? 0.0 : (A ? (UNI ? 0.375 : w[2]) : (first ? (UNI ? 1.0 : w[0]) : 0.0));
  const double ap = !live ? 0.0 : (A ? (UNI ? 0.125 : w[3]) : (first ? 0.0 : (UNI ? 1.0 : w[1])));
  const double cm = !live ? 0.0 : (B ? (UNI ? 0.125 : w[4]) : (first ? (UNI ? 1.0 : lw[0]) : 0.0));
  const double cp = !live ? 0.0 : (B ? (UNI ? 0.375 : w[5]) : (first ? 0.0 : (UNI ? 1.0 : lw[1])));
  const double dmb = fma(gp, cm, -(gm * am)), dpb = fma(gp, cp, -(gm * ap));
  bm = -dmb;
  bp = dpb;
  b0 = (gm + gp) + (dmb - dpb);
}

// ------------------------------------------------------------------ drag and source adjoints
// Cotangent li of the drag input U (pre-drag state) for a cotangent lo of its
// output (apply_drag over tau); returns lo . dD/dSt.
__device__ __forceinline__ double drag_vjp(const DevGrid& g, int i, const double* U, const double* lo, double* li,
                                           double tau, const DragArgs& d) {
#pragma unroll
  for (int f = 0; f < 9; ++f) li[f] = lo[f];
  const double rg = U[RHO], rd = U[DRHO];
  if (!has_mass(rd) || !positive(rg)) return 0.0;
  const double ig = recip(rg), id = recip(rd);
  double P = 0.0;
  if (d.law != 0) P = (g.gamma - 1.0) * fma(-0.5 * ig, fma(U[MU], U[MU], fma(U[MV], U[MV], U[MW] * U[MW])), U[EN]);
  const double a = tau * inv_stopping_time<true>(g, i, rg, ig, P, d, 0);
  // the momentum that changes hands is K (v_d - v_g), K = rho_d a / (1 + k),
  // k = a (1 + rho_d / rho_g)
  const double eps = rd * ig, q = recip(1.0 + fma(a, eps, a)), aq = a * q, K = rd * aq;
  const double e = lo[EN];
  double Kb = 0.0, rgb = 0.0, rdb = 0.0;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double vg = U[MU + c] * ig;
    const double vd = U[DMU + c] * id;
    const double dv = vd - vg;
    const double X = K * dv;
    const double vp = fma(X, ig, vg);
    const double dE = 0.5 * X * (vp + vg);
    const double Xb = fma(e, vp, lo[MU + c] - lo[DMU + c]);
    const double dvb = Xb * K, dg = dvb * ig, dd = dvb * id;
    li[MU + c] += fma(e * X, ig, -dg);
    li[DMU + c] += dd;
    rgb += fma(dg, vg, -(e * dE * ig));
    rdb = fma(-dd, vd, rdb);
    Kb = fma(Xb, dv, Kb);
  }
  rdb = fma(Kb * aq, fma(-aq, eps, 1.0), rdb);
  rgb = fma(Kb * (K * aq), eps * ig, rgb);
  const double ab = Kb * (rd * (q * q)), aab = ab * a;  // cotangent of a, times a
  if (d.law != 0) {
    // 1 / t_s = rho_g c_s / rhos_rp with c_s = sqrt(gamma P / rho_g); in the
    // Stokes regime (drag law 2 above r_p = 9 lambda / 4, the forward's branch)
    // 1 / t_s = (9/4) c_s / (kappa rhos_rp), with no explicit rho_g
    const bool stokes_regime = d.law == 2 && positive(d.kappa * rg - 2.25);
    if (!stokes_regime) rgb = fma(aab, ig, rgb);
    const double Pb = 0.5 * aab * recip(P), gm1 = g.gamma - 1.0;
    rgb = fma(-0.5 * aab, ig, rgb);
    li[EN] += Pb * gm1;
    double k2 = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double v = U[MU + c] * ig;
      li[MU + c] -= Pb * gm1 * v;
      k2 = fma(v, v, k2);
    }
    rgb += Pb * gm1 * 0.5 * k2;
  }
  li[RHO] += rgb;
  li[DRHO] += rdb;
  return -aab * d.ist[0];  // t_s is proportional to St in every law: -a a_b = t_s t_s_b
}

// out += s S'(U)^T for the App. B sources at a cell (cylindrical only).
__device__ __forceinline__ void sources_vjp(const DevGrid& g, int i, int k, const double* U, const double* s,
                                            double* out) {
  const double ir = g.ir[i], Om2 = 2.0 * g.omega;
  const size_t o = (size_t)k * g.nr + i;
  const double A1 = g.grav[o], fz = g.grav[(size_t)g.nz * g.nr + o];
  const double gm1 = g.gamma - 1.0;
  {
    const double iq = recip(U[RHO]);
    const double u = U[MU] * iq, v = U[MV] * iq, w = U[MW] * iq;
    const double sg = s[MU] * (gm1 * ir), vr = v * ir, ur = u * ir;
    out[MU] += fma(s[EN], A1, -fma(sg, u, s[MV] * (vr + Om2)));
    out[MV] += fma(s[MU], fma(2.0, vr, Om2), -fma(sg, v, s[MV] * ur));
    out[MW] += fma(s[EN], fz, -(sg * w));
    out[EN] += sg;
    out[RHO] += fma(s[MU], fma(-v, vr, A1), fma(0.5 * sg, fma(u, u, fma(v, v, w * w)), fma(s[MV] * u, vr, s[MW] * fz)));
  }
  if (g.nf > 5 && has_mass(U[DRHO])) {
    const double iq = recip(U[DRHO]);
    const double u = U[DMU] * iq, v = U[DMV] * iq, vr = v * ir;
    out[DMU] -= s[DMV] * (vr + Om2);
    out[DMV] += fma(s[DMU], fma(2.0, vr, Om2), -(s[DMV] * (u * ir)));
    out[DRHO] += fma(s[DMU], fma(-v, vr, A1), fma(s[DMV] * u, vr, s[DMW] * fz));
  }
}

// ------------------------------------------------------------------ kernels
struct AdjPointArgs {
  DevGrid g;
  const double* Y[9];      // pre-drag stage output
  const double* lout[9];   // cotangent of the stage output
  const double* Ein[9];    // stage input (the sources are evaluated on it)
  double* M[9];            // out: mu' = tau / V mu
  double* lam_n[9];        // cotangent of E^n: written in stage 2, accumulated in stage 1
  double* lam_in[9];       // stage 2: cotangent of E*, written (stage 1: unused)
  double tau;
  DragArgs drag;
  int stage2;
  double* partials;        // [gridDim.x] block sums of lambda_out . dD/dSt
  double* ind_partials;    // indirect gravity on: [2][gridDim.x] block sums of dJ/dA, dJ/dB (without X_ref)
};

constexpr int ADJ_PT_NT = 256;

template <int NF>
__global__ void __launch_bounds__(ADJ_PT_NT) adj_point_kernel(const AdjPointArgs a) {
  __shared__ double red[ADJ_PT_NT / 32];
  const DevGrid& g = a.g;
  const size_t ncell = (size_t)g.nr * g.nth * g.nz;
  double dst = 0.0;
  double pa = 0.0, pb = 0.0;  // indirect gravity: cotangents of A_disc, B_disc (over X_ref)
  for (size_t lin = blockIdx.x * (size_t)ADJ_PT_NT + threadIdx.x; lin < ncell; lin += (size_t)gridDim.x * ADJ_PT_NT) {
    const int gi = (int)(lin % g.nr);
    const int gk = (int)(lin / ((size_t)g.nr * g.nth));
    double lo[9], mu[9], U[9];
#pragma unroll
    for (int f = 0; f < 9; ++f) lo[f] = U[f] = 0.0;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      lo[f] = a.lout[f][lin];
      U[f] = a.Y[f][lin];
    }
    if (NF == 9) {
      dst += drag_vjp(g, gi, U, lo, mu, a.tau, a.drag);
    } else {
#pragma unroll
      for (int f = 0; f < 9; ++f) mu[f] = lo[f];
    }
    const double iv = g.ivol[gi];
    double src[9];
#pragma unroll
    for (int f = 0; f < 9; ++f) src[f] = 0.0;
    if (g.geom == GEOM_CYL) {
      double E[9], s[9];
#pragma unroll
      for (int f = 0; f < 9; ++f) {
        E[f] = f < NF ? a.Ein[f][lin] : 0.0;
        s[f] = a.tau * mu[f];
      }
      sources_vjp(g, gi, gk, E, s, src);
      if (g.damp_k) {  // wave-killing zones: d(-V k E'_f)/dE_f = -V k
        const double kd = g.damp_k[(size_t)gk * g.nr + gi];
#pragma unroll
        for (int f = 0; f < 5; ++f) src[f] -= kd * s[f];
      }
      if (g.x_ind != 0.0) {
        // indirect gravity, S = -(rho gr, rho gt, 0, m_u gr + m_v gt) and
        // -(rho_d gr, rho_d gt, 0) for dust: its local part at fixed
        // (gr, gt), and P = dJ/dgr, Q = dJ/dgt, which reach A and B through
        // gr = X (A c + B s), gt = X (-A s + B c)
        const int gj = (int)((lin / g.nr) % g.nth);
        const double gr = g.ind_g[gj], gt = g.ind_g[g.nth + gj];
        src[RHO] -= s[MU] * gr + s[MV] * gt;
        src[MU] -= s[EN] * gr;
        src[MV] -= s[EN] * gt;
        double P = -(s[MU] * E[RHO] + s[EN] * E[MU]);
        double Q = -(s[MV] * E[RHO] + s[EN] * E[MV]);
        if (NF == 9 && has_mass(E[DRHO])) {
          src[DRHO] -= s[DMU] * gr + s[DMV] * gt;
          P -= s[DMU] * E[DRHO];
          Q -= s[DMV] * E[DRHO];
        }
        const double c = g.ind_cs[gj], sn = g.ind_cs[g.nth + gj];
        pa += P * c - Q * sn;
        pb += P * sn + Q * c;
      }
    }
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      a.M[f][lin] = a.tau * iv * mu[f];
      if (a.stage2) {
        a.lam_n[f][lin] = mu[f];
        a.lam_in[f][lin] = src[f];
      } else {
        a.lam_n[f][lin] += mu[f] + src[f];
      }
    }
  }
  const double t = block_sum<ADJ_PT_NT>(dst, red);
  if (threadIdx.x == 0) a.partials[blockIdx.x] = t;
  if (g.x_ind != 0.0) {
    const double ta = block_sum<ADJ_PT_NT>(pa, red);
    const double tb = block_sum<ADJ_PT_NT>(pb, red);
    if (threadIdx.x == 0) {
      a.ind_partials[blockIdx.x] = ta;
      a.ind_partials[gridDim.x + blockIdx.x] = tb;
    }
  }
}

// The cotangent that reaches the stage input through the disc moments:
// A = sum w (rho - rho_0 + rho_d) cos(theta), B likewise with sin, so
// lam[RHO] and lam[DRHO] gain X_ref w (dA cos(theta_j) + dB sin(theta_j)),
// (dA, dB) the reduced point-kernel partials; w = V r / R^3 [nz][nr].
static __global__ void __launch_bounds__(ADJ_PT_NT) adj_indirect_bcast_kernel(const DevGrid g, const double* w,
                                                                       const double* dAB, double* lam_rho,
                                                                       double* lam_drho) {
  const size_t ncell = (size_t)g.nr * g.nth * g.nz;
  const double dA = g.x_ind * dAB[0], dB = g.x_ind * dAB[1];
  for (size_t lin = blockIdx.x * (size_t)ADJ_PT_NT + threadIdx.x; lin < ncell; lin += (size_t)gridDim.x * ADJ_PT_NT) {
    const int i = (int)(lin % g.nr);
    const size_t jk = lin / g.nr;
    const int j = (int)(jk % g.nth), k = (int)(jk / g.nth);
    const double v = w[(size_t)k * g.nr + i] * (dA * g.ind_cs[j] + dB * g.ind_cs[g.nth + j]);
    lam_rho[lin] += v;
    if (lam_drho) lam_drho[lin] += v;
  }
}

struct AdjFluxArgs {
  DevGrid g;
  const double* E[9];      // stage input state (full)
  const double* M[9];      // mu'
  double* lam[9];          // += flux part of G'(E)^T mu'
  unsigned* status;
};

// Shared memory of adj_flux_kernel in doubles.
template <int NF, int L, int NL>
constexpr size_t adj_flux_smem_doubles() {
  return (size_t)NF * ((L + 2) + L) * (NL + 1);
}

template <int NF, int D, int L, int NL, int RC>
__global__ void __launch_bounds__(L * NL, 2) adj_flux_kernel(const AdjFluxArgs a) {
  constexpr int T = L - 4;      // cells per line owned by a block
  constexpr int PE = T + 6;     // staged E': cells c0 - 3 .. c0 + T + 2
  constexpr int PM = T + 4;     // staged mu': cells c0 - 2 .. c0 + T + 1
  constexpr int NLP = NL + 1;   // padded line stride
  constexpr int NT = L * NL;
  constexpr unsigned FULL = 0xffffffffu;
  static_assert(L <= 32 && (32 % L) == 0, "a line must fit a warp");
  extern __shared__ double smem[];
  double* sE = smem;
  double* sM = smem + (size_t)NF * PE * NLP;
  const DevGrid& g = a.g;
  const int nd = D == 0 ? g.nr : (D == 1 ? g.nth : g.nz);
  const int na = D == 0 ? g.nth : g.nr;                  // fastest transverse extent
  const int nlines = D == 0 ? g.nth * g.nz : (D == 1 ? g.nr * g.nz : g.nr * g.nth);
  const int ntiles = (nd + T - 1) / T;
  const int c0 = (blockIdx.x % ntiles) * T;
  const int line0 = (blockIdx.x / ntiles) * NL;
  const bool periodic = g.bc_lo[D] == BC_PERIODIC;
  auto cell_of = [&](int line, int cd, int c[3]) {
    const int ta = line % na, tb = line / na;
    c[0] = D == 0 ? cd : ta;
    c[1] = D == 1 ? cd : (D == 0 ? ta : tb);
    c[2] = D == 2 ? cd : tb;
  };

  for (int idx = threadIdx.x; idx < PE * NL; idx += NT) {
    const int pos = D == 0 ? idx % PE : idx / NL;
    const int l = D == 0 ? idx / PE : idx % NL;
    const int line = line0 + l;
    double* dst = sE + pos * NLP + l;
    int c[3];
    cell_of(line, c0 - 3 + pos, c);
    if (line >= nlines || !resolve_cell(g, c)) {
#pragma unroll
      for (int f = 0; f < NF; ++f) dst[(size_t)f * PE * NLP] = 0.0;
      continue;
    }
    const size_t lin = ((size_t)c[2] * g.nth + c[1]) * g.nr + c[0];
    double U[5], W[5];
#pragma unroll
    for (int f = 0; f < 5; ++f) U[f] = a.E[f][lin];
    if (RC == RECON_PRIM) cell_prim_rounded(g.gamma, U, W);
    const double* e0 = RC == RECON_PRIM ? g.w0c : g.e0c;
#pragma unroll
    for (int f = 0; f < 5; ++f) {
      const double v = RC == RECON_PRIM ? W[f] : U[f];
      dst[(size_t)f * PE * NLP] = g.has_eq ? v - e0[((size_t)f * g.nz + c[2]) * g.nr + c[0]] : v;
    }
    if (NF == 9) {  // the dust as primitives (u, v, w, rho_d)
      const double rd = a.E[DRHO][lin], id = has_mass(rd) ? recip(rd) : 0.0;
#pragma unroll
      for (int q = 0; q < 3; ++q) dst[(size_t)(DMU + q) * PE * NLP] = a.E[DMU + q][lin] * id;
      dst[(size_t)DRHO * PE * NLP] = rd;
    }
  }
  for (int idx = threadIdx.x; idx < PM * NL; idx += NT) {
    const int pos = D == 0 ? idx % PM : idx / NL;
    const int l = D == 0 ? idx / PM : idx % NL;
    const int line = line0 + l;
    double* dst = sM + pos * NLP + l;
    int cd = c0 - 2 + pos;
    bool ok = line < nlines;
    if (cd < 0 || cd >= nd) {
      if (periodic) {
        cd %= nd;
        if (cd < 0) cd += nd;
      } else {
        ok = false;  // no cell: faces beyond the domain carry no cotangent
      }
    }
    if (!ok) {
#pragma unroll
      for (int f = 0; f < NF; ++f) dst[(size_t)f * PM * NLP] = 0.0;
      continue;
    }
    int c[3];
    cell_of(line, cd, c);
    const size_t lin = ((size_t)c[2] * g.nth + c[1]) * g.nr + c[0];
#pragma unroll
    for (int f = 0; f < NF; ++f) dst[(size_t)f * PM * NLP] = a.M[f][lin];
  }
  __syncthreads();

  const int p = threadIdx.x % L, l = threadIdx.x / L;
  const int line = line0 + l;
  const bool line_ok = line < nlines;
  const int c = c0 - 2 + p;
  int cc[3];
  cell_of(line_ok ? line : 0, c, cc);
  const int gi = cc[0], gk = cc[2];
  const int ci = clampi(gi, 0, g.nr - 1), ck = clampi(gk, 0, g.nz - 1);
  const double gam = g.gamma;
  unsigned status = 0;
  auto sv = [&](int f, int q) -> double { return sE[((size_t)f * PE + q) * NLP + l]; };
  auto sm = [&](int f, int q) -> double { return sM[((size_t)f * PM + q) * NLP + l]; };
  // equilibrium on a face: conservative, or primitive with RC = RECON_PRIM
  auto eq_face = [&](int f, int fd) -> double {
    const double* tc = RC == RECON_PRIM ? g.w0c : g.e0c;
    const double* tr = RC == RECON_PRIM ? g.w0r : g.e0r;
    const double* tz = RC == RECON_PRIM ? g.w0z : g.e0z;
    if (D == 0) return tr[((size_t)f * g.nz + ck) * (g.nr + 1) + clampi(fd, 0, g.nr)];
    if (D == 1) return tc[((size_t)f * g.nz + ck) * g.nr + ci];
    return tz[((size_t)f * (g.nz + 1) + clampi(fd, 0, g.nz)) * g.nr + ci];
  };
  constexpr bool UNI = D != 0;
  double w[RCW], lw[2];
  parabola_weights<double, D>(g.rcoef, gi, g.nr, w);
  if (!UNI) {
    lw[0] = w[6] * w[0];
    lw[1] = w[6] * w[1];
  }

  // ---- forward reconstruction of this lane's cell: the primitives of the
  // right state of its lower face (WR, 1 / rho irm) and of the left state of
  // its upper face (WP, irp), and the branches taken
  double WR[5], WP[5], irm = 0.0, irp = 0.0;
  unsigned br[5];
  bool fallback = false;
  {
    double qm[5], qp[5];
    if (RC == RECON_PRIM) {
      double v[9];
      slope_weights<D>(g, gi, v);
#pragma unroll
      for (int f = 0; f < 5; ++f) br[f] = slope_branches(sv(f, p), sv(f, p + 1), sv(f, p + 2), v, qm[f], qp[f]);
    } else {
#pragma unroll
      for (int f = 0; f < 5; ++f)
        br[f] = parabola_branches<UNI>(sv(f, p), sv(f, p + 1), sv(f, p + 2), w, qm[f], qp[f]);
    }
    auto face_states = [&]() {
      if (g.has_eq) {  // its radial and vertical velocities are zero
#pragma unroll
        for (int f : {MV, EN, RHO}) {
          qm[f] += eq_face(f, c);
          qp[f] += eq_face(f, c + 1);
        }
      }
      if (RC == RECON_PRIM) {
#pragma unroll
        for (int f = 0; f < 5; ++f) {
          WR[f] = qm[f];
          WP[f] = qp[f];
        }
      } else {
        irm = gas_prim(gam, qm, WR);
        irp = gas_prim(gam, qp, WP);
      }
      return positive(qm[RHO]) && positive(qp[RHO]) && positive(WR[EN]) && positive(WP[EN]);
    };
    if (!face_states() && line_ok) {  // the forward's positivity fallback: flat departures
      fallback = true;
#pragma unroll
      for (int f = 0; f < 5; ++f) qm[f] = qp[f] = sv(f, p + 1);
      face_states();
    }
  }
  // ---- the face below this cell: cotangents of its two states
  const bool has_face = line_ok && p >= 1;
  const double area = D == 0 ? g.area_r[clampi(c, 0, g.nr)] : (D == 1 ? g.area_t[ci] : g.area_z[ci]);
  auto flux_cot = [&](int f) -> double { return has_face ? area * (sm(f, p) - sm(f, p - 1)) : 0.0; };
  const bool own = line_ok && p >= 2 && p < T + 2 && c < nd;
  const size_t lin = ((size_t)cc[2] * g.nth + cc[1]) * g.nr + cc[0];
  // what a cell receives of field cotangents tm, t0, tp on the cells c - 1, c,
  // c + 1, the zero-gradient ghosts' folded into the edge cell they copy
  const bool out_lo = g.bc_lo[D] == BC_OUTFLOW, out_hi = g.bc_hi[D] == BC_OUTFLOW;
  auto gather = [&](double tm, double t0, double tp) -> double {
    const double from_above = __shfl_down_sync(FULL, tm, 1, L);
    const double from_below = __shfl_up_sync(FULL, tp, 1, L);
    double tot = t0 + (p < L - 1 ? from_above : 0.0) + (p > 0 ? from_below : 0.0);
    if (out_lo || out_hi) {
      const double u1 = __shfl_up_sync(FULL, tot, 1, L), u2 = __shfl_up_sync(FULL, tot, 2, L);
      const double d1 = __shfl_down_sync(FULL, tot, 1, L), d2 = __shfl_down_sync(FULL, tot, 2, L);
      if (out_lo && c == 0 && p >= 2) tot += u1 + u2;
      if (out_hi && c == nd - 1 && p + 2 < L) tot += d1 + d2;
    }
    return tot;
  };
  {
    double ULb[5], URb[5];  // of the left state (the lane below's WP) and of this lane's WR
    {
      double WL[5], Fb[5];
#pragma unroll
      for (int f = 0; f < 5; ++f) {
        WL[f] = __shfl_up_sync(FULL, WP[f], 1, L);
        Fb[f] = flux_cot(f);
      }
      if (has_face) {
        gas_flux_vjp<D, RC>(g.near, WL, WR, Fb, ULb, URb, status);
      } else {
#pragma unroll
        for (int f = 0; f < 5; ++f) ULb[f] = URb[f] = 0.0;
      }
    }
    // cotangents of this cell's face values: lower from its own face, upper from the lane above
    double gp[5], tot[5];
#pragma unroll
    for (int f = 0; f < 5; ++f) {
      const double up = __shfl_down_sync(FULL, ULb[f], 1, L);
      gp[f] = p < L - 1 ? up : 0.0;
    }
    if (RC != RECON_PRIM) {  // through W = gas_prim(U) of the face states
      prim_vjp(gam, irm, WR, URb);
      prim_vjp(gam, irp, WP, gp);
    }
#pragma unroll
    for (int f = 0; f < 5; ++f) {
      double tm, t0, tp;
      if (fallback) {
        tm = tp = 0.0;
        t0 = URb[f] + gp[f];
      } else {
        parabola_vjp<UNI>(br[f], w, lw, URb[f], gp[f], tm, t0, tp);
      }
      tot[f] = gather(tm, t0, tp);
    }
    if (own) {
      if (RC == RECON_PRIM) {  // primitive-deviation cotangents back to the conservative fields
        double U[5], Ub[5];
#pragma unroll
        for (int f = 0; f < 5; ++f) U[f] = a.E[f][lin];
        gas_prim_vjp(gam, U, tot, Ub);
#pragma unroll
        for (int f = 0; f < 5; ++f) a.lam[f][lin] += Ub[f];
      } else {
#pragma unroll
        for (int f = 0; f < 5; ++f) a.lam[f][lin] += tot[f];
      }
    }
  }
  if (NF == 9) {  // the dust, whose fluxes and sums share nothing with the gas's
    double WLb[4], WRb[4], dm[4], dp[4], tot[4];
    unsigned bd[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      bd[q] = parabola_branches<UNI>(sv(5 + q, p), sv(5 + q, p + 1), sv(5 + q, p + 2), w, dm[q], dp[q]);
    {
      double WL[4], Fb[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        WL[q] = __shfl_up_sync(FULL, dp[q], 1, L);
        Fb[q] = flux_cot(5 + q);
      }
      if (has_face) {
        dust_flux_vjp<D>(WL, dm, Fb, WLb, WRb);
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) WLb[q] = WRb[q] = 0.0;
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double up = __shfl_down_sync(FULL, WLb[q], 1, L);
      double tm, t0, tp;
      parabola_vjp<UNI>(bd[q], w, lw, WRb[q], p < L - 1 ? up : 0.0, tm, t0, tp);
      tot[q] = gather(tm, t0, tp);
    }
    if (own) {  // the primitives' cotangents back to (rho_d u, rho_d v, rho_d w, rho_d)
      const double rd = sv(8, p + 1), id = has_mass(rd) ? recip(rd) : 0.0;
      double rb = tot[3];
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const double m = tot[q] * id;
        a.lam[5 + q][lin] += m;
        rb = fma(-m, sv(5 + q, p + 1), rb);
      }
      a.lam[DRHO][lin] += rb;
    }
  }
  if (status) atomicOr(a.status, status);
}

struct Fields9 {
  double* p[9];
};

// Stage-1 drag on its own: out = D(Y) over tau (E* from the pre-drag state).
static __global__ void __launch_bounds__(ADJ_PT_NT) drag_only_kernel(DevGrid g, const Fields9 Y, const Fields9 out,
                                                             double tau, DragArgs d) {
  const size_t ncell = (size_t)g.nr * g.nth * g.nz;
  for (size_t lin = blockIdx.x * (size_t)ADJ_PT_NT + threadIdx.x; lin < ncell; lin += (size_t)gridDim.x * ADJ_PT_NT) {
    double U[9];
#pragma unroll
    for (int f = 0; f < 9; ++f) U[f] = Y.p[f][lin];
    const double id = recip(U[DRHO]);
    apply_drag<true, 1>(g, (int)(lin % g.nr), U, tau, d, recip(U[RHO]), &id);
#pragma unroll
    for (int f = 0; f < 9; ++f) out.p[f][lin] = U[f];
  }
}

// Fixed-order sum of the d/dSt block partials of both stages; adds the
// result to this call's slot [0] and to the running total [1].
static __global__ void __launch_bounds__(512) adj_dst_reduce_kernel(const double* partials, int n, double* slots) {
  __shared__ double red[512 / 32];
  double v = 0.0;
  for (int b = threadIdx.x; b < n; b += 512) v += partials[b];
  v = block_sum<512>(v, red);
  if (threadIdx.x == 0) {
    slots[0] = v;
    slots[1] += v;
  }
}

}  // namespace rossbi
