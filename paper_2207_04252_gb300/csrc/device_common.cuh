// Device-side data structures and per-cell / per-face physics of the RoSSBi3D
// step (arXiv:2207.04252).  Included by the kernel translation units only.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "riemann_near.cuh"

namespace rossbi {

// Conservative variables in App. B order, then the dust fluid; dust species
// s occupies fields 5 + 4 s .. 8 + 4 s in the same order (species 0 is DMU ..
// DRHO).
enum { MU = 0, MV = 1, MW = 2, EN = 3, RHO = 4, DMU = 5, DMV = 6, DMW = 7, DRHO = 8 };
constexpr int ND_MAX = 4;                 // dust species
constexpr int NF_MAX = 5 + 4 * ND_MAX;    // conservative fields
enum { GEOM_BOX = 0, GEOM_CYL = 1 };
enum { BC_PERIODIC = 0, BC_OUTFLOW = 1, BC_EQUILIBRIUM = 2 };
enum { STATUS_NONPHYSICAL = 1u, STATUS_RIEMANN = 2u };
// Gas reconstruction (Sect. 2.7): the paper's component-wise parabola on the
// conservative departures E' = E - E0 of App. B's variables, or the parabola
// on the departures of the primitive variables (rho, u, v, w, P).
enum { RECON_CONS = 0, RECON_PRIM = 1 };

constexpr int RCW = 8;  // parabola weights per axis-0 cell

// Grid data the kernels read.  Passed by value as a kernel parameter; the
// pointers are device tables owned by the host runtime.
struct DevGrid {
  int geom, nr, nth, nz, nf, has_eq;
  int recon;             // RECON_CONS or RECON_PRIM
  int bc_lo[3], bc_hi[3];
  double gamma, gm, omega, cfl;
  double dx[3];          // spacing of the uniform axes 1, 2 (and axis 0 of the Box)
  const double* rcoef;   // axis-0 parabola weights for cells i in [-1, nr]: RCW per cell at (i + 1) * RCW
  const double* rslope;  // axis-0 slopes and distances for slope_branches: 9 per cell at (i + 1) * 9
  const double* vol;     // V(i)
  const double* ivol;    // 1 / V(i)
  const double* area_r;  // A of the axis-0 face i - 1/2, i in [0, nr]
  const double* area_t;  // A of an axis-1 face of a cell with radial index i
  const double* area_z;  // A of an axis-2 face of a cell with radial index i
  const double* aov;     // largest face area of a cell with radial index i over its volume
  const double* ir;      // 1 / r of the cell centre (cylindrical)
  const double* omk;     // Omega_K at the cell centre (cylindrical), 1 in the Box
  const double* grav;    // [2][nz][nr] cylindrical: f_r + Omega^2 r, f_z at the cell centres
  const double* e0c;     // equilibrium gas state at centres   [5][nz][nr]
  const double* e0r;     // equilibrium gas state at r faces   [5][nz][nr + 1]
  const double* e0z;     // equilibrium gas state at z faces   [5][nz + 1][nr]
  const double* w0c;     // equilibrium primitive gas state (u, v, w, P, rho in the
  const double* w0r;     //   field slots MU, MV, MW, EN, RHO) at centres, r faces and
  const double* w0z;     //   z faces, same layouts as e0c / e0r / e0z
  const double* r0;      // balanced residual G(E0)            [5][nz][nr]
  // indirect gravity (Sect. 2.10): X_ref (0 = off); cos / sin of the
  // axis-1 cell centres [2][nth]; and, for the stage's input state, the
  // gradient of the indirect potential in (r, theta) components at each
  // axis-1 index [2][nth], in double and in float
  double x_ind;
  const double* ind_cs;
  const double* ind_g;
  const float* ind_gf;
  // damping zones (Sect. 2.4; the de Val-Borro et al. 2006 relaxation): the
  // rate of the radial wave-killing zones plus that of the vertical damped
  // boundary at each cell centre [nz][nr], in double and in float, or null
  const double* damp_k;
  const float* damp_kf;
  // dust species s has the Stokes number St x st_factor[s] (st_factor[0] = 1)
  double st_factor[ND_MAX];
  NearCoef near;         // series of the exact Riemann solution near p_K
};

// Division of 0 <= n < 2^31 by a divisor fixed on the host (multiplication by
// a rounded-up reciprocal; Granlund & Montgomery 1994): three instructions
// where a division takes about 25, in every warp of every block.
struct FastDiv {
  unsigned d, mul, shift;
  __device__ __forceinline__ int operator()(int n) const { return (int)((__umulhi((unsigned)n, mul) + (unsigned)n) >> shift); }
};
inline FastDiv fast_div(unsigned d) {
  FastDiv f{d, 0, 0};
  while ((1ull << f.shift) < d) ++f.shift;
  f.mul = (unsigned)(((1ull << 32) * ((1ull << f.shift) - d)) / d + 1);
  return f;
}
// Tile numbers run r fastest, then z, then theta: the tiles whose halos a tile
// re-reads (its r, z and theta neighbours) run at most tiles_r x tiles_z
// blocks apart, so the re-reads hit in L2.
struct TileOrder {
  FastDiv r, z;  // tiles along r and z
  int k_first;   // first z index of the tiles (0, or a slab's)
  __device__ __forceinline__ void origin(int tile, int tr, int tt, int tz, int& i0, int& j0, int& k0) const {
    const int rest = r(tile), t = z(rest);
    i0 = (tile - rest * (int)r.d) * tr;
    k0 = k_first + (rest - t * (int)z.d) * tz;
    j0 = t * tt;
  }
};

__host__ __device__ constexpr int pow2ceil(int v) {
  int p = 1;
  while (p < v) p <<= 1;
  return p;
}

// Normal / transverse momentum fields for a face normal to axis D.
template <int D> struct Axes;
template <> struct Axes<0> { static constexpr int n = MU, t1 = MV, t2 = MW; };
template <> struct Axes<1> { static constexpr int n = MV, t1 = MU, t2 = MW; };
template <> struct Axes<2> { static constexpr int n = MW, t1 = MU, t2 = MV; };

// ------------------------------------------------------------------ Riemann
// Exact solution of the 1D Riemann problem (Sect. 2.6; the paper takes the
// solver of Toro, ch. 4), sampled on the face (x/t = 0).  Newton iteration on
// the star pressure from the primitive-variable estimate, then the wave
// pattern decides which state sits on the face.
struct RSide {
  double rho, u, p, c;
};

__device__ __forceinline__ void pressure_fn(double g, const RSide& K, double p, double& f, double& fd) {
  if (p <= K.p) {  // rarefaction branch
    const double prat = p / K.p;
    const double e = pow(prat, (g - 1.0) / (2.0 * g));
    f = 2.0 * K.c / (g - 1.0) * (e - 1.0);
    fd = e / (prat * K.rho * K.c);
  } else {         // shock branch
    const double A = 2.0 / ((g + 1.0) * K.rho);
    const double B = (g - 1.0) / (g + 1.0) * K.p;
    const double q = sqrt(A / (B + p));
    f = (p - K.p) * q;
    fd = (1.0 - 0.5 * (p - K.p) / (B + p)) * q;
  }
}

// Fan state at x/t = 0 inside a left (sgn = +1) or right (sgn = -1) rarefaction.
__device__ __forceinline__ void fan_state(double g, const RSide& K, double sgn, double& rho, double& u, double& p) {
  const double cf = 2.0 / (g + 1.0) * (K.c + sgn * 0.5 * (g - 1.0) * K.u);
  u = sgn * cf;
  const double ratio = cf / K.c;
  rho = K.rho * pow(ratio, 2.0 / (g - 1.0));
  p = K.p * pow(ratio, 2.0 * g / (g - 1.0));
}

// Returns the face state (rho, u_n, p) and the side (-1 left, +1 right, 0 vacuum)
// whose transverse velocity is carried.
__device__ __forceinline__ int riemann_face(double g, double rl, double ul, double pl, double rr, double ur, double pr,
                                            double& rho, double& u, double& p, unsigned& status) {
  const RSide L{rl, ul, pl, sqrt(g * pl / rl)};
  const RSide R{rr, ur, pr, sqrt(g * pr / rr)};
  if (2.0 / (g - 1.0) * (L.c + R.c) <= ur - ul) {  // the waves open a vacuum
    const double sl_star = ul + 2.0 * L.c / (g - 1.0);
    const double sr_star = ur - 2.0 * R.c / (g - 1.0);
    if (0.0 <= sl_star) {
      if (0.0 <= ul - L.c) { rho = rl; u = ul; p = pl; }
      else fan_state(g, L, 1.0, rho, u, p);
      return -1;
    }
    if (0.0 >= sr_star) {
      if (0.0 >= ur + R.c) { rho = rr; u = ur; p = pr; }
      else fan_state(g, R, -1.0, rho, u, p);
      return 1;
    }
    rho = u = p = 0.0;
    return 0;
  }
  const double pfloor = 1e-8 * fmin(pl, pr);
  double ps = fmax(pfloor, 0.5 * (pl + pr) - 0.125 * (ur - ul) * (rl + rr) * (L.c + R.c));
  double fl, fdl, fr, fdr, step = 0.0;
  bool conv = false;
  for (int it = 0; it < 100; ++it) {
    pressure_fn(g, L, ps, fl, fdl);
    pressure_fn(g, R, ps, fr, fdr);
    const double pn = fmax(pfloor, ps - (fl + fr + ur - ul) / (fdl + fdr));
    const double change = 2.0 * fabs(pn - ps) / (pn + ps);
    step = pn - ps;
    ps = pn;
    if (change <= 1e-12) { conv = true; break; }
  }
  if (!conv) status |= STATUS_RIEMANN;
  // f_K at the converged p* from the last evaluation, one Newton step away:
  // the neglected second-order term is below rounding once the change is
  // under 1e-12
  fl += fdl * step;
  fr += fdr * step;
  const double us = 0.5 * (ul + ur) + 0.5 * (fr - fl);
  if (0.0 <= us) {  // face lies left of the contact
    if (ps <= pl) {
      if (0.0 <= ul - L.c) { rho = rl; u = ul; p = pl; return -1; }
      const double ratio = ps / pl;
      if (0.0 > us - L.c * pow(ratio, (g - 1.0) / (2.0 * g))) {
        rho = rl * pow(ratio, 1.0 / g); u = us; p = ps; return -1;
      }
      fan_state(g, L, 1.0, rho, u, p);
      return -1;
    }
    const double ratio = ps / pl;
    if (0.0 <= ul - L.c * sqrt((g + 1.0) / (2.0 * g) * ratio + (g - 1.0) / (2.0 * g))) {
      rho = rl; u = ul; p = pl; return -1;
    }
    const double g6 = (g - 1.0) / (g + 1.0);
    rho = rl * (ratio + g6) / (ratio * g6 + 1.0); u = us; p = ps;
    return -1;
  }
  if (ps > pr) {  // right shock
    const double ratio = ps / pr;
    if (0.0 >= ur + R.c * sqrt((g + 1.0) / (2.0 * g) * ratio + (g - 1.0) / (2.0 * g))) {
      rho = rr; u = ur; p = pr; return 1;
    }
    const double g6 = (g - 1.0) / (g + 1.0);
    rho = rr * (ratio + g6) / (ratio * g6 + 1.0); u = us; p = ps;
    return 1;
  }
  if (0.0 >= ur + R.c) { rho = rr; u = ur; p = pr; return 1; }
  const double ratio = ps / pr;
  if (0.0 <= us + R.c * pow(ratio, (g - 1.0) / (2.0 * g))) {
    rho = rr * pow(ratio, 1.0 / g); u = us; p = ps; return 1;
  }
  fan_state(g, R, -1.0, rho, u, p);
  return 1;
}

// The same solver for gamma = 7/5.  With z_K = (p / p_K)^(1/7) the pressure
// functions, the star density behind a rarefaction and the fan state are
// polynomials in z (exponents (gamma-1)/(2 gamma) = 1/7, 1/gamma = 5/7 ... in
// units of 1/7).  Newton runs on z_L (p = p_L z_L^7, z_R = z_L k with
// k = (p_L / p_R)^(1/7)), so a face takes two powers instead of two per
// iteration; the iterates, the stopping test on p and the sampling are those
// of riemann_face.
// Side constants of the gamma = 7/5 pressure functions, formed once per face:
// 1/(rho c), the shock coefficients A = 2/((gamma+1) rho) (as sqrt(A) and
// 1/A) and B = (gamma-1)/(gamma+1) p_K.
struct RSideZ {
  double irc, sqA, iA, B;
};
__device__ __forceinline__ RSideZ side_z(const RSide& K) {
  RSideZ s;
  s.irc = 1.0 / (K.rho * K.c);
  s.iA = 1.2 * K.rho;
  s.sqA = rsqrt(s.iA);
  s.B = K.p * (1.0 / 6.0);
  return s;
}

// Pressure function of side K at p = p_K z^7 (iz = 1/z): rarefaction
// f = 5 c (z - 1), df/dp = 1 / (rho c z^6); shock f = (p - p_K) q with
// q = sqrt(A / (B + p)), df/dp = (1 - (p - p_K) / (2 (B + p))) q, where
// (p - p_K)/(B + p) = (p - p_K) q^2 / A: no division.
__device__ __forceinline__ void pressure_fn_z(const RSide& K, const RSideZ& S, double p, double z, double iz,
                                              double& f, double& fd) {
  if (z <= 1.0) {
    const double i3 = iz * iz * iz;
    f = 5.0 * K.c * (z - 1.0);
    fd = S.irc * i3 * i3;
  } else {
    const double q = S.sqA * rsqrt(S.B + p);
    const double dp = p - K.p;
    f = dp * q;
    fd = (1.0 - 0.5 * dp * q * q * S.iA) * q;
  }
}

// Newton on z_L = (p / p_L)^(1/7) (p = p_L z_L^7, z_R = z_L k with
// k = (p_L / p_R)^(1/7)) from the start ps, z; on return ps, z are the last
// iterate, f*, fd* the pressure functions at the one before and step the last
// change of p.  The stopping test 2 |dp| <= 1e-12 (p_new + p_old) is that of
// riemann_face without its division.
__device__ __forceinline__ bool newton_z_g75(const RSide& L, const RSide& R, double du, double pfloor, double k,
                                             double& ps, double& z, double& fl, double& fdl, double& fr,
                                             double& fdr, double& step) {
  const RSideZ SL = side_z(L), SR = side_z(R);
  const double ik = 1.0 / k;
  for (int it = 0; it < 100; ++it) {
    const double iz = 1.0 / z;
    pressure_fn_z(L, SL, ps, z, iz, fl, fdl);
    pressure_fn_z(R, SR, ps, z * k, iz * ik, fr, fdr);
    // Newton on z_L: dp/dz_L = 7 p / z_L
    double zn = z - (fl + fr + du) * z / (7.0 * ps * (fdl + fdr));
    double z2 = zn * zn, z7 = z2 * z2 * z2 * zn;
    double pn = L.p * z7;
    if (!(pn >= pfloor)) {
      pn = pfloor;
      zn = pow(pfloor / L.p, 1.0 / 7.0);
    }
    step = pn - ps;
    const bool done = 2.0 * fabs(step) <= 1e-12 * (pn + ps);
    ps = pn;
    z = zn;
    if (done) return true;
  }
  return false;
}

// y^(1/7).  Near 1 (|y - 1| <= 2^-10, the common case of smooth flow, where
// p* and the two side pressures differ little) the binomial series of
// (1 + x)^(1/7) to x^5, whose truncation is below 2e-20 relative, saves
// GB300's narrow FP64 pipe a logarithm and an exponential; pow elsewhere.
__device__ __forceinline__ double root7(double y) {
  const double x = y - 1.0;
  if (fabs(x) <= 0.0009765625) {
    return 1.0 + x * (0.14285714285714285714 +           // 1/7
                      x * (-0.061224489795918367347 +    // -3/49
                           x * (0.037900874635568513120 +   // 13/343
                                x * (-0.027072053311120366514 +  // -65/2401
                                     x * 0.020884155411435413816))));  // 351/16807
  }
  return pow(y, 1.0 / 7.0);
}

__device__ __forceinline__ void fan_state_g75(const RSide& K, double sgn, double& rho, double& u, double& p) {
  const double cf = (K.c + sgn * 0.2 * K.u) / 1.2;
  u = sgn * cf;
  const double r = cf / K.c, r2 = r * r, r5 = r2 * r2 * r;
  rho = K.rho * r5;
  p = K.p * r5 * r2;
}

__device__ __forceinline__ int riemann_face_g75(double rl, double ul, double pl, double rr, double ur, double pr,
                                                double& rho, double& u, double& p, unsigned& status) {
  constexpr double g = 1.4;
  const RSide L{rl, ul, pl, sqrt(g * pl / rl)};
  const RSide R{rr, ur, pr, sqrt(g * pr / rr)};
  if (5.0 * (L.c + R.c) <= ur - ul) {  // the waves open a vacuum
    const double sl_star = ul + 5.0 * L.c;
    const double sr_star = ur - 5.0 * R.c;
    if (0.0 <= sl_star) {
      if (0.0 <= ul - L.c) { rho = rl; u = ul; p = pl; }
      else fan_state_g75(L, 1.0, rho, u, p);
      return -1;
    }
    if (0.0 >= sr_star) {
      if (0.0 >= ur + R.c) { rho = rr; u = ur; p = pr; }
      else fan_state_g75(R, -1.0, rho, u, p);
      return 1;
    }
    rho = u = p = 0.0;
    return 0;
  }
  const double pfloor = 1e-8 * fmin(pl, pr);
  double ps = fmax(pfloor, 0.5 * (pl + pr) - 0.125 * (ur - ul) * (rl + rr) * (L.c + R.c));
  const double k = root7(pl / pr);
  double z = root7(ps / pl);
  double fl, fdl, fr, fdr, step = 0.0;
  if (!newton_z_g75(L, R, ur - ul, pfloor, k, ps, z, fl, fdl, fr, fdr, step)) status |= STATUS_RIEMANN;
  fl += fdl * step;  // f_K at the converged p*, one Newton step from the last evaluation
  fr += fdr * step;
  const double us = 0.5 * (ul + ur) + 0.5 * (fr - fl);
  if (0.0 <= us) {  // face lies left of the contact
    if (ps <= pl) {
      if (0.0 <= ul - L.c) { rho = rl; u = ul; p = pl; return -1; }
      if (0.0 > us - L.c * z) {
        const double z2 = z * z;
        rho = rl * z2 * z2 * z; u = us; p = ps; return -1;
      }
      fan_state_g75(L, 1.0, rho, u, p);
      return -1;
    }
    const double ratio = ps / pl;
    if (0.0 <= ul - L.c * sqrt((g + 1.0) / (2.0 * g) * ratio + (g - 1.0) / (2.0 * g))) {
      rho = rl; u = ul; p = pl; return -1;
    }
    const double g6 = (g - 1.0) / (g + 1.0);
    rho = rl * (ratio + g6) / (ratio * g6 + 1.0); u = us; p = ps;
    return -1;
  }
  if (ps > pr) {  // right shock
    const double ratio = ps / pr;
    if (0.0 >= ur + R.c * sqrt((g + 1.0) / (2.0 * g) * ratio + (g - 1.0) / (2.0 * g))) {
      rho = rr; u = ur; p = pr; return 1;
    }
    const double g6 = (g - 1.0) / (g + 1.0);
    rho = rr * (ratio + g6) / (ratio * g6 + 1.0); u = us; p = ps;
    return 1;
  }
  if (0.0 >= ur + R.c) { rho = rr; u = ur; p = pr; return 1; }
  const double zr = z * k;
  if (0.0 <= us + R.c * zr) {
    const double z2 = zr * zr;
    rho = rr * z2 * z2 * zr; u = us; p = ps; return 1;
  }
  fan_state_g75(R, -1.0, rho, u, p);
  return 1;
}

// The general solver, out of line: faces near a strong wave or in the sonic
// band.  By value: pointers would keep the callers' face states in memory.
struct RFace {
  double rho, u, p;
  int side;         // -1 left, +1 right, 0 vacuum: whose transverse velocity is carried
  unsigned status;
};
static __device__ __noinline__ RFace riemann_general(double g, double rl, double ul, double pl, double rr, double ur,
                                                     double pr) {
  RFace o;
  o.status = 0;
  o.side = g == 1.4 ? riemann_face_g75(rl, ul, pl, rr, ur, pr, o.rho, o.u, o.p, o.status)
                    : riemann_face(g, rl, ul, pl, rr, ur, pr, o.rho, o.u, o.p, o.status);
  return o;
}

// Primitive gas state (u, v, w, P, rho), in the field slots MU, MV, MW, EN,
// RHO, of a conservative gas state; returns 1 / rho.
__device__ __forceinline__ double gas_prim(double g, const double* U, double* W) {
  const double ir = recip(U[RHO]);
  W[MU] = U[MU] * ir;
  W[MV] = U[MV] * ir;
  W[MW] = U[MW] * ir;
  W[EN] = (g - 1.0) * fma(-0.5, fma(U[MU], W[MU], fma(U[MV], W[MV], U[MW] * W[MW])), U[EN]);
  W[RHO] = U[RHO];
  return ir;
}

// The conversion of a cell that the primitive option takes its departures
// from, with a rounded division.  Departures can be nothing but this rounding
// (an isobaric density perturbation has no pressure departure), and then the
// limiter's branches, which the adjoint differentiates, are decided by it: the
// arithmetic here and in slope_branches is part of the result.
__device__ __forceinline__ void cell_prim_rounded(double g, const double* U, double* W) {
  const double ir = 1.0 / U[RHO];
  W[MU] = U[MU] * ir;
  W[MV] = U[MV] * ir;
  W[MW] = U[MW] * ir;
  W[EN] = (g - 1.0) * (U[EN] - 0.5 * (U[MU] * U[MU] + U[MV] * U[MV] + U[MW] * U[MW]) * ir);
  W[RHO] = U[RHO];
}

// Cotangent Ub of the conservative gas state U for a cotangent Wb of its
// primitive state W = gas_prim(U) (the transpose of the conversion's
// Jacobian at U).
__device__ __forceinline__ void gas_prim_vjp(double g, const double* U, const double* Wb, double* Ub) {
  const double ir = recip(U[RHO]), gm1 = g - 1.0;
  const double v0 = U[MU] * ir, v1 = U[MV] * ir, v2 = U[MW] * ir;
  const double bP = Wb[EN];
  Ub[MU] = Wb[MU] * ir - gm1 * bP * v0;
  Ub[MV] = Wb[MV] * ir - gm1 * bP * v1;
  Ub[MW] = Wb[MW] * ir - gm1 * bP * v2;
  Ub[EN] = gm1 * bP;
  Ub[RHO] = Wb[RHO] - (Wb[MU] * v0 + Wb[MV] * v1 + Wb[MW] * v2) * ir + gm1 * bP * 0.5 * (v0 * v0 + v1 * v1 + v2 * v2);
}

// The same in place, b the cotangent of W on entry and of U on return, from
// W and ir = 1 / rho.
__device__ __forceinline__ void prim_vjp(double g, double ir, const double* W, double* b) {
  const double pb = (g - 1.0) * b[EN];
  const double k2 = fma(W[MU], W[MU], fma(W[MV], W[MV], W[MW] * W[MW]));
  const double dot = fma(b[MU], W[MU], fma(b[MV], W[MV], b[MW] * W[MW]));
  b[RHO] = fma(0.5 * pb, k2, fma(-dot, ir, b[RHO]));
  b[MU] = fma(b[MU], ir, -(pb * W[MU]));
  b[MV] = fma(b[MV], ir, -(pb * W[MV]));
  b[MW] = fma(b[MW], ir, -(pb * W[MW]));
  b[EN] = pb;
}

// Gas flux A F(E*) through a face of area A normal to axis D from the
// reconstructed left and right primitive states (App. B flux vector; energy
// flux (E + P) u_n).
template <int D>
__device__ __forceinline__ void gas_face_flux(const NearCoef& C, double area, const double* WL, const double* WR,
                                              double* F, unsigned& status) {
  constexpr int n = Axes<D>::n, t1 = Axes<D>::t1, t2 = Axes<D>::t2;
  if (!positive(WL[RHO]) || !positive(WR[RHO]) || !positive(WL[EN]) || !positive(WR[EN])) {
    status |= STATUS_NONPHYSICAL;
#pragma unroll
    for (int f = 0; f < 5; ++f) F[f] = 0.0;
    return;
  }
  NearStar<double> s;
  const int kind = near_riemann<NEAR_STATE>(C, WL[RHO], WL[n], WL[EN], WR[RHO], WR[n], WR[EN], WR[EN] - WL[EN],
                                        WR[n] - WL[n], 0.0, false, WL[n], WR[n], s);
  const bool left = kind == NEAR_LEFT || kind == NEAR_STAR_L;
  double rho = left ? WL[RHO] : WR[RHO], u = left ? WL[n] : WR[n], p = left ? WL[EN] : WR[EN];
  double ut1 = left ? WL[t1] : WR[t1], ut2 = left ? WL[t2] : WR[t2];
  if (kind >= NEAR_STAR_L) {
    rho += s.drho;
    u = s.us;
    p = WL[EN] + s.d;
  }
  if (kind == NEAR_GENERAL) {
    const RFace o = riemann_general(C.gamma, WL[RHO], WL[n], WL[EN], WR[RHO], WR[n], WR[EN]);
    status |= o.status;
    rho = o.rho;
    u = o.u;
    p = o.p;
    ut1 = o.side < 0 ? WL[t1] : (o.side > 0 ? WR[t1] : 0.0);
    ut2 = o.side < 0 ? WL[t2] : (o.side > 0 ? WR[t2] : 0.0);
  }
  const double m = area * (rho * u), pa = area * p;
  F[RHO] = m;
  F[n] = fma(m, u, pa);
  F[t1] = m * ut1;
  F[t2] = m * ut2;
  F[EN] = fma(scale_down<1>(m), fma(u, u, fma(ut1, ut1, ut2 * ut2)), C.g_gm1 * (pa * u));
}

// Flux of the pressureless dust fluid (Sect. 2.9 "adapted" solver) by kinetic
// flux-vector splitting (Bouchut, Jin & Li 2003): the matter moving right
// crosses from the left face state, the matter moving left from the right one.
// WL, WR hold face primitives (u, v, w, rho_d); F the dust fluxes in the
// order (rho_d u, rho_d v, rho_d w, rho_d), times the face's area, for a face
// normal to axis D.
template <int D, class T>
__device__ __forceinline__ void dust_kinetic_flux(T area, const T* WL, const T* WR, T* F) {
  constexpr int n = Axes<D>::n, t1 = Axes<D>::t1, t2 = Axes<D>::t2;  // 0..2 in the dust block
  if constexpr (sizeof(T) == 8) {
    // one of the two parts is zero unless the streams collide (u_L > 0 > u_R):
    // five FP64 operations for the upwind side instead of eleven for both
    const bool fromL = positive(WL[n]);
    const T rho = fromL ? WL[3] : WR[3], un = fromL ? WL[n] : neg_part(WR[n]);
    F[3] = area * (rho * un);
#pragma unroll
    for (int q = 0; q < 3; ++q) F[q] = F[3] * (fromL ? WL[q] : WR[q]);
    if (fromL && sign_bit(WR[n])) {
      const T mr = area * (WR[3] * WR[n]);
      F[3] += mr;
#pragma unroll
      for (int q = 0; q < 3; ++q) F[q] = fma(mr, WR[q], F[q]);
    }
    return;
  }
  const T ml = area * (WL[3] * pos_part(WL[n]));
  const T mr = area * (WR[3] * neg_part(WR[n]));
  F[3] = ml + mr;
  F[n] = ml * WL[n] + mr * WR[n];
  F[t1] = ml * WL[t1] + mr * WR[t1];
  F[t2] = ml * WL[t2] + mr * WR[t2];
}

// ------------------------------------------------------------------ sources
// G += V S, S the App. B sources per unit volume at the cell centre: geometric
// terms, stellar gravity (Sect. 2.1), the rotating-frame Coriolis /
// centrifugal terms and, when switched on, the indirect gravity of Sect. 2.10
// (force -grad Phi_ind on gas and dust, and its work on the gas); the Box has
// none.  W: the cell's primitive gas state; Vd: the azimuthal dust velocity
// of each species, zero where it has no mass.  XT = false compiles the optional
// terms out.
template <bool XT, int NF>
__device__ __forceinline__ void add_sources(const DevGrid& g, int i, int j, int k, const double* U, const double* W,
                                            const double* Vd, double* G) {
  const double V = g.vol[i], ir = g.ir[i], Om2 = 2.0 * g.omega;
  const size_t o = (size_t)k * g.nr + i;
  const double a1 = g.grav[o], fz = g.grav[(size_t)g.nz * g.nr + o];
  double gr = 0.0, gt = 0.0;
  const bool ind = XT && g.x_ind != 0.0;
  if (ind) {
    gr = g.ind_g[j];
    gt = g.ind_g[g.nth + j];  // grad Phi_ind, (r, theta)
  }
  const double ar = XT ? a1 - gr : a1;
  G[MU] = fma(V, fma(ir, fma(U[MV], W[MV], W[EN]), fma(U[RHO], ar, Om2 * U[MV])), G[MU]);
  double sv = -U[MU] * fma(W[MV], ir, Om2), se = fma(U[MU], ar, U[MW] * fz);
  if (ind) {
    sv -= U[RHO] * gt;
    se -= U[MV] * gt;
  }
  G[MV] = fma(V, sv, G[MV]);
  G[MW] = fma(V, U[RHO] * fz, G[MW]);
  G[EN] = fma(V, se, G[EN]);
#pragma unroll
  for (int b = 5; b < NF; b += 4) {  // each dust species
    const double v = Vd[(b - 5) / 4], rd = U[b + 3];
    if (!has_mass(rd)) continue;
    G[b] = fma(V, fma(U[b + 1], fma(v, ir, Om2), rd * ar), G[b]);
    double sd = -U[b] * fma(v, ir, Om2);
    if (ind) sd -= rd * gt;
    G[b + 1] = fma(V, sd, G[b + 1]);
    G[b + 2] = fma(V, rd * fz, G[b + 2]);
  }
}

// ------------------------------------------------------------------ drag
struct DragArgs {
  double stokes;
  double rhos_rp;  // Epstein constant rho_s r_p (drag laws 1 and 2)
  int law;
  double kappa;    // drag law 2: r_p / lambda_0, the mean free path being lambda_0 / rho_g
  // 1 / (St x factor) and 1 / (rho_s r_p x factor) of each species, formed on
  // the host: a division per cell and species is eight FP64 operations
  double ist[ND_MAX], irr[ND_MAX];
};

// 1 / t_s of dust species s (Stokes number St x st_factor[s]) in a cell of
// radial index i with gas density rg (ig = 1 / rg) and pressure P (Sect. 2.9): drag law 0
// t_s = St / Omega_K(r) (the Box: St); laws 1 and 2 Epstein t_s = rho_s r_p /
// (rho_g c_s), rho_s r_p proportional to St, with c_s = sqrt(gamma P / rho_g)
// (gamma P rho_g underflows in a thin atmosphere); law 2 (compiled in with XT) adds the Stokes regime of Sect. 2.9:
// above r_p = 9 lambda / 4 the Epstein time grows by (4/9) r_p / lambda.
template <bool XT>
__device__ __forceinline__ double inv_stopping_time(const DevGrid& g, int i, double rg, double ig, double P,
                                                    const DragArgs& d, int s) {
  if (d.law == 0) return g.omk[i] * d.ist[s];
  double it = rg * root(g.gamma * P * ig) * d.irr[s];
  if (XT && d.law == 2) {
    const double x = d.kappa * rg;
    if (positive(x - 2.25)) it *= 2.25 * recip(x);
  }
  return it;
}

// Semi-implicit drag over a stage of length tau (Sect. 2.9 drag law).  One
// dust species: the relative gas-dust velocity relaxes by 1 / (1 + k), k =
// tau (1 + eps) / t_s, at fixed barycentric velocity; with a = tau / t_s the
// momentum that changes hands is rho_d a / (1 + k) times the velocity
// difference (no reduced mass to form).  ND > 1 species: the backward-Euler
// system of the gas coupled to each species (no dust-dust exchange) in closed
// form, v_g' = (rho_g v_g + sum rho_k w_k v_k) / (rho_g + sum rho_k w_k),
// v_k' = (v_k + a_k v_g') / (1 + a_k), with a_k = tau / t_k and w_k =
// a_k / (1 + a_k).  The gas energy gains the work done on the gas in both.
// ig = 1 / rho_g, id = 1 / rho_d of each species (any value without mass).
template <bool XT, int ND>
__device__ __forceinline__ void apply_drag(const DevGrid& g, int i, double* U, double tau, const DragArgs& d,
                                           double ig, const double* id) {
  const double rg = U[RHO];
  if (!positive(rg)) return;
  double P = 0.0;
  if (d.law != 0)
    P = (g.gamma - 1.0) * fma(-0.5 * ig, fma(U[MU], U[MU], fma(U[MV], U[MV], U[MW] * U[MW])), U[EN]);
  if constexpr (ND == 1) {
    const double rd = U[DRHO];
    if (!has_mass(rd)) return;
    const double a = tau * inv_stopping_time<XT>(g, i, rg, ig, P, d, 0);
    const double K = rd * a * recip(1.0 + fma(a * rd, ig, a));
    double dE = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double vg = U[MU + c] * ig;
      const double X = K * fma(U[DMU + c], id[0], -vg);
      U[MU + c] += X;
      U[DMU + c] -= X;
      dE = fma(X, fma(0.5 * ig, X, vg), dE);
    }
    U[EN] += dE;
  } else {
    double a[ND], h[ND], num[3], den = rg;  // h = 1 / (1 + a), 0 for a species without mass
#pragma unroll
    for (int c = 0; c < 3; ++c) num[c] = U[MU + c];
#pragma unroll
    for (int s = 0; s < ND; ++s) {
      const int b = 5 + 4 * s;
      a[s] = h[s] = 0.0;
      if (!has_mass(U[b + 3])) continue;
      a[s] = tau * inv_stopping_time<XT>(g, i, rg, ig, P, d, s);
      h[s] = recip(1.0 + a[s]);
      const double w = a[s] * h[s];
      den = fma(U[b + 3], w, den);
#pragma unroll
      for (int c = 0; c < 3; ++c) num[c] = fma(U[b + c], w, num[c]);
    }
    const double iden = recip(den);
    double dE = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double vg = num[c] * iden, m = rg * vg;
      const double X = m - U[MU + c];  // what the gas gains
#pragma unroll
      for (int s = 0; s < ND; ++s) {
        const int b = 5 + 4 * s;
        if (!has_mass(U[b + 3])) continue;
        U[b + c] = h[s] * fma(U[b + 3] * a[s], vg, U[b + c]);
      }
      dE = fma(0.5 * X, fma(U[MU + c], ig, vg), dE);
      U[MU + c] = m;
    }
    U[EN] += dE;
  }
}

// ------------------------------------------------------------------ CFL
// Sect. 2.5, Eq. (cfl condition): the largest (|v| + c) A / V and |v_d| A / V
// of one cell of radial index i (the step is N_CFL over their maximum: one
// division per block instead of one per cell), and whether the cell is not
// physical.  ig, id: as apply_drag.
template <int NF>
__device__ __forceinline__ double cell_rate(const DevGrid& g, int i, const double* U, double ig, const double* id,
                                            bool& bad) {
  const double u = U[MU] * ig, v = U[MV] * ig, w = U[MW] * ig;
  const double q = fma(u, u, fma(v, v, w * w));
  const double P = (g.gamma - 1.0) * fma(-0.5 * U[RHO], q, U[EN]);
  bad = !positive(U[RHO]) || !positive(P);
  double rate = root(g.gamma * P * ig) + (positive(q) ? root(q) : 0.0);
#pragma unroll
  for (int b = 5; b < NF; b += 4) {
    const double j = id[(b - 5) / 4], ud = U[b] * j, vd = U[b + 1] * j, wd = U[b + 2] * j;
    const double d2 = fma(ud, ud, fma(vd, vd, wd * wd));
    if (has_mass(U[b + 3]) && positive(d2)) {
      const double vel = root(d2);
      if (mag_less(rate, vel)) rate = vel;
    }
    bad |= !non_negative(U[b + 3]);
  }
  return rate * g.aov[i];
}

}  // namespace rossbi
