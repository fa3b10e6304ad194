// The physics of the perturbation forms (state E' = E - E0) and the RK2 stage
// kernel of the double one (the float one has stage_f32.cuh).
//
// Same tiling and sweeps as the FP64 full-state kernel, but every quantity is
// formed as an exact algebraic difference from the equilibrium state E0
// (App. A), so that the balanced right-hand side G(E0 + E') - G(E0) of Sect.
// 2.8 is computed without ever forming the large equilibrium terms (the
// Keplerian centrifugal and gravity terms are O(rho v_K^2 / r), the
// perturbations 1e-4 of that and less):
//   - the parabola and limiter of Sect. 2.7 act on the conservative
//     departures E' themselves (the state), and the face state E0 + q is
//     turned into primitive perturbations about the face equilibrium,
//     rho = rho0 + rho', du = (m' - rho' u0)/rho,
//     dP = (gamma-1)(E' - [rho' |u0|^2/2 + rho u0.du + rho |du|^2/2]);
//     with RC = RECON_PRIM the same conversion is applied to each cell and
//     the parabola acts on the primitive perturbations instead;
//   - the exact Riemann solution (Sect. 2.6) comes from the series near p_K
//     (riemann_near.cuh) in the differences of the two side perturbations;
//     where they do not reach, a solver out of line iterates on dp* = p* - p0
//     with the pressure functions written in p/p_K - 1 (log1p / expm1 for the
//     rarefaction powers), samples the wave pattern on full values and returns
//     the face-state perturbation; near-sonic fans use the FP64-derived
//     u0 -/+ c0 of the face;
//   - fluxes are differences F(W0 + dW) - F(W0) expanded by hand;
//   - sources use the FP64-derived equilibrium coefficient
//     C_r = f_r + Omega^2 r + v0^2/r + 2 Omega v0 = (1/rho0) dP0/dr.
// The Riemann problem falls back to the FP64 full-state solver on vacuum
// generation, strong rarefaction (p* < p_K / 10) or slow Newton convergence;
// the fallbacks are counted.
//
// The double kernel is bound as the full-state one is, by the FP64 pipe (84 %
// busy), and laid out the same; one bi-fluid step of 93 x 131 x 37 cells took
// 9.75 ms with an FP64 Newton iteration and divisions per face, and takes 2.5.
#pragma once
#include "stage_full.cuh"

namespace rossbi {

// Equilibrium and metric tables in the state precision.  A cell's or a face's
// values are adjacent, so that a lane takes them in 16-byte loads from one
// address.
template <class T>
struct PertTables {
  const T* cen;      // [nz][nr][8] rho0, v0, p0, C_r, f_z, f_r + Omega^2 r, 2 v0/r + 2 Omega, 1/r
  const T* face[3];  // [..][4] rho0, v0, p0, h0 (= E0 + p0) on r faces [nz][nr+1], theta faces (= centres)
                     // [nz][nr] and z faces [nz+1][nr]
  const T* wave[3];  // [..][4] c0, u0 - c0, u0 + c0 (u0 normal to the face), for the general solver
  const T* rcoef;  // axis-0 parabola weights, RCW per cell as DevGrid::rcoef
  const T* vol;
  const T* ivol;
  const T* area_r;
  const T* area_t;
  const T* area_z;
  const T* aov;    // largest face area over the volume
  const T* omk;    // Omega_K at the cell-centre radius (constant-St drag)
  unsigned long long* fallbacks;  // count of FP64 fallback Riemann faces
};

template <class T> struct Math;
template <> struct Math<float> {
  static __device__ __forceinline__ float log1p_(float x) { return log1pf(x); }
  static __device__ __forceinline__ float expm1_(float x) { return expm1f(x); }
  static __device__ __forceinline__ float sqrt_(float x) { return sqrtf(x); }
  static __device__ __forceinline__ float abs_(float x) { return fabsf(x); }
  static constexpr float eps = 1.1920929e-7f;
  static constexpr int max_iter = 24;
};
template <> struct Math<double> {
  static __device__ __forceinline__ double log1p_(double x) { return log1p(x); }
  static __device__ __forceinline__ double expm1_(double x) { return expm1(x); }
  static __device__ __forceinline__ double sqrt_(double x) { return sqrt(x); }
  static __device__ __forceinline__ double abs_(double x) { return fabs(x); }
  static constexpr double eps = 2.220446049250313e-16;
  static constexpr int max_iter = 60;
};

// (1 + x)^a - 1, accurate for small x.
template <class T>
__device__ __forceinline__ T pow1pm1(T x, T a) {
  return Math<T>::expm1_(a * Math<T>::log1p_(x));
}
// sqrt(1 + t) - 1, accurate for small t.
template <class T>
__device__ __forceinline__ T sqrt1pm1(T t) {
  return t / (Math<T>::sqrt_(T(1) + t) + T(1));
}

// Powers of the exact solver, (1 + x)^a - 1 for the exponents it needs.
// Generic gamma: log1p / expm1.
template <class T>
struct PowGeneric {
  static constexpr bool series = false;
  static __device__ __forceinline__ T rar(T x, T g) { return pow1pm1(x, (g - T(1)) / (T(2) * g)); }
  static __device__ __forceinline__ T dens(T x, T g, T) { return pow1pm1(x, T(1) / g); }
  static __device__ __forceinline__ T fan_rho(T y, T g) { return pow1pm1(y, T(2) / (g - T(1))); }
  static __device__ __forceinline__ T fan_p(T y, T g) { return pow1pm1(y, T(2) * g / (g - T(1))); }
};
// gamma = 7/5 in float: with z = (1 + x)^(1/7), z^7 - 1 = (z - 1)(1 + z + ... + z^6)
// gives (1 + x)^(1/7) - 1 = x / sum z^k, accurate to a few times the error of
// the hardware log2 / exp2 estimate of z; (1 + x)^(5/7) - 1 = (z - 1)(1 + z +
// z^2 + z^3 + z^4); the fan exponents 5 and 7 are exact polynomials.
struct PowG75 {
  // Near p = p_K (|x| <= xs, x = p/p_K - 1) the pressure function of a side
  // is f = (c/gamma) x S(x) and f' = T(x)/(rho c), with S, T the Taylor
  // series of the rarefaction branch (x <= 0: S = ((1+x)^(1/7) - 1)/(x/7),
  // T = (1+x)^(-6/7)) or the shock branch (x > 0: S = (1 + 6x/7)^(-1/2),
  // T = (1 + 6x/7)^(-3/2) (1 + 3x/7)) to x^4; the branches agree to x^2 (f is
  // C^2 at p_K).  Truncation at |x| = 1/32: 4e-9 relative in f, 2.2e-8 in f'.
  static constexpr bool series = true;
  static constexpr float xs = 0.03125f;
  static constexpr float inv_gamma = 0.714285714f;
  static constexpr float beta = 0.142857143f;  // (gamma - 1) / (2 gamma)
  static __device__ __forceinline__ void pressure_series(float x, float& S, float& Td) {
    const bool rar = x <= 0.0f;
    const float s2 = rar ? 0.265306122f : 0.275510204f;    // 13/49 | 27/98
    const float s3 = rar ? -0.189504373f : -0.196793003f;  // -65/343 | -135/686
    const float s4 = rar ? 0.146189088f : 0.147594752f;    // 351/2401 | 2835/19208
    const float t2 = rar ? 0.795918367f : 0.826530612f;    // 39/49 | 81/98
    const float t3 = rar ? -0.758017493f : -0.787172012f;  // -260/343 | -270/343
    const float t4 = rar ? 0.730945440f : 0.737973761f;    // 1755/2401 | 14175/19208
    S = 1.0f + x * (-0.428571429f + x * (s2 + x * (s3 + x * s4)));
    Td = 1.0f + x * (-0.857142857f + x * (t2 + x * (t3 + x * t4)));
  }
  static __device__ __forceinline__ float rar(float x, float) {
    const float z = exp2f(__log2f(1.0f + x) * 0.142857142857f);
    const float s = 1.0f + z * (1.0f + z * (1.0f + z * (1.0f + z * (1.0f + z * (1.0f + z)))));
    return __fdividef(x, s);
  }
  static __device__ __forceinline__ float dens(float, float, float r) {
    const float z = 1.0f + r;
    return r * (1.0f + z * (1.0f + z * (1.0f + z * (1.0f + z))));
  }
  static __device__ __forceinline__ float fan_rho(float y, float) {
    return y * (5.0f + y * (10.0f + y * (10.0f + y * (5.0f + y))));
  }
  static __device__ __forceinline__ float fan_p(float y, float) {
    return y * (7.0f + y * (21.0f + y * (35.0f + y * (35.0f + y * (21.0f + y * (7.0f + y))))));
  }
};

// Face equilibrium as the general solver takes it, in the frame of the face's normal.
template <class T>
struct PFace {
  T rho, un, p, c, un_mc, un_pc;
};

// Perturbation of one side of a face, with the full values the wave pattern needs.
template <class T>
struct PSide {
  T drho, dun, dp;  // perturbations
  T rho, un, p, c;  // full values
};

template <class T>
__device__ __forceinline__ PSide<T> pert_side(T g, const PFace<T>& W0, T drho, T dun, T dp) {
  PSide<T> s;
  s.drho = drho;
  s.dun = dun;
  s.dp = dp;
  s.rho = W0.rho + drho;
  s.p = W0.p + dp;
  s.un = W0.un + dun;
  s.c = Math<T>::sqrt_(g * s.p / s.rho);
  return s;
}

// Reciprocals of a side that the series form of its pressure function uses.
template <class T>
struct PSideInv {
  T ip, cg, irc;  // 1/p, c/gamma, 1/(rho c)
};

// Pressure function of side K at trial p = p0 + d, in perturbation form.
template <class T, class P>
__device__ __forceinline__ void pert_pressure_fn(T g, const PSide<T>& K, const PSideInv<T>& I, T p, T d, T& f,
                                                 T& fd) {
  const T dpk = d - K.dp;  // p - p_K
  if constexpr (P::series) {
    const T x = dpk * I.ip;
    if (Math<T>::abs_(x) <= P::xs) {
      T S, Td;
      P::pressure_series(x, S, Td);
      f = I.cg * x * S;
      fd = I.irc * Td;
      return;
    }
  }
  if (dpk <= T(0)) {
    const T x = dpk / K.p;
    const T r = P::rar(x, g);  // (p/p_K)^((g-1)/2g) - 1
    f = T(2) * K.c / (g - T(1)) * r;
    fd = (T(1) + r) / ((T(1) + x) * K.rho * K.c);
  } else {
    const T A = T(2) / ((g + T(1)) * K.rho);
    const T B = (g - T(1)) / (g + T(1)) * K.p;
    const T q = Math<T>::sqrt_(A / (B + p));
    f = dpk * q;
    fd = (T(1) - T(0.5) * dpk / (B + p)) * q;
  }
}

template <class T, class P>
__device__ __forceinline__ void fan_pert(T g, const PFace<T>& W0, const PSide<T>& K, bool has_eq, bool left, T& drho,
                                         T& dun, T& dp) {
  const T g6 = (g - T(1)) / (g + T(1));
  // c - c0
  const T dc = has_eq ? W0.c * sqrt1pm1((K.dp * W0.rho - W0.p * K.drho) / (W0.p * K.rho)) : K.c;
  if (left) {  // (u_L - c_L) = (u0 - c0) + du_L - dc_L
    const T y = g6 * (W0.un_mc + K.dun - dc) / K.c;
    drho = K.drho + K.rho * P::fan_rho(y, g);
    dp = K.dp + K.p * P::fan_p(y, g);
    dun = -W0.un_mc + dc + K.c * y;
  } else {     // (-u_R - c_R) = -(u0 + c0) - du_R - dc_R
    const T y = g6 * (-W0.un_pc - K.dun - dc) / K.c;
    drho = K.drho + K.rho * P::fan_rho(y, g);
    dp = K.dp + K.p * P::fan_p(y, g);
    dun = -W0.un_pc - dc - K.c * y;
  }
}

// Perturbation of the face state of the exact Riemann solution.  Returns
// 0 on success, 1 when the caller must use the FP64 full-state solver.
template <class T, class P>
__device__ __forceinline__ int pert_riemann(T g, const PFace<T>& W0, const PSide<T>& L, const PSide<T>& R, bool has_eq,
                                            T& drho, T& dun, T& dp, int& side) {
  if (T(2) / (g - T(1)) * (L.c + R.c) <= R.un - L.un) return 1;  // vacuum generation
  const T du = R.dun - L.dun;
  const T floor_p = T(1e-8) * fmin(L.p, R.p);
  T d = T(0.5) * (L.dp + R.dp) - T(0.125) * du * (L.rho + R.rho) * (L.c + R.c);  // PVRS in dp
  if (W0.p + d < floor_p) d = floor_p - W0.p;
  const T scale = Math<T>::abs_(L.dp) + Math<T>::abs_(R.dp) + (L.rho * L.c + R.rho * R.c) * Math<T>::abs_(du);
  PSideInv<T> IL{}, IR{};
  if constexpr (P::series) {
    IL.ip = T(1) / L.p;
    IR.ip = T(1) / R.p;
    IL.cg = L.c * P::inv_gamma;
    IR.cg = R.c * P::inv_gamma;
    IL.irc = T(1) / (L.rho * L.c);
    IR.irc = T(1) / (R.rho * R.c);
  }
  T fl, fdl, fr, fdr, step = T(0);
  bool conv = false;
  for (int it = 0; it < Math<T>::max_iter; ++it) {
    const T p = W0.p + d;
    pert_pressure_fn<T, P>(g, L, IL, p, d, fl, fdl);
    pert_pressure_fn<T, P>(g, R, IR, p, d, fr, fdr);
    T dn = d - (fl + fr + du) / (fdl + fdr);
    if (W0.p + dn < floor_p) dn = floor_p - W0.p;
    step = dn - d;
    const T change = Math<T>::abs_(step);
    d = dn;
    if (change <= T(8) * Math<T>::eps * (scale + Math<T>::abs_(d))) {
      conv = true;
      break;
    }
  }
  if (!conv) return 1;
  const T ps = W0.p + d;
  if (ps < T(0.1) * fmin(L.p, R.p)) return 1;  // strong rarefaction: near vacuum
  // p*/p_K - 1 and the rarefaction power (p*/p_K)^((g-1)/2g) - 1 of a side,
  // from the series near p_K
  auto rel = [&](T dpk, T pk, const PSideInv<T>& I) -> T {
    if constexpr (P::series) return dpk * I.ip;
    else return dpk / pk;
  };
  auto rar = [&](T x) -> T {
    if constexpr (P::series) {
      if (Math<T>::abs_(x) <= P::xs) {
        T S, Td;
        P::pressure_series(x, S, Td);
        return P::beta * x * S;
      }
    }
    return P::rar(x, g);
  };
  // f_K at the converged p* from the last evaluation, one (converged) Newton
  // step away; the second-order remainder is below rounding
  fl += fdl * step;
  fr += fdr * step;
  const T dus = T(0.5) * (L.dun + R.dun) + T(0.5) * (fr - fl);
  const T us = W0.un + dus;
  const T g6 = (g - T(1)) / (g + T(1));
  if (us >= T(0)) {
    side = -1;
    const T x = rel(d - L.dp, L.p, IL);  // p*/p_L - 1
    if (d <= L.dp) {
      if (L.un - L.c >= T(0)) { drho = L.drho; dun = L.dun; dp = L.dp; return 0; }
      const T r = rar(x);
      const T cs = L.c * (T(1) + r);
      if (us - cs < T(0)) { drho = L.drho + L.rho * P::dens(x, g, r); dun = dus; dp = d; return 0; }
      fan_pert<T, P>(g, W0, L, has_eq, true, drho, dun, dp);
      return 0;
    }
    if (L.un - L.c * Math<T>::sqrt_(T(1) + (g + T(1)) / (T(2) * g) * x) >= T(0)) {
      drho = L.drho; dun = L.dun; dp = L.dp; return 0;
    }
    drho = L.drho + L.rho * x * (T(1) - g6) / (T(1) + g6 * (T(1) + x));
    dun = dus;
    dp = d;
    return 0;
  }
  side = 1;
  const T x = rel(d - R.dp, R.p, IR);  // p*/p_R - 1
  if (d > R.dp) {
    if (R.un + R.c * Math<T>::sqrt_(T(1) + (g + T(1)) / (T(2) * g) * x) <= T(0)) {
      drho = R.drho; dun = R.dun; dp = R.dp; return 0;
    }
    drho = R.drho + R.rho * x * (T(1) - g6) / (T(1) + g6 * (T(1) + x));
    dun = dus;
    dp = d;
    return 0;
  }
  if (R.un + R.c <= T(0)) { drho = R.drho; dun = R.dun; dp = R.dp; return 0; }
  const T r = rar(x);
  const T cs = R.c * (T(1) + r);
  if (us + cs > T(0)) { drho = R.drho + R.rho * P::dens(x, g, r); dun = dus; dp = d; return 0; }
  fan_pert<T, P>(g, W0, R, has_eq, false, drho, dun, dp);
  return 0;
}

// Equilibrium of a face: density, azimuthal velocity, pressure and E0 + p0.
template <class T>
struct PEq {
  T rho, v, p, h;
};
__device__ __forceinline__ PEq<float> load_eq(const float* t) {
  const float4 q = *reinterpret_cast<const float4*>(t);
  return {q.x, q.y, q.z, q.w};
}
__device__ __forceinline__ PEq<double> load_eq(const double* t) {
  const double2 q = reinterpret_cast<const double2*>(t)[0], r = reinterpret_cast<const double2*>(t)[1];
  return {q.x, q.y, r.x, r.y};
}

// A (F(W0 + dW) - F(W0)) through a face of area A (App. B flux components,
// energy flux (E + P) u_n), written without forming the equilibrium flux: the
// face state differs from the equilibrium by drho, dp and the velocity
// departures d[MU], d[MV], d[MW].  F in the field slots.
template <class T, int D>
__device__ __forceinline__ void pert_flux(T g_gm1, T area, const PEq<T>& W0, T drho, const T* d, T dp, T* F) {
  constexpr int n = Axes<D>::n;
  T v[3] = {d[MU], W0.v + d[MV], d[MW]};
  const T un = v[n];
  const T dm = drho * un + W0.rho * d[n];  // of the mass flux
  const T du2 = d[MU] * d[MU] + d[MV] * (W0.v + v[MV]) + d[MW] * d[MW];
  const T q2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
  const T dh = T(0.5) * (drho * q2 + W0.rho * du2) + g_gm1 * dp;
  const T dmA = area * dm;
#pragma unroll
  for (int q = 0; q < 3; ++q) F[q] = dmA * v[q];
  if (D == 1) {  // the equilibrium mass flux rho0 v0 carries the velocity departures
    const T m0 = area * (W0.rho * W0.v);
#pragma unroll
    for (int q = 0; q < 3; ++q) F[q] += m0 * d[q];
  }
  F[n] += area * dp;
  F[EN] = area * (dh * un + W0.h * d[n]);
  F[RHO] = dmA;
}

// Face state perturbation of a Riemann solve, the side whose transverse
// velocity it carries (-1 left, +1 right, 0 vacuum) and status bits.
template <class T>
struct PStar {
  T drho, dun, dp;
  int side;
  unsigned status, fallback;  // fallback: the FP64 solver took the face
};

// FP64 full-state solver on W0 + dW for the faces the perturbation solver
// hands back; kept out of line so the common path stays small.  Arguments
// and result by value: a pointer or reference into the caller's frame would
// keep the caller's face states in local memory.
template <class T>
__device__ __noinline__ PStar<T> pert_fallback_fp64(T g, const PFace<T> W0, const PSide<T> L, const PSide<T> R) {
  const double rl = (double)W0.rho + (double)L.drho, rr = (double)W0.rho + (double)R.drho;
  const double ul = (double)W0.un + (double)L.dun, ur = (double)W0.un + (double)R.dun;
  const double pl = (double)W0.p + (double)L.dp, pr = (double)W0.p + (double)R.dp;
  double rho, u, p;
  PStar<T> o;
  o.status = o.fallback = 0;
  o.side = riemann_face((double)g, rl, ul, pl, rr, ur, pr, rho, u, p, o.status);
  o.drho = (T)(rho - (double)W0.rho);
  o.dun = (T)(u - (double)W0.un);
  o.dp = (T)(p - (double)W0.p);
  return o;
}

// The general solver of a face: near a strong wave or in the sonic band.
template <class T, class P>
__device__ __forceinline__ PStar<T> pert_general(T g, const PFace<T> W0, T lr, T lu, T lp, T rr, T ru, T rp,
                                              bool has_eq) {
  PStar<T> o;
  o.side = 0;
  o.status = o.fallback = 0;
  o.drho = o.dun = o.dp = T(0);
  if (!(W0.rho + lr > T(0)) || !(W0.rho + rr > T(0)) || !(W0.p + lp > T(0)) || !(W0.p + rp > T(0))) {
    o.status = STATUS_NONPHYSICAL;
    return o;
  }
  const PSide<T> L = pert_side(g, W0, lr, lu, lp), R = pert_side(g, W0, rr, ru, rp);
  if (pert_riemann<T, P>(g, W0, L, R, has_eq, o.drho, o.dun, o.dp, o.side) != 0) {
    o = pert_fallback_fp64(g, W0, L, R);
    o.fallback = 1;
  }
  return o;
}

// The same out of line for the double kernel, whose sweeps mostly pass it by: one
// copy serves the three directions; arguments and result by value.
template <class T, class P>
__device__ __noinline__ PStar<T> pert_general_call(T g, const PFace<T> W0, T lr, T lu, T lp, T rr, T ru, T rp,
                                                   bool has_eq) {
  return pert_general<T, P>(g, W0, lr, lu, lp, rr, ru, rp, has_eq);
}

template <class T>
struct PertArgs {
  DevGrid g;          // geometry, sizes, boundary conditions, double tables
  PertTables<T> t;
  const T* in[NF_MAX];
  const T* base[NF_MAX];
  T* out[NF_MAX];
  double dt_host;
  const unsigned long long* rate_in;  // as StageArgs
  unsigned long long* rate_out;
  double tau_frac;
  DragArgs drag;
  int stage2;
  unsigned* status;
  TileOrder order;
  int sms;               // SMs of the device
  int tile;              // double form: TILE_*, chosen by the host
  // the grid's and the drag's parameters in the state precision, converted
  // once on the host (GB300's FP64 pipe is narrow: per-use conversions of the
  // double originals cost latency in the float kernel)
  T gam, gm1, g_gm1, om, kappa;
  T ist[ND_MAX], irr[ND_MAX];  // 1 / (St x factor), 1 / (rho_s r_p x factor) of each dust species
};

// Primitive perturbations (du, dv, dw, dP, drho in the field slots MU, MV,
// MW, EN, RHO) of the conservative departure q about an equilibrium state of
// density rho0 and azimuthal velocity v0 (r and z velocities zero):
// rho = rho0 + rho', du = (m' - rho' u0)/rho,
// dP = (gamma-1)(E' - [rho' |u0|^2/2 + rho u0.du + rho |du|^2/2]).
// ir = 1 / rho.
template <class T>
__device__ __forceinline__ void face_prim(T gm1, T v0, const T* q, T ir, T* w) {
  const T m1 = q[MV] - q[RHO] * v0;  // rho dv
  w[MU] = q[MU] * ir;
  w[MV] = m1 * ir;
  w[MW] = q[MW] * ir;
  const T ke = q[MU] * w[MU] + m1 * w[MV] + q[MW] * w[MW];
  w[EN] = gm1 * (q[EN] - (v0 * (T(0.5) * q[RHO] * v0 + m1) + T(0.5) * ke));
  w[RHO] = q[RHO];
}

// Area times the gas flux perturbation through a face normal to axis D of
// equilibrium Em, from the primitive perturbations wl, wm of its left and right
// states; wave_at(): the face's place in the table of wave speeds.  Returns
// whether the face needs the general solver; with GENERAL = false F is then
// left as it is.  In float GENERAL = true takes the general solver at once: its
// faces are those that the other one has left.
template <class T, int D, class P, bool GENERAL, class W>
__device__ __forceinline__ bool pert_face(const PertArgs<T>& a, const PEq<T>& Em, T area, const T* wl, const T* wm,
                                          W&& wave_at, T* F, unsigned& status, unsigned& nfallback) {
  constexpr int n = Axes<D>::n;
  const DevGrid& g = a.g;
  const T un0 = D == 1 ? Em.v : T(0);
  const T rl = Em.rho + wl[RHO], pl = Em.p + wl[EN], rr = Em.rho + wm[RHO], pr = Em.p + wm[EN];
  NearStar<T> st;
  int kind = NEAR_GENERAL;
  if (sizeof(T) == 4 ? !GENERAL : positive(rl) && positive(rr) && positive(pl) && positive(pr))
    kind = near_riemann<NEAR_DEPARTURES>(g.near, rl, wl[n], pl, rr, wm[n], pr, wm[EN] - wl[EN], wm[n] - wl[n], un0, D == 1,
                           un0 + wl[n], un0 + wm[n], st);
  if (!GENERAL && kind == NEAR_GENERAL) return true;
  const bool left = kind == NEAR_LEFT || kind == NEAR_STAR_L;
  T d[3], drho = left ? wl[RHO] : wm[RHO], dp = left ? wl[EN] : wm[EN];
#pragma unroll
  for (int q = 0; q < 3; ++q) d[q] = left ? wl[q] : wm[q];
  if (kind >= NEAR_STAR_L) {
    drho += st.drho;
    d[n] = st.us;
    dp = wl[EN] + st.d;
  }
  bool ok = true;
  if (GENERAL && kind == NEAR_GENERAL) {
    PFace<T> W0{Em.rho, un0, Em.p, T(0), T(0), T(0)};
    if (g.has_eq) {
      const T* wv = a.t.wave[D] + 4 * (size_t)wave_at();
      W0.c = wv[0];
      W0.un_mc = wv[1];
      W0.un_pc = wv[2];
    }
    constexpr auto solve = sizeof(T) == 4 ? pert_general<T, P> : pert_general_call<T, P>;
    const PStar<T> o = solve(a.gam, W0, wl[RHO], wl[n], wl[EN], wm[RHO], wm[n], wm[EN], g.has_eq != 0);
    status |= o.status;
    nfallback += o.fallback;
    ok = !(o.status & STATUS_NONPHYSICAL);
    // the transverse velocity of the side that the face lies on; a vacuum has none
#pragma unroll
    for (int q = 0; q < 3; ++q) d[q] = o.side < 0 ? wl[q] : (o.side > 0 ? wm[q] : (q == MV ? -Em.v : T(0)));
    drho = o.drho;
    d[n] = o.dun;
    dp = o.dp;
  }
  if (ok) pert_flux<T, D>(a.g_gm1, area, Em, drho, d, dp, F);
  return kind == NEAR_GENERAL;
}

// The gas sweep along axis D of the double form: sE holds the staged gas
// departures (conservative, or primitive with RC = RECON_PRIM).
template <int TR, int TT, int TZ, int NT, int D, class P, int RC>
__device__ __forceinline__ void sweep_pert_gas(const PertArgs<double>& a, const double* sE, double* sG, int i0, int j0,
                                               int k0, unsigned& status, unsigned& nfallback) {
  using S = SweepLane<TR, TT, TZ, D>;
  constexpr int BOX = S::BOX, L = S::L, STRIDE = S::STRIDE;
  constexpr unsigned FULL = 0xffffffffu;
  constexpr bool UNI = D != 0;
  const DevGrid& g = a.g;
  for (int base = threadIdx.x & ~31; base < S::ITEMS; base += NT) {
    const S s(g, base + (threadIdx.x & 31), i0, j0, k0);
    if (!__any_sync(FULL, s.do_face)) continue;  // a warp of lines beyond a ragged grid's edge
    double w[RCW];
    parabola_weights<double, D>(g.rcoef, s.gi, g.nr, w);
    const int ci = clampi(s.gi, 0, g.nr - 1), ck = clampi(s.gk, 0, g.nz - 1);
    // the equilibrium of this cell's lower and upper face (clamped; one face
    // for a theta line, whose cells share the radius and height)
    PEq<double> Em{0.0, 0.0, 0.0, 0.0}, Ep{0.0, 0.0, 0.0, 0.0};
    int of = 0;
    if (g.has_eq) {
      const double* f = a.t.face[D];
      if (D == 0) {
        of = ck * (g.nr + 1) + clampi(s.gd, 0, g.nr);
        Em = load_eq(f + 4 * (size_t)of);
        Ep = load_eq(f + 4 * (size_t)(ck * (g.nr + 1) + clampi(s.gd + 1, 0, g.nr)));
      } else if (D == 1) {
        of = ck * g.nr + ci;
        Em = Ep = load_eq(f + 4 * (size_t)of);
      } else {
        of = clampi(s.gd, 0, g.nz) * g.nr + ci;
        Em = load_eq(f + 4 * (size_t)of);
        Ep = load_eq(f + 4 * (size_t)(clampi(s.gd + 1, 0, g.nz) * g.nr + ci));
      }
    }
    double wm[5], wp[5];  // primitive perturbations: right state of the lower face, left state of the upper face
    {
      double qm[5], qp[5];
#pragma unroll
      for (int f = 0; f < 5; ++f) {
        const double* e = sE + f * BOX + s.sidx;
        parabola<UNI>(e[-STRIDE], e[0], e[STRIDE], w, qm[f], qp[f]);
      }
      auto face_states = [&]() {
        if (RC == RECON_PRIM) {
#pragma unroll
          for (int f = 0; f < 5; ++f) {
            wm[f] = qm[f];
            wp[f] = qp[f];
          }
        } else {
          face_prim(a.gm1, Em.v, qm, recip(Em.rho + qm[RHO]), wm);
          face_prim(a.gm1, Ep.v, qp, recip(Ep.rho + qp[RHO]), wp);
        }
        return positive(Em.rho + wm[RHO]) && positive(Ep.rho + wp[RHO]) && positive(Em.p + wm[EN]) &&
               positive(Ep.p + wp[EN]);
      };
      if (!face_states()) {  // positivity fallback: flat reconstruction of the gas fields
#pragma unroll
        for (int f = 0; f < 5; ++f) qm[f] = qp[f] = sE[f * BOX + s.sidx];
        face_states();
      }
    }
    double F[5], wl[5];
#pragma unroll
    for (int f = 0; f < 5; ++f) {
      wl[f] = __shfl_up_sync(FULL, wp[f], 1, L);  // upper face state of the lower neighbour
      F[f] = 0.0;
    }
    if (s.do_face)
      pert_face<double, D, P, true>(a, Em, face_area<D>(g, s.gi, ci), wl, wm, [&]() { return of; }, F, status, nfallback);
#pragma unroll
    for (int f = 0; f < 5; ++f) accumulate<D, L>(F[f], sG + f * S::NCORE + s.core, s.do_acc);
  }
}

// Cell-centre equilibrium coefficients.
template <class T>
struct PCell {
  T rho0, v0, p0, Cr, fz, gr, cor, ir;
};

template <class T>
__device__ __forceinline__ PCell<T> cell_eq(const PertTables<T>& t, const DevGrid& g, int i, int k) {
  PCell<T> c{};
  if (!g.has_eq) return c;
  const T* q = t.cen + 8 * ((size_t)k * g.nr + i);
  const PEq<T> lo = load_eq(q), hi = load_eq(q + 4);
  c.rho0 = lo.rho;
  c.v0 = lo.v;
  c.p0 = lo.p;
  c.Cr = lo.h;
  c.fz = hi.rho;
  c.gr = hi.v;
  c.cor = hi.p;
  c.ir = hi.h;
  return c;
}

// G += V (S(E0 + E') - S(E0)) (App. B sources, stellar gravity, rotating
// frame), cylindrical geometry, plus the whole indirect-gravity source of
// Sect. 2.10 when it is on (the equilibrium's residual carries none).
// w: the cell's primitive gas perturbations; rd, vd: density and velocity
// (u, v, w) of each dust species, zero without mass.
template <class T, int NF, bool XT>
__device__ __forceinline__ void pert_sources(const PertArgs<T>& a, const PCell<T>& c, int j, T V, const T* w,
                                             const T (*dust)[4], T* G) {
  const DevGrid& g = a.g;
  const T Om2 = T(2) * a.om;
  const T rho = c.rho0 + w[RHO], du = w[MU], dv = w[MV], dw = w[MW], dp = w[EN];
  const T v = c.v0 + dv, rv = rho * dv;
  T gr = T(0), gt = T(0);  // grad Phi_ind, (r, theta), tabulated per axis-1 index in the state precision
  const bool ind = XT && g.x_ind != 0.0;
  if (ind) {
    if constexpr (sizeof(T) == 4) {
      gr = g.ind_gf[j];
      gt = g.ind_gf[g.nth + j];
    } else {
      gr = g.ind_g[j];
      gt = g.ind_g[g.nth + j];
    }
  }
  T sr = w[RHO] * c.Cr + rv * (c.cor + dv * c.ir) + dp * c.ir;
  T st = -rho * du * (v * c.ir + Om2);
  T se = rho * (du * c.gr + dw * c.fz);
  if (ind) {
    sr -= rho * gr;
    st -= rho * gt;
    se -= rho * (du * gr + v * gt);
  }
  G[MU] += V * sr;
  G[MV] += V * st;
  G[MW] += V * (w[RHO] * c.fz);
  G[EN] += V * se;
#pragma unroll
  for (int b = 5; b < NF; b += 4) {  // each dust species
    const T* d = dust[(b - 5) / 4];
    const T Vr = has_mass(d[3]) ? V * d[3] : T(0);
    const T dvd = d[1] - c.v0;  // v_d - v0
    T s0 = c.Cr + dvd * (c.cor + dvd * c.ir), s1 = -d[0] * (d[1] * c.ir + Om2);
    if (ind) {
      s0 -= gr;
      s1 -= gt;
    }
    G[b] += Vr * s0;
    G[b + 1] += Vr * s1;
    G[b + 2] += Vr * c.fz;
  }
}

// 1 / t_s of dust species s in a perturbation-form cell (as inv_stopping_time
// of the full-state kernel; gas density rg, ig = 1 / rg, pressure p).
template <class T, bool XT, class I>
__device__ __forceinline__ T pert_inv_stopping_time(const PertArgs<T>& a, int i, T rg, T ig, T p, int s, I&& inverse) {
  if (a.drag.law == 0) return a.t.omk[i] * a.ist[s];
  T it = rg * root(a.gam * p * ig) * a.irr[s];
  if (XT && a.drag.law == 2) {  // Stokes regime of Sect. 2.9 above r_p = 9 lambda / 4
    const T x = a.kappa * rg;
    if (positive(x - T(2.25))) it *= T(2.25) * inverse(x);
  }
  return it;
}

// Semi-implicit drag on a perturbation-form cell state (the closed forms of
// apply_drag; the gas velocity is u0 + du).  Several species: the gas
// velocity moves by D = sum rho_k w_k (v_k - v_g) / (rho_g + sum rho_k w_k)
// and species k by w_k (D - (v_k - v_g)), w_k = a_k / (1 + a_k), every
// quantity a difference of velocities, never the large u0 itself.
// ig = 1 / rho_g, id = 1 / rho_d of each species (any value without mass);
// inverse(x): 1 / x.
template <class T, int NF, bool XT, class I>
__device__ __forceinline__ void pert_drag(const PertArgs<T>& a, const PCell<T>& c, int i, T* q, T tau, T ig,
                                          const T* id, I&& inverse) {
  const T rg = c.rho0 + q[RHO];
  if (!positive(rg)) return;
  const T m1 = q[MV] - q[RHO] * c.v0;
  const T u0[3] = {T(0), c.v0, T(0)};
  const T dug[3] = {q[MU] * ig, m1 * ig, q[MW] * ig};
  T p = T(0);
  if (a.drag.law != 0) {
    const T ke = q[MU] * dug[0] + m1 * dug[1] + q[MW] * dug[2];
    p = c.p0 + a.gm1 * (q[EN] - (c.v0 * (T(0.5) * q[RHO] * c.v0 + m1) + T(0.5) * ke));
  }
  T dE = T(0);
  if constexpr (NF == 9) {
    const T rd = q[DRHO];
    if (!has_mass(rd)) return;
    const T ak = tau * pert_inv_stopping_time<T, XT>(a, i, rg, ig, p, 0, inverse);
    const T K = rd * ak * inverse(T(1) + ak * (T(1) + rd * ig));
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const T vd = (q[DMU + k] - rd * u0[k]) * id[0];  // v_d - u0
      const T X = K * (vd - dug[k]);
      q[MU + k] += X;
      q[DMU + k] -= X;
      dE += X * ((u0[k] + dug[k]) + T(0.5) * ig * X);
    }
  } else {
    constexpr int ND = (NF - 5) / 4;
    T wk[ND], den = rg, num[3] = {T(0), T(0), T(0)};
#pragma unroll
    for (int s = 0; s < ND; ++s) {
      const int b = 5 + 4 * s;
      const T rd = q[b + 3];
      wk[s] = T(0);
      if (!has_mass(rd)) continue;
      const T ak = tau * pert_inv_stopping_time<T, XT>(a, i, rg, ig, p, s, inverse);
      wk[s] = ak * inverse(T(1) + ak);
      den += rd * wk[s];
#pragma unroll
      for (int k = 0; k < 3; ++k) num[k] += rd * wk[s] * ((q[b + k] - rd * u0[k]) * id[s] - dug[k]);
    }
    const T iden = inverse(den);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const T D = num[k] * iden;  // v_g' - v_g
#pragma unroll
      for (int s = 0; s < ND; ++s) {
        const int b = 5 + 4 * s;
        const T rd = q[b + 3];
        if (!has_mass(rd)) continue;
        const T rel = (q[b + k] - rd * u0[k]) * id[s] - dug[k];  // v_k - v_g
        q[b + k] += rd * wk[s] * (D - rel);
      }
      q[MU + k] += rg * D;
      dE += T(0.5) * rg * D * (T(2) * (u0[k] + dug[k]) + D);
    }
  }
  q[EN] += dE;
}

// The largest (|v| + c) A / V and |v_d| A / V of a cell (the CFL step is N_CFL
// over their maximum) and whether the cell is not physical.  ig, id: as pert_drag.
template <class T, int NF>
__device__ __forceinline__ T pert_cell_rate(const PertArgs<T>& a, const PCell<T>& c, int i, const T* q, T ig,
                                            const T* id, bool& bad) {
  const T rho = c.rho0 + q[RHO], m1 = q[MV] - q[RHO] * c.v0;
  const T du = q[MU] * ig, dv = m1 * ig, dw = q[MW] * ig, v = c.v0 + dv;
  const T ke = q[MU] * du + m1 * dv + q[MW] * dw;
  const T p = c.p0 + a.gm1 * (q[EN] - (c.v0 * (T(0.5) * q[RHO] * c.v0 + m1) + T(0.5) * ke));
  bad = !positive(rho) || !positive(p);
  const T v2 = du * du + v * v + dw * dw;
  T rate = root(a.gam * p * ig) + (positive(v2) ? root(v2) : T(0));
#pragma unroll
  for (int b = 5; b < NF; b += 4) {
    const T j = id[(b - 5) / 4], ud = q[b] * j, vd = q[b + 1] * j, wd = q[b + 2] * j;
    const T d2 = ud * ud + vd * vd + wd * wd;
    if (has_mass(q[b + 3]) && positive(d2)) {
      const T vel = root(d2);
      if (!(vel <= rate)) rate = vel;
    }
    bad |= !non_negative(q[b + 3]);
  }
  return rate * a.t.aov[i];
}

// The stage update of cell (gi, gj, gk) from its staged gas e (conservative
// departures, or primitive ones with RC = RECON_PRIM), the primitives of its
// dust and its flux divergence G, raising the thread's CFL rate.  XT: the
// optional terms (indirect gravity, wave-killing zones) are compiled in; the
// plain instantiation carries none of their code.  ce: the cell's equilibrium;
// inverse(x): 1 / x.
template <class T, int NF, int RC, bool XT, class I>
__device__ __forceinline__ void pert_update(const PertArgs<T>& a, const PCell<T>& ce, int gi, int gj, int gk, const T* e,
                                            const T (*dust)[4], T* G, T tau, T& rate, unsigned& status, I&& inverse) {
  constexpr int ND = NF > 5 ? (NF - 5) / 4 : 1;
  const DevGrid& g = a.g;
  const size_t lin = ((size_t)gk * g.nth + gj) * g.nr + gi;
  T w[5];  // primitive perturbations
  if (RC == RECON_CONS) {
    face_prim(a.gm1, ce.v0, e, inverse(ce.rho0 + e[RHO]), w);
  } else {
#pragma unroll
    for (int f = 0; f < 5; ++f) w[f] = e[f];
  }
  if (g.geom == GEOM_CYL) pert_sources<T, NF, XT>(a, ce, gj, a.t.vol[gi], w, dust, G);
  if (XT && g.damp_k) {  // wave-killing zones: the gas departures E' relax towards 0
    T kd;
    if constexpr (sizeof(T) == 4) kd = g.damp_kf[(size_t)gk * g.nr + gi];
    else kd = g.damp_k[(size_t)gk * g.nr + gi];
    if (positive(kd)) {
      const T V = a.t.vol[gi];
#pragma unroll
      for (int f = 0; f < 5; ++f) G[f] -= V * kd * a.in[f][lin];
    }
  }
  const T tv = tau * a.t.ivol[gi];
  T E[NF], ig = T(0), id[ND];
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    // stage 1 updates its own input, whose gas is staged as it is stored
    const T b = !a.stage2 && RC == RECON_CONS && f < 5 ? e[f] : a.base[f][lin];
    E[f] = b + tv * G[f];
  }
  if (NF > 5 || a.stage2) ig = inverse(ce.rho0 + E[RHO]);
#pragma unroll
  for (int b = 5; b < NF; b += 4) {
    E[b + 3] = dust_density(E[b + 3]);
    id[(b - 5) / 4] = inverse(E[b + 3]);
  }
  if constexpr (NF > 5) pert_drag<T, NF, XT>(a, ce, gi, E, tau, ig, id, inverse);
#pragma unroll
  for (int f = 0; f < NF; ++f) a.out[f][lin] = E[f];
  bool bad = false;
  if (a.stage2) {
    const T c = pert_cell_rate<T, NF>(a, ce, gi, E, ig, id, bad);
    if (positive(c) && !(c <= rate)) rate = c;
  } else {
    bad = !positive(ce.rho0 + w[RHO]) || !positive(ce.p0 + w[EN]);
#pragma unroll
    for (int s = 0; s < (NF - 5) / 4; ++s) bad |= !non_negative(dust[s][3]);
  }
  if (bad) status |= STATUS_NONPHYSICAL;
}

// One RK stage of one tile per block (double form).
template <int NF, int TR, int TT, int TZ, int NT, int MINB, class P, bool XT, int RC>
__global__ void __launch_bounds__(NT, MINB) stage_pert_kernel(const PertArgs<double> a) {
  using S = SweepLane<TR, TT, TZ, 0>;
  constexpr int BOX = S::BOX, NCORE = S::NCORE, ND = NF > 5 ? (NF - 5) / 4 : 1;
  extern __shared__ double smem[];
  double* sE = smem;             // [5][BOX] the gas departures, then the four primitives of one dust species at a time
  double* sG = smem + 5 * BOX;   // [NF][NCORE] flux divergence
  const DevGrid& g = a.g;
  int i0, j0, k0;
  a.order.origin(blockIdx.x, TR, TT, TZ, i0, j0, k0);
  unsigned status = 0, nfallback = 0;
  __shared__ double s_tau;
  publish_tau(&s_tau, a.tau_frac, a.dt_host, a.rate_in, g.cfl);
  if (!a.stage2) clear_rate(a.rate_out);
  auto stage = [&](auto&& put) { walk_box<TR, TT, TZ, NT>(g, i0, j0, k0, put); };
  stage([&](int idx, const int* c) {
    double q[5], w[5];
    if (!c) {
#pragma unroll
      for (int f = 0; f < 5; ++f) sE[f * BOX + idx] = 0.0;
      return;
    }
    const size_t lin = ((size_t)c[2] * g.nth + c[1]) * g.nr + c[0];
#pragma unroll
    for (int f = 0; f < 5; ++f) q[f] = a.in[f][lin];
    if (RC == RECON_PRIM) {
      const PEq<double> eq = g.has_eq ? load_eq(a.t.cen + 8 * ((size_t)c[2] * g.nr + c[0])) : PEq<double>{};
      face_prim(a.gm1, eq.v, q, recip(eq.rho + q[RHO]), w);
    }
#pragma unroll
    for (int f = 0; f < 5; ++f) sE[f * BOX + idx] = RC == RECON_PRIM ? w[f] : q[f];
  });
  __syncthreads();
  sweep_pert_gas<TR, TT, TZ, NT, 0, P, RC>(a, sE, sG, i0, j0, k0, status, nfallback);
  __syncthreads();
  sweep_pert_gas<TR, TT, TZ, NT, 1, P, RC>(a, sE, sG, i0, j0, k0, status, nfallback);
  __syncthreads();
  sweep_pert_gas<TR, TT, TZ, NT, 2, P, RC>(a, sE, sG, i0, j0, k0, status, nfallback);
  __syncthreads();
  dust_species<NF, TR, TT, TZ, NT>(g, a.in, sE, sG, stage, i0, j0, k0);
  double rate = 0.0;
  for (int cidx = threadIdx.x; cidx < NCORE; cidx += NT) {
    const int x = cidx % TR, y = (cidx / TR) % TT, z = cidx / (TR * TT);
    const int gi = i0 + x, gj = j0 + y, gk = k0 + z;
    if (gi >= g.nr || gj >= g.nth || gk >= g.nz) continue;
    const size_t lin = ((size_t)gk * g.nth + gj) * g.nr + gi;
    double e[5], dust[ND][4], G[NF];
#pragma unroll
    for (int f = 0; f < 5; ++f) e[f] = a.in[f][lin];
#pragma unroll
    for (int f = 0; f < NF; ++f) G[f] = sG[f * NCORE + cidx];
#pragma unroll
    for (int b = 5; b < NF; b += 4) {
      double* d = dust[(b - 5) / 4];
      d[3] = a.in[b + 3][lin];
      const double id = has_mass(d[3]) ? recip(d[3]) : 0.0;
#pragma unroll
      for (int q = 0; q < 3; ++q) d[q] = a.in[b + q][lin] * id;
    }
    // e is the state as it is stored, whatever the sweeps reconstructed from
    pert_update<double, NF, RECON_CONS, XT>(a, cell_eq(a.t, g, gi, gk), gi, gj, gk, e, dust, G, s_tau, rate, status,
                                            [](double x) { return recip(x); });
  }
  if (a.stage2) raise_rate(a.rate_out, rate);
  if (status) atomicOr(a.status, status);
  if (nfallback) atomicAdd(a.t.fallbacks, (unsigned long long)nfallback);
}

// Largest CFL rate of a perturbation-form state (Sect. 2.5) into *slot.
template <class T, int NF>
__global__ void pert_cfl_kernel(const PertArgs<T> a, unsigned long long* slot) {
  const DevGrid& g = a.g;
  const size_t ncell = (size_t)g.nr * g.nth * g.nz;
  T rate = T(0);
  unsigned status = 0;
  for (size_t lin = blockIdx.x * (size_t)256 + threadIdx.x; lin < ncell; lin += (size_t)gridDim.x * 256) {
    T q[NF], id[NF > 5 ? (NF - 5) / 4 : 1];
#pragma unroll
    for (int f = 0; f < NF; ++f) q[f] = a.in[f][lin];
#pragma unroll
    for (int b = 5; b < NF; b += 4) id[(b - 5) / 4] = recip(q[b + 3]);
    const int i = (int)(lin % g.nr), k = (int)(lin / ((size_t)g.nr * g.nth));
    const PCell<T> ce = cell_eq(a.t, g, i, k);
    bool bad = false;
    const T c = pert_cell_rate<T, NF>(a, ce, i, q, recip(ce.rho0 + q[RHO]), id, bad);
    if (positive(c) && !(c <= rate)) rate = c;
    if (bad) status |= STATUS_NONPHYSICAL;
  }
  raise_rate(slot, rate);
  if (status) atomicOr(a.status, status);
}

// Per-block FP64 partial sums of V * E'_f.
template <class T, int NF>
__global__ void pert_sums_kernel(const PertArgs<T> a, double* partials) {
  __shared__ double red[256 / 32];
  const DevGrid& g = a.g;
  const size_t ncell = (size_t)g.nr * g.nth * g.nz;
  double s[NF];
#pragma unroll
  for (int f = 0; f < NF; ++f) s[f] = 0.0;
  for (size_t lin = blockIdx.x * (size_t)256 + threadIdx.x; lin < ncell; lin += (size_t)gridDim.x * 256) {
    const double V = g.vol[lin % g.nr];
#pragma unroll
    for (int f = 0; f < NF; ++f) s[f] += V * (double)a.in[f][lin];
  }
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    const double t = block_sum<256>(s[f], red);
    if (threadIdx.x == 0) partials[(size_t)f * gridDim.x + blockIdx.x] = t;
  }
}

}  // namespace rossbi
