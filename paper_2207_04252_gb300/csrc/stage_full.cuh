// Fused RK2 stage kernel of the FP64 (full conservative state) form.
//
// One CTA owns a TR x TT x TZ tile of cells.  It stages the tile and a 2-deep
// halo along each axis into shared memory as deviations from the equilibrium
// (Sect. 2.7: the conservative departures E' = E - E0 of the gas, or with
// RC = RECON_PRIM the primitive departures u', v', w', P', rho'), then
// sweeps the three directions.  In a sweep, lines along the
// direction map onto groups of L = pow2(T + 2) lanes: lane p reconstructs cell
// p - 1 (parabola + MinMod), receives the upper face state of its lower
// neighbour by a shuffle, solves the exact Riemann problem on its lower face
// (Sect. 2.6) and the dust flux, and receives the flux of its upper face by a
// second shuffle, so each face is solved once per tile.  The flux divergence
// is accumulated in shared memory; the epilogue adds the sources (App. B),
// subtracts the balanced residual R0 (Sect. 2.8), applies the RK stage update
// (Sect. 2.5) and the semi-implicit drag (Sect. 2.9), and in stage 2 fuses the
// CFL rate of the new state.
//
// The FP64 pipe (two lanes per SM and clock) bounds it, at 84 % busy in the main
// tile, not memory (2 % of a copy's bandwidth).  So what needs no 64-bit rounding
// runs on the bits or in float (narrow.cuh), the Riemann solution near p_K is a
// series (riemann_near.cuh), the parabola is two weights per side on
// differences, divisions are one reciprocal per density, and the tile is the
// one with the fewest idle lanes that leaves two blocks to an SM (14 x 6 x 6:
// 1.27 lanes per cell; 14 x 14 x 6 has 1.21, but at one block of 12 warps per SM
// took 4.69 ms where this takes 4.53).  One step:
//   gas and dust, 128 x 256 x 32: 14.4 -> 4.53 ms;
//   gas disc, 128 x 256 x 32, with the next step's dt and the sums: 10.8 -> 3.03 ms;
//   cylindrical explosion, 1600 x 3200: 29.4 -> 8.35 ms.
#pragma once
#include "device_common.cuh"

namespace rossbi {

struct StageArgs {
  DevGrid g;
  int tile;                    // TILE_*, chosen by the host
  const double* in[NF_MAX];    // stage input (stencil) state
  const double* base[NF_MAX];  // E^n, base of the update
  double* out[NF_MAX];         // updated state
  double* gout;            // mode 1: G(E) - R0 written here, [nf][ncell]
  double dt_host;
  const unsigned long long* rate_in;  // if set, dt = N_CFL / (the rate in this device slot)
  unsigned long long* rate_out;       // the largest CFL rate of the output: cleared by stage 1, raised by stage 2
  double tau_frac;                    // 0.5 (stage 1) or 1.0 (stage 2)
  DragArgs drag;
  int stage2;                         // fuse the CFL rate of the output
  unsigned* status;
  int mode;                          // 0 update, 1 residual only (empty run)
  TileOrder order;
};

// Parabola through three deviations (Sect. 2.7) with the MinMod limiter: each
// face deviation is limited to minmod(deviation, s h), s the minmod slope and
// h the limiter reach of that side.  With the differences dm = e0 - em and
// dp = ep - e0 the parabola's face deviations are -(am dm + ap dp) and bm dm +
// bp dp with positive weights (of the geometry alone, tabulated), so that
// where dm and dp have one sign they have it too, and the limiter is a
// minimum of magnitudes: w = {lm, lp, am, ap, bm, bp, h+/h-}, the lower
// limit min(lm dm, lp dp) being h- times the slope.  UNI: a uniform axis, where
// in units of the spacing am = bp = 3/8, ap = bm = 1/8 and all limits 1.
// 6 (uniform) or 11 FP64 operations; forming the slopes, the curvature and the
// limiter's products took 17 and four compares.
template <bool UNI>
__device__ __forceinline__ void parabola(double em, double e0, double ep, const double* w, double& qm, double& qp) {
  const double dm = e0 - em, dp = ep - e0;
  if (UNI) {
    const double s = minmod_bits(dm, dp);
    qm = e0 - min_mag(fma(0.375, dm, scale_down<3>(dp)), s);
    qp = e0 + min_mag(fma(0.375, dp, scale_down<3>(dm)), s);
  } else {
    const double s = minmod_bits(dm * w[0], dp * w[1]);
    qm = e0 - min_mag(fma(w[2], dm, w[3] * dp), s);
    qp = e0 + min_mag(fma(w[4], dm, w[5] * dp), w[6] * s);
  }
}
template <bool UNI>
__device__ __forceinline__ void parabola(float em, float e0, float ep, const float* w, float& qm, float& qp) {
  const float dm = e0 - em, dp = ep - e0;
  if (UNI) {
    const float s = fmaxf(min_xorsign(dm, dp), 0.0f), u = 0.125f * (dm + dp);
    qm = e0 - min_xorsign(fmaf(0.25f, dm, u), s);
    qp = e0 + min_xorsign(fmaf(0.25f, dp, u), s);
  } else {
    const float s = fmaxf(min_xorsign(dm * w[0], dp * w[1]), 0.0f);
    qm = e0 - min_xorsign(fmaf(w[2], dm, w[3] * dp), s);
    qp = e0 + min_xorsign(fmaf(w[4], dm, w[5] * dp), w[6] * s);
  }
}

// The branches of a double-precision parabola, for its adjoint: bit 0 the
// slopes have one sign (the face values move with the neighbours), bit 1 the
// lower slope is the smaller, bits 2, 3 the parabola's own lower / upper face
// value is inside the limiter.
template <bool UNI>
__device__ __forceinline__ unsigned parabola_branches(double em, double e0, double ep, const double* w, double& qm,
                                                      double& qp) {
  const double dm = e0 - em, dp = ep - e0;
  double sm = dm, sp = dp, A, B, lo, up;
  if (UNI) {
    A = fma(0.375, dm, scale_down<3>(dp));
    B = fma(0.375, dp, scale_down<3>(dm));
  } else {
    sm = dm * w[0];
    sp = dp * w[1];
    A = fma(w[2], dm, w[3] * dp);
    B = fma(w[4], dm, w[5] * dp);
  }
  const double s = minmod_bits(sm, sp);
  lo = s;
  up = UNI ? s : w[6] * s;
  const bool a = mag_less(A, lo), b = mag_less(B, up);
  qm = e0 - (a ? A : lo);
  qp = e0 + (b ? B : up);
  return (((unsigned long long)__double_as_longlong(s) << 1) != 0 ? 1u : 0u) | (mag_less(sm, sp) ? 2u : 0u) |
         (a ? 4u : 0u) | (b ? 8u : 0u);
}

// parabola_branches on slopes: s the minmod slope, the parabola's face deviation
// against s times the limiter's reach.  v = {1/(x0-xm), 1/(xp-x0), 1/(xp-xm),
// x0-xm, xp-x0, fm-x0, fp-x0, -h-, h+}.  For the adjoint of the primitive option
// only (the forward takes parabola(), equal to rounding), see cell_prim_rounded:
// neither its branches nor the rounding of its face values may depend on how the
// forward's weights are arranged for speed.  (Beside an equilibrium
// ghost the limited velocity of a wall's face is e0 - e0, whose rounding decides
// which side of the contact the face takes.)
__device__ __forceinline__ double slope_minmod(double a, double b) {
  if (a * b <= 0.0) return 0.0;
  return fabs(a) < fabs(b) ? a : b;
}
__device__ __forceinline__ unsigned slope_branches(double em, double e0, double ep, const double* v, double& qm,
                                                   double& qp) {
  const double sm = (e0 - em) * v[0];
  const double sp = (ep - e0) * v[1];
  const double s = slope_minmod(sm, sp);
  const double a = (sp - sm) * v[2];
  const double b = (sp * v[3] + sm * v[4]) * v[2];
  const double A = v[5] * (a * v[5] + b), B = s * v[7];
  const double C = v[6] * (a * v[6] + b), D = s * v[8];
  qm = e0 + slope_minmod(A, B);
  qp = e0 + slope_minmod(C, D);
  return (sm * sp > 0.0 ? 1u : 0u) | (fabs(sm) < fabs(sp) ? 2u : 0u) | (fabs(A) < fabs(B) ? 4u : 0u) |
         (fabs(C) < fabs(D) ? 8u : 0u);
}
template <int D>
__device__ __forceinline__ void slope_weights(const DevGrid& g, int gi, double* v) {
  if (D == 0) {
    const int c = gi < -1 ? -1 : (gi > g.nr ? g.nr : gi);
#pragma unroll
    for (int q = 0; q < 9; ++q) v[q] = g.rslope[(c + 1) * 9 + q];
  } else {
    const double h = g.dx[D];
    v[0] = v[1] = 1.0 / h;
    v[2] = 0.5 / h;
    v[3] = v[4] = h;
    v[5] = -0.5 * h;
    v[6] = 0.5 * h;
    v[7] = -h;
    v[8] = h;
  }
}

// Parabola weights of a cell of axis 0 (the uniform axes 1, 2 need none).
template <class T, int D>
__device__ __forceinline__ void parabola_weights(const T* rcoef, int gi, int nr, T* w) {
  if (D == 0) {
    const int c = gi < -1 ? -1 : (gi > nr ? nr : gi);
    const T* cw = rcoef + (c + 1) * RCW;
#pragma unroll
    for (int q = 0; q < RCW; ++q) w[q] = cw[q];
  }
}

// Dust reconstruction of the cell at s (stride S along the sweep) from the
// staged primitives (u, v, w, rho_d) in the fields b .. b + 3.
template <class T, int BOX, int S, bool UNI>
__device__ __forceinline__ void dust_recon(const T* sE, int sidx, int b, const T* w, T* wm, T* wp) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const T* r = sE + (b + q) * BOX + sidx;
    parabola<UNI>(r[-S], r[0], r[S], w, wm[q], wp[q]);
  }
}

// Ghost rule of Sect. 2.4 for a cell index of one axis, possibly outside the
// domain.  Returns false for an equilibrium ghost (E' = 0).
__device__ __forceinline__ bool resolve_axis(const DevGrid& g, int ax, int& c) {
  const int n = ax == 0 ? g.nr : (ax == 1 ? g.nth : g.nz);
  if (c >= 0 && c < n) return true;
  const int bc = c < 0 ? g.bc_lo[ax] : g.bc_hi[ax];
  if (bc == BC_EQUILIBRIUM) return false;
  if (bc == BC_PERIODIC) {
    c %= n;
    if (c < 0) c += n;
  } else {
    c = c < 0 ? 0 : n - 1;
  }
  return true;
}
__device__ __forceinline__ bool resolve_cell(const DevGrid& g, int c[3]) {
  return resolve_axis(g, 0, c[0]) && resolve_axis(g, 1, c[1]) && resolve_axis(g, 2, c[2]);
}

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

// One lane of a sweep along axis D of a TR x TT x TZ tile: its cell, and
// what of it is inside the grid.
template <int TR, int TT, int TZ, int D>
struct SweepLane {
  static constexpr int ZH = TZ == 1 ? 0 : 2;  // z halo (none in the flat one-z-cell tile)
  static constexpr int BX = TR + 4, BY = TT + 4, BZ = TZ + 2 * ZH, BOX = BX * BY * BZ, NCORE = TR * TT * TZ;
  static constexpr int TD = D == 0 ? TR : (D == 1 ? TT : TZ);
  static constexpr int L = pow2ceil(TD + 2);
  static constexpr int NA = D == 0 ? TT : TR;
  static constexpr int NB = D == 2 ? TT : TZ;
  static constexpr int ITEMS = NA * NB * L;
  static constexpr int STRIDE = D == 0 ? 1 : (D == 1 ? BX : BX * BY);
  static_assert(L <= 32, "line does not fit a warp");
  int gi, gk, gd, sidx, core;
  bool do_recon, do_face, do_acc;
  __device__ __forceinline__ SweepLane(const DevGrid& g, int item, int i0, int j0, int k0) {
    const bool valid = item < ITEMS;
    const int line = valid ? item / L : 0;
    const int c = item % L - 1;
    const int ta = line % NA, tb = line / NA;
    const int x = D == 0 ? c : ta;
    const int y = D == 1 ? c : (D == 0 ? ta : tb);
    const int z = D == 2 ? c : tb;
    gi = i0 + x;
    gk = k0 + z;
    const int gj = j0 + y;
    const bool line_ok = valid && (D == 0 ? (gj < g.nth && gk < g.nz)
                                          : (D == 1 ? (gi < g.nr && gk < g.nz) : (gi < g.nr && gj < g.nth)));
    gd = D == 0 ? gi : (D == 1 ? gj : gk);
    const int nd = D == 0 ? g.nr : (D == 1 ? g.nth : g.nz);
    do_recon = line_ok && c <= TD && gd <= nd;
    do_face = do_recon && c >= 0;
    do_acc = line_ok && c >= 0 && c < TD && gd < nd;
    sidx = do_recon ? ((z + ZH) * BY + (y + 2)) * BX + (x + 2) : (ZH * BY + 2) * BX + 2;
    core = (z * TT + y) * TR + x;
  }
};

template <int D>
__device__ __forceinline__ double face_area(const DevGrid& g, int gi, int ci) {
  return D == 0 ? g.area_r[clampi(gi, 0, g.nr)] : (D == 1 ? g.area_t[ci] : g.area_z[ci]);
}

// Writes (D = 0) or adds the flux divergence F - (F of the lane above) of the
// lane's cell to the field's accumulator.
template <int D, int L>
__device__ __forceinline__ void accumulate(double F, double* dst, bool own) {
  const double Fu = __shfl_down_sync(0xffffffffu, F, 1, L);
  if (own) {
    if (D == 0) *dst = F - Fu;
    else *dst += F - Fu;
  }
}

// The gas sweep along axis D: sE holds the five staged gas departures.
template <int TR, int TT, int TZ, int NT, int D, int RC>
__device__ __forceinline__ void sweep_gas(const StageArgs& a, const double* sE, double* sG, int i0, int j0, int k0,
                                          unsigned& status) {
  using S = SweepLane<TR, TT, TZ, D>;
  constexpr int BOX = S::BOX, STRIDE = S::STRIDE, L = S::L;
  constexpr unsigned FULL = 0xffffffffu;
  constexpr bool UNI = D != 0;
  const DevGrid& g = a.g;
  const double gam = g.gamma;
  for (int base = threadIdx.x & ~31; base < S::ITEMS; base += NT) {
    const S s(g, base + (threadIdx.x & 31), i0, j0, k0);
    if (!__any_sync(FULL, s.do_face)) continue;  // a warp of lines beyond a ragged grid's edge
    double w[RCW];
    parabola_weights<double, D>(g.rcoef, s.gi, g.nr, w);
    // equilibrium gas state (conservative, or primitive with RC = RECON_PRIM)
    // on the lower face of this cell (index along D = gd) and on its upper
    // face; table indices clamped.  Its radial and vertical velocities are zero.
    const int ci = clampi(s.gi, 0, g.nr - 1), ck = clampi(s.gk, 0, g.nz - 1);
    auto eq_face = [&](int f, int fd) -> double {
      const double* tc = RC == RECON_PRIM ? g.w0c : g.e0c;
      const double* tr = RC == RECON_PRIM ? g.w0r : g.e0r;
      const double* tz = RC == RECON_PRIM ? g.w0z : g.e0z;
      if (D == 0) return tr[((size_t)f * g.nz + ck) * (g.nr + 1) + clampi(fd, 0, g.nr)];
      if (D == 1) return tc[((size_t)f * g.nz + ck) * g.nr + ci];
      return tz[((size_t)f * (g.nz + 1) + clampi(fd, 0, g.nz)) * g.nr + ci];
    };
    double WR[5], WP[5];  // primitives: right state of the lower face, left state of the upper face
    {
      double qm[5], qp[5];
#pragma unroll
      for (int f = 0; f < 5; ++f) {
        const double* e = sE + f * BOX + s.sidx;
        parabola<UNI>(e[-STRIDE], e[0], e[STRIDE], w, qm[f], qp[f]);
      }
      // face states E0 + q on both faces of this cell (Sect. 2.7); flat
      // departures if either is not physical
      auto face_states = [&]() {
        if (g.has_eq) {
#pragma unroll
          for (int f : {MV, EN, RHO}) {
            qm[f] += eq_face(f, s.gd);
            qp[f] += eq_face(f, s.gd + 1);
          }
        }
        if (RC == RECON_PRIM) {
#pragma unroll
          for (int f = 0; f < 5; ++f) {
            WR[f] = qm[f];
            WP[f] = qp[f];
          }
        } else {
          gas_prim(gam, qm, WR);
          gas_prim(gam, qp, WP);
        }
        return positive(qm[RHO]) && positive(qp[RHO]) && positive(WR[EN]) && positive(WP[EN]);
      };
      if (!face_states() && s.do_recon) {
#pragma unroll
        for (int f = 0; f < 5; ++f) qm[f] = qp[f] = sE[f * BOX + s.sidx];
        face_states();
      }
    }
    double F[5], WL[5];
#pragma unroll
    for (int f = 0; f < 5; ++f) WL[f] = __shfl_up_sync(FULL, WP[f], 1, L);
    if (s.do_face) {
      gas_face_flux<D>(g.near, face_area<D>(g, s.gi, ci), WL, WR, F, status);
    } else {
#pragma unroll
      for (int f = 0; f < 5; ++f) F[f] = 0.0;
    }
#pragma unroll
    for (int f = 0; f < 5; ++f) accumulate<D, L>(F[f], sG + f * S::NCORE + s.core, s.do_acc);
  }
}

// The sweep of one dust species along axis D: sE holds its staged primitives
// (u, v, w, rho_d), sG its accumulators.
template <int TR, int TT, int TZ, int NT, int D>
__device__ __forceinline__ void sweep_dust(const DevGrid& g, const double* sE, double* sG, int i0, int j0, int k0) {
  using S = SweepLane<TR, TT, TZ, D>;
  constexpr int L = S::L;
  constexpr unsigned FULL = 0xffffffffu;
  for (int base = threadIdx.x & ~31; base < S::ITEMS; base += NT) {
    const S s(g, base + (threadIdx.x & 31), i0, j0, k0);
    if (!__any_sync(FULL, s.do_face)) continue;
    double w[RCW], qm[4], qp[4], F[4], WL[4];
    parabola_weights<double, D>(g.rcoef, s.gi, g.nr, w);
    dust_recon<double, S::BOX, S::STRIDE, D != 0>(sE, s.sidx, 0, w, qm, qp);
#pragma unroll
    for (int f = 0; f < 4; ++f) WL[f] = __shfl_up_sync(FULL, qp[f], 1, L);
    if (s.do_face) {
      dust_kinetic_flux<D>(face_area<D>(g, s.gi, clampi(s.gi, 0, g.nr - 1)), WL, qm, F);
    } else {
#pragma unroll
      for (int f = 0; f < 4; ++f) F[f] = 0.0;
    }
#pragma unroll
    for (int f = 0; f < 4; ++f) accumulate<D, L>(F[f], sG + f * S::NCORE + s.core, s.do_acc);
  }
}

// Every dust species of a tile through the gas's staging buffer sE, as
// primitives (u, v, w, rho_d) converted once per staged cell, into its
// accumulators in sG; `stage` walks the box (put(idx, cell or null)).  One
// species at a time keeps a nine-field block at 108 KB, two blocks to an SM,
// whose barriers and staging overlap (all fields staged at once: 166 KB, one
// block of six warps, FP64 pipe 75 % busy), and lets every species count have
// the 14 x 6 x 6 tile.
template <int NF, int TR, int TT, int TZ, int NT, class Stage>
__device__ __forceinline__ void dust_species(const DevGrid& g, const double* const* in, double* sE, double* sG,
                                             Stage& stage, int i0, int j0, int k0) {
  constexpr int BOX = SweepLane<TR, TT, TZ, 0>::BOX, NCORE = TR * TT * TZ;
#pragma unroll 1
  for (int b = 5; b < NF; b += 4) {
    stage([&](int idx, const int* c) {
      if (!c) {
#pragma unroll
        for (int f = 0; f < 4; ++f) sE[f * BOX + idx] = 0.0;
        return;
      }
      const size_t lin = ((size_t)c[2] * g.nth + c[1]) * g.nr + c[0];
      const double rd = in[b + 3][lin], id = has_mass(rd) ? recip(rd) : 0.0;
#pragma unroll
      for (int q = 0; q < 3; ++q) sE[q * BOX + idx] = in[b + q][lin] * id;
      sE[3 * BOX + idx] = rd;
    });
    __syncthreads();
    double* sD = sG + b * NCORE;
    sweep_dust<TR, TT, TZ, NT, 0>(g, sE, sD, i0, j0, k0);
    __syncthreads();
    sweep_dust<TR, TT, TZ, NT, 1>(g, sE, sD, i0, j0, k0);
    __syncthreads();
    if constexpr (TZ > 1) {
      sweep_dust<TR, TT, TZ, NT, 2>(g, sE, sD, i0, j0, k0);
      __syncthreads();
    }
  }
}

// Walks the staged box of a tile: put(idx, cell or null) for every cell that
// a sweep reads (tile and halo without edges and corners), null for an
// equilibrium ghost.
template <int TR, int TT, int TZ, int NT, class F>
__device__ __forceinline__ void walk_box(const DevGrid& g, int i0, int j0, int k0, F&& put) {
  constexpr int ZH = TZ == 1 ? 0 : 2, BX = TR + 4, BY = TT + 4, BOX = BX * BY * (TZ + 2 * ZH);
  for (int idx = threadIdx.x; idx < BOX; idx += NT) {
    const int x = idx % BX - 2, y = (idx / BX) % BY - 2, z = idx / (BX * BY) - ZH;
    const int outside = (x < 0 || x >= TR) + (y < 0 || y >= TT) + (z < 0 || z >= TZ);
    if (outside > 1) continue;
    int c[3] = {i0 + x, j0 + y, k0 + z};
    put(idx, resolve_cell(g, c) ? c : nullptr);
  }
}

// Fixed-order block sum (deterministic for a fixed launch shape).
template <int NT>
__device__ __forceinline__ double block_sum(double v, double* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) red[warp] = v;
  __syncthreads();
  double s = 0.0;
  for (int q = 0; q < NT / 32; ++q) s += red[q];
  __syncthreads();
  return s;
}

// The stage's length tau, formed by one thread (an FP64 division is worth
// eight operations of the two-lane pipe) for all to read after a barrier.
__device__ __forceinline__ void publish_tau(double* tau, double frac, double dt_host, const unsigned long long* rate_in,
                                            double cfl) {
  if (threadIdx.x == 0) *tau = frac * (rate_in ? cfl / __longlong_as_double((long long)*rate_in) : dt_host);
}
// Stage 1 clears the slot that stage 2 of the step raises (in slabs: the first
// launch does; the host passes no slot to the others of stage 1).
__device__ __forceinline__ void clear_rate(unsigned long long* rate_out) {
  if (rate_out && blockIdx.x == 0 && threadIdx.x == 0) *rate_out = 0;
}
// Raises the slot to the warp's largest rate (non-negative values order like
// their bits: exact and independent of the order).  The CFL step is N_CFL over
// the maximum, so that no block divides and no launch reduces partials.
__device__ __forceinline__ void raise_rate(unsigned long long* rate_out, float rate) {
  const float m = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(rate)));
  if ((threadIdx.x & 31) == 0 && positive(m))
    atomicMax(rate_out, (unsigned long long)__double_as_longlong((double)m));
}
__device__ __forceinline__ void raise_rate(unsigned long long* rate_out, double rate) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double other = __shfl_xor_sync(0xffffffffu, rate, o);
    if (mag_less(rate, other)) rate = other;
  }
  if ((threadIdx.x & 31) == 0 && positive(rate)) atomicMax(rate_out, (unsigned long long)__double_as_longlong(rate));
}

// XT: the optional terms (indirect gravity, wave-killing zones) are compiled
// in; the plain instantiation carries none of their code.
// TZ = 1 is the flat tile of a grid one z cell thick whose z boundaries are
// periodic or outflow: both z ghosts of the cell are the cell itself, its two
// z faces carry the same flux, and the z sweep, whose divergence is exactly
// zero, is skipped (as is the z halo).
template <int NF, int TR, int TT, int TZ, int NT, int MINB, bool XT, int RC>
__global__ void __launch_bounds__(NT, MINB) stage_full_kernel(const StageArgs a) {
  constexpr int ZH = TZ == 1 ? 0 : 2;
  constexpr int BX = TR + 4, BY = TT + 4, BZ = TZ + 2 * ZH, BOX = BX * BY * BZ, NCORE = TR * TT * TZ;
  extern __shared__ double smem[];
  double* sE = smem;             // [5][BOX] the gas departures, then the four primitives of one dust species at a time
  double* sG = smem + 5 * BOX;   // [NF][NCORE] flux divergence
  const DevGrid& g = a.g;
  int i0, j0, k0;
  a.order.origin(blockIdx.x, TR, TT, TZ, i0, j0, k0);
  unsigned status = 0;
  __shared__ double s_tau;
  publish_tau(&s_tau, a.tau_frac, a.dt_host, a.rate_in, g.cfl);
  if (!a.stage2) clear_rate(a.rate_out);

  auto stage = [&](auto&& put) { walk_box<TR, TT, TZ, NT>(g, i0, j0, k0, put); };
  // the gas as deviations E' = E - E0 (or, with RC = RECON_PRIM, the primitive
  // departures u', v', w', P', rho') in slots 0..4
  stage([&](int idx, const int* c) {
    if (!c) {
#pragma unroll
      for (int f = 0; f < 5; ++f) sE[f * BOX + idx] = 0.0;
      return;
    }
    const size_t lin = ((size_t)c[2] * g.nth + c[1]) * g.nr + c[0];
    const size_t e0o = (size_t)c[2] * g.nr + c[0], e0s = (size_t)g.nz * g.nr;
    double U[5], W[5];
#pragma unroll
    for (int f = 0; f < 5; ++f) U[f] = a.in[f][lin];
    if (RC == RECON_PRIM) cell_prim_rounded(g.gamma, U, W);
    const double* e0 = RC == RECON_PRIM ? g.w0c : g.e0c;
#pragma unroll
    for (int f = 0; f < 5; ++f) {
      double v = RC == RECON_PRIM ? W[f] : U[f];
      if (g.has_eq && f != MU && f != MW) v -= e0[f * e0s + e0o];
      sE[f * BOX + idx] = v;
    }
  });
  __syncthreads();
  sweep_gas<TR, TT, TZ, NT, 0, RC>(a, sE, sG, i0, j0, k0, status);
  __syncthreads();
  sweep_gas<TR, TT, TZ, NT, 1, RC>(a, sE, sG, i0, j0, k0, status);
  __syncthreads();
  if constexpr (TZ > 1) {
    sweep_gas<TR, TT, TZ, NT, 2, RC>(a, sE, sG, i0, j0, k0, status);
    __syncthreads();
  }
  dust_species<NF, TR, TT, TZ, NT>(g, a.in, sE, sG, stage, i0, j0, k0);

  const double tau = s_tau;
  const size_t ncell = (size_t)g.nr * g.nth * g.nz;
  constexpr int ND = NF > 5 ? (NF - 5) / 4 : 1;
  double rate = 0.0;
  for (int cidx = threadIdx.x; cidx < NCORE; cidx += NT) {
    const int x = cidx % TR, y = (cidx / TR) % TT, z = cidx / (TR * TT);
    const int gi = i0 + x, gj = j0 + y, gk = k0 + z;
    if (gi >= g.nr || gj >= g.nth || gk >= g.nz) continue;
    const size_t lin = ((size_t)gk * g.nth + gj) * g.nr + gi;
    double U[NF], G[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      U[f] = a.in[f][lin];
      G[f] = sG[f * NCORE + cidx];
    }
    {
      double W[5], Vd[ND];
      gas_prim(g.gamma, U, W);
      bool bad = !positive(U[RHO]) || !positive(W[EN]);
#pragma unroll
      for (int b = 5; b < NF; b += 4) {
        bad |= !non_negative(U[b + 3]);
        Vd[(b - 5) / 4] = has_mass(U[b + 3]) ? U[b + 1] * recip(U[b + 3]) : 0.0;
      }
      if (bad) status |= STATUS_NONPHYSICAL;
      if (g.geom == GEOM_CYL) add_sources<XT, NF>(g, gi, gj, gk, U, W, Vd, G);
    }
    if (g.r0) {
#pragma unroll
      for (int f = 0; f < 5; ++f) G[f] -= g.r0[((size_t)f * g.nz + gk) * g.nr + gi];
    }
    if (XT && g.damp_k) {  // wave-killing zones: the gas departures relax towards E0
      const double kd = g.damp_k[(size_t)gk * g.nr + gi];
      if (positive(kd)) {
        const double V = g.vol[gi];
#pragma unroll
        for (int f = 0; f < 5; ++f) G[f] -= V * kd * (U[f] - g.e0c[((size_t)f * g.nz + gk) * g.nr + gi]);
      }
    }
    if (a.mode == 1) {
#pragma unroll
      for (int f = 0; f < NF; ++f) a.gout[f * ncell + lin] = G[f];
      continue;
    }
    const double tv = tau * g.ivol[gi];
    double E[NF], ig = 0.0, id[ND];
#pragma unroll
    for (int f = 0; f < NF; ++f) E[f] = fma(tv, G[f], a.base[f][lin]);
    if (NF > 5 || a.stage2) ig = recip(E[RHO]);
#pragma unroll
    for (int b = 5; b < NF; b += 4) {
      E[b + 3] = dust_density(E[b + 3]);
      id[(b - 5) / 4] = recip(E[b + 3]);
    }
    if constexpr (NF > 5) apply_drag<XT, ND>(g, gi, E, tau, a.drag, ig, id);
#pragma unroll
    for (int f = 0; f < NF; ++f) a.out[f][lin] = E[f];
    if (a.stage2) {
      bool bad = false;
      const double c = cell_rate<NF>(g, gi, E, ig, id, bad);
      if (bad) status |= STATUS_NONPHYSICAL;
      if (positive(c) && mag_less(rate, c)) rate = c;
    }
  }
  if (a.mode == 0 && a.stage2) raise_rate(a.rate_out, rate);
  if (status) atomicOr(a.status, status);
}

}  // namespace rossbi
