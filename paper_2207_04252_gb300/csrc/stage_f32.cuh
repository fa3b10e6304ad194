// Fused RK2 stage kernel of the FP32 perturbation form.
//
// The physics is that of stage_pert.cuh (its face solver, flux, sources, drag
// and update are called from here); the layout is made for the issue slots,
// which bound this kernel (a face's work is a few hundred FP32 instructions
// against nine loads of its state):
//   - the staged box and the accumulators hold quads, {rho u', rho v', rho w',
//     E'} of the gas and {u, v, w, rho_d} of a dust species, so that a
//     reconstruction reads its nine fields at three cells with nine loads
//     instead of 27, and works on two fields per instruction (the packed f32x2
//     arithmetic of sm_100 and later);
//   - row and plane strides are odd numbers of quads (an odd number times four
//     for single floats), so that the eight lanes of a quarter warp's quads, or
//     four lines of eight lanes, fall into different banks along any axis;
//   - the equilibrium of the tile's faces, the parabola weights and the face
//     areas are copied to shared memory with the box: the sweeps load nothing
//     from global memory and form no 64-bit address;
//   - 24 warps share an SM, which takes 80 registers: the general Riemann solver
//     is out of line, after the sweeps (redo).
// A bi-fluid step of 512 x 1024 x 128 cells (12.1 GB that it cannot do without,
// 1.8 ms of a copy's rate) took 28.9 ms with single-word staging and an FP32
// Newton iteration on every face, and takes 12.8: 166 -> 73 warp instructions
// per cell and stage.  A step of 256 x 512 x 64: 3.6 -> 1.55 ms.
#pragma once
#include "stage_pert.cuh"

namespace rossbi {

// ---------------------------------------------------------------- two fields at a time
// min(|a|, |b|) with the sign of a b, and the MinMod slope, of both halves
__device__ __forceinline__ f32x2 min_xorsign2(f32x2 a, f32x2 b) {
  float a0, a1, b0, b1;
  unpack2(a, a0, a1);
  unpack2(b, b0, b1);
  return pack2(min_xorsign(a0, b0), min_xorsign(a1, b1));
}
__device__ __forceinline__ f32x2 minmod2(f32x2 a, f32x2 b) {
  float a0, a1, b0, b1;
  unpack2(a, a0, a1);
  unpack2(b, b0, b1);
  return pack2(fmaxf(min_xorsign(a0, b0), 0.0f), fmaxf(min_xorsign(a1, b1), 0.0f));
}

// parabola() of two fields.
template <bool UNI>
__device__ __forceinline__ void parabola2(f32x2 em, f32x2 e0, f32x2 ep, const float* w, f32x2& qm, f32x2& qp) {
  const f32x2 dm = sub2(e0, em), dp = sub2(ep, e0);
  if (UNI) {
    const f32x2 c3 = pack2(0.375f, 0.375f), c1 = pack2(0.125f, 0.125f), s = minmod2(dm, dp);
    qm = sub2(e0, min_xorsign2(fma2(c3, dm, mul2(c1, dp)), s));
    qp = add2(e0, min_xorsign2(fma2(c3, dp, mul2(c1, dm)), s));
  } else {
    auto two = [&](int q) { return pack2(w[q], w[q]); };
    const f32x2 s = minmod2(mul2(dm, two(0)), mul2(dp, two(1)));
    qm = sub2(e0, min_xorsign2(fma2(two(2), dm, mul2(two(3), dp)), s));
    qp = add2(e0, min_xorsign2(fma2(two(4), dm, mul2(two(5), dp)), mul2(two(6), s)));
  }
}

// ---------------------------------------------------------------- shared memory
template <int BYTES>
__device__ __forceinline__ void copy_async(void* smem, const void* gmem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(s), "l"(gmem), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Offsets in floats of a block's arrays; quads on 16-byte boundaries.
template <int NF, int TR, int TT, int TZ>
struct F32Smem {
  static constexpr int ND = (NF - 5) / 4, NQ = 1 + ND;  // quads per cell: the gas's, then each dust species'
  static constexpr int BX = TR + 4, BY = TT + 4, BZ = TZ + 4;
  static constexpr int ROW = BX | 1, PLANE = (ROW * BY) | 1, BOX = PLANE * BZ;  // staged box, in cells
  static constexpr int CROW = TR | 1, CPLANE = (CROW * TT) | 1, CORE = CPLANE * TZ;  // accumulators
  __host__ __device__ static constexpr int up4(int n) { return (n + 3) & ~3; }
  __host__ __device__ static constexpr int up_odd4(int n) { return (n + 3) / 4 % 2 ? up4(n) : up4(n) + 4; }
  static constexpr int RROW = up_odd4(BX), RPLANE = up_odd4(RROW * BY);      // staged rho'
  static constexpr int CRROW = up_odd4(TR), CRPLANE = up_odd4(CRROW * TT);  // its accumulator
  static constexpr int ZROW = TR | 1;                                       // z faces, in quads
  __host__ __device__ static constexpr int quad(int q) { return 4 * BOX * q; }             // [BOX] quads
  static constexpr int rho = 4 * BOX * NQ;                             // [RPLANE BZ] rho'
  static constexpr int acc0 = up4(rho + RPLANE * BZ);
  __host__ __device__ static constexpr int acc(int q) { return acc0 + 4 * CORE * q; }      // [CORE] quads
  static constexpr int acc_rho = acc0 + 4 * CORE * NQ;                 // [CRPLANE TZ]
  static constexpr int face0 = up4(acc_rho + CRPLANE * TZ);                    // r faces -1 .. TR + 1 of each z: [TZ][TR + 3]
  static constexpr int face1 = face0 + 4 * (TR + 3) * TZ;              // theta faces: [TZ][TR]
  static constexpr int face2 = face1 + 4 * TR * TZ;                    // z faces -1 .. TZ + 1: [TZ + 3][ZROW]
  static constexpr int wgt = face2 + 4 * ZROW * (TZ + 3);              // [2][TR + 2] quads: weights of cells -1 .. TR
  static constexpr int area = wgt + RCW * (TR + 2);                    // areas: TR + 1 r faces, TR theta, TR z
  static constexpr int total = up4(area + 3 * TR + 1);
  static constexpr size_t bytes = (size_t)total * sizeof(float);
  __host__ __device__ static constexpr int face(int axis) { return axis == 0 ? face0 : (axis == 1 ? face1 : face2); }
};

// The sweeps' work on a tile, whatever the block's shape (so that both shapes share
// one copy of redo(), and with it the bits of its results).
template <int NF, int TR, int TT, int TZ, int RC>
struct F32Lines {
  using M = F32Smem<NF, TR, TT, TZ>;
  int i0, j0, k0;
  bool full;  // the tile lies within the grid
  __device__ __forceinline__ F32Lines(const PertArgs<float>& a, int tile) {
    a.order.origin(tile, TR, TT, TZ, i0, j0, k0);
    full = i0 + TR <= a.g.nr && j0 + TT <= a.g.nth && k0 + TZ <= a.g.nz;
  }

  // One 32-lane chunk of the sweep along axis D: items base .. base + 31 (whole
  // lines of L lanes).  Lane p of a line reconstructs cell p - 1, takes the
  // upper face state of its lower neighbour by a shuffle, solves its lower
  // face and takes the flux of its upper face by a second shuffle.
  // Returns whether the lane's face needs the general solver or a flat
  // reconstruction; its flux then counts as zero until the chunk is taken again
  // with REDO, which solves the faces of the `again` lanes and adds their fluxes.
  template <int D, class P, bool REDO>
  __device__ __forceinline__ bool chunk(const PertArgs<float>& a, float* sm, int base, bool again, unsigned& status,
                                        unsigned& nfallback) const {
    constexpr int TD = D == 0 ? TR : (D == 1 ? TT : TZ), L = pow2ceil(TD + 2);
    constexpr int NA = D == 0 ? TT : TR;
    constexpr int ITEMS = items<D>();
    constexpr int ST = D == 0 ? 1 : (D == 1 ? M::ROW : M::PLANE);
    constexpr unsigned FULL = 0xffffffffu;
    constexpr bool UNI = D != 0;
    static_assert(L <= 32, "line does not fit a warp");
    static_assert(ITEMS % 32 == 0, "whole chunks");
    const DevGrid& g = a.g;
    const int item = base + (threadIdx.x & 31);
    const int line = item / L, c = item % L - 1;
    const int ta = line % NA, tb = line / NA;
    const int x = D == 0 ? c : ta, y = D == 1 ? c : (D == 0 ? ta : tb), z = D == 2 ? c : tb;
    // Every cell -1 .. TD of every line is staged, also beyond the grid's edge,
    // so that only what a lane contributes needs conditions; none in a tile
    // within the grid.
    bool do_face = c >= 0, do_acc = c >= 0 && c < TD;
    if (!full) {
      const bool line_ok = D == 0 ? (j0 + y < g.nth && k0 + z < g.nz)
                                  : (D == 1 ? (i0 + x < g.nr && k0 + z < g.nz) : (i0 + x < g.nr && j0 + y < g.nth));
      const int gd = D == 0 ? i0 + x : (D == 1 ? j0 + y : k0 + z), nd = D == 0 ? g.nr : (D == 1 ? g.nth : g.nz);
      do_face = do_face && line_ok && gd <= nd;
      do_acc = do_acc && line_ok && gd < nd;
      if (!__any_sync(FULL, do_face)) return false;  // a warp of lines beyond the edge
    }
    const int s = (z + 2) * M::PLANE + (y + 2) * M::ROW + (x + 2);
    const int sr = (z + 2) * M::RPLANE + (y + 2) * M::RROW + (x + 2);
    const int fx = D == 0 ? z * (TR + 3) + x + 1 : (D == 1 ? z * TR + x : (z + 1) * M::ZROW + x);
    const int core = z * M::CPLANE + y * M::CROW + x;
    float w[RCW];
    if (!UNI) {
      const float4* q = reinterpret_cast<const float4*>(sm + M::wgt) + (x + 1);
      const float4 q0 = q[0], q1 = q[TR + 2];
      w[0] = q0.x; w[1] = q0.y; w[2] = q0.z; w[3] = q0.w;
      w[4] = q1.x; w[5] = q1.y; w[6] = q1.z;
    }
    const float area = sm[M::area + (D == 0 ? 0 : (D == 1 ? TR + 1 : 2 * TR + 1)) + x];
    // the divergence of dust species q: primitive reconstruction, kinetic flux
    auto dust_flux = [&](int q, float* F) {
      const ulonglong2* e = reinterpret_cast<const ulonglong2*>(sm + M::quad(q)) + s;
      const ulonglong2 em = e[-ST], e0 = e[0], ep = e[ST];
      f32x2 lo[2], up[2];
      parabola2<UNI>(em.x, e0.x, ep.x, w, lo[0], up[0]);
      parabola2<UNI>(em.y, e0.y, ep.y, w, lo[1], up[1]);
      float qm[4], qp[4], WL[4];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        unpack2(lo[h], qm[2 * h], qm[2 * h + 1]);
        unpack2(up[h], qp[2 * h], qp[2 * h + 1]);
      }
#pragma unroll
      for (int f = 0; f < 4; ++f) WL[f] = __shfl_up_sync(FULL, qp[f], 1, L);
      dust_kinetic_flux<D>(area, WL, qm, F);
    };
    // The first species' flux has no branch and nothing in common with the
    // gas's: here its instructions fill the latencies of the gas's
    // reconstruction.
    float Fd[4];
    if constexpr (M::NQ > 1 && !REDO) dust_flux(1, Fd);
    {
      const float4* ft = reinterpret_cast<const float4*>(sm + M::face(D)) + fx;
      constexpr int FS = D == 0 ? 1 : (D == 1 ? 0 : M::ZROW);  // to the upper face (theta: the same)
      const float4 fm = ft[0], fp = ft[FS];
      const PEq<float> Em{fm.x, fm.y, fm.z, fm.w};
      float wm[5], wp[5];  // primitive perturbations: right state of the lower face, left state of the upper face
      {
        float qm[5], qp[5];
        {
          const ulonglong2* e = reinterpret_cast<const ulonglong2*>(sm) + s;
          const ulonglong2 em = e[-ST], e0 = e[0], ep = e[ST];
          constexpr int SR = D == 0 ? 1 : (D == 1 ? M::RROW : M::RPLANE);
          const float* r = sm + M::rho + sr;
          f32x2 lo[2], up[2];
          parabola2<UNI>(em.x, e0.x, ep.x, w, lo[0], up[0]);
          parabola2<UNI>(em.y, e0.y, ep.y, w, lo[1], up[1]);
          parabola<UNI>(r[-SR], r[0], r[SR], w, qm[RHO], qp[RHO]);
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            unpack2(lo[q], qm[2 * q], qm[2 * q + 1]);
            unpack2(up[q], qp[2 * q], qp[2 * q + 1]);
          }
        }
        auto face_states = [&](auto reciprocal) {
          if (RC == RECON_PRIM) {
#pragma unroll
            for (int f = 0; f < 5; ++f) {
              wm[f] = qm[f];
              wp[f] = qp[f];
            }
          } else {
            face_prim(a.gm1, Em.v, qm, reciprocal(Em.rho + qm[RHO]), wm);
            face_prim(a.gm1, fp.y, qp, reciprocal(fp.x + qp[RHO]), wp);
          }
          return positive(min_nan(Em.rho + wm[RHO], fp.x + wp[RHO])) &&
                 positive(min_nan(Em.p + wm[EN], fp.z + wp[EN]));
        };
        if constexpr (!REDO) {
          // states that are not physical (or seem so by a subnormal density): NaN
          // leaves both faces of the cell to redo()
          if (!face_states([](float x) { return recip_normal(x); })) wm[EN] = wp[EN] = __int_as_float(0x7fffffff);
        } else if (!face_states([](float x) { return recip(x); })) {
          // positivity fallback: flat reconstruction of the gas fields
          const float4 e = reinterpret_cast<const float4*>(sm)[s];
          qm[0] = qp[0] = e.x;
          qm[1] = qp[1] = e.y;
          qm[2] = qp[2] = e.z;
          qm[3] = qp[3] = e.w;
          qm[RHO] = qp[RHO] = sm[M::rho + sr];
          face_states([](float x) { return recip(x); });
        }
      }
      float F[5], wl[5];
#pragma unroll
      for (int f = 0; f < 5; ++f) {
        wl[f] = __shfl_up_sync(FULL, wp[f], 1, L);  // upper face state of the lower neighbour
        F[f] = 0.0f;
      }
      bool general = false;
      if (do_face && (!REDO || again))
        general = pert_face<float, D, P, REDO>(
            a, Em, area, wl, wm,
            [&]() {
              const int k = k0 + z;  // in the grid: do_face
              return (size_t)k * (D == 0 ? g.nr + 1 : g.nr) + i0 + x;
            },
            F, status, nfallback);
      constexpr bool WRITE = D == 0 && !REDO;
      add_divergence<WRITE, L>(F, sm + M::acc0, core, do_acc);
      const float Fu = __shfl_down_sync(FULL, F[RHO], 1, L);
      if (do_acc) {
        float* d = sm + M::acc_rho + z * M::CRPLANE + y * M::CRROW + x;
        *d = WRITE ? F[RHO] - Fu : *d + (F[RHO] - Fu);
      }
      if constexpr (M::NQ > 1 && !REDO) {
        add_divergence<D == 0, L>(Fd, sm + M::acc(1), core, do_acc);
#pragma unroll 1
        for (int q = 2; q < M::NQ; ++q) {
          dust_flux(q, Fd);
          add_divergence<D == 0, L>(Fd, sm + M::acc(q), core, do_acc);
        }
      }
      return general;
    }
  }

  // Writes or adds the divergence F - (F of the lane above) of a quad.
  template <bool WRITE, int L>
  __device__ __forceinline__ static void add_divergence(const float* F, float* acc, int core, bool own) {
    float u[4];
#pragma unroll
    for (int f = 0; f < 4; ++f) u[f] = __shfl_down_sync(0xffffffffu, F[f], 1, L);
    if (own) {
      ulonglong2* d = reinterpret_cast<ulonglong2*>(acc) + core;
      ulonglong2 v;
      v.x = sub2(pack2(F[0], F[1]), pack2(u[0], u[1]));
      v.y = sub2(pack2(F[2], F[3]), pack2(u[2], u[3]));
      if (!WRITE) {
        const ulonglong2 o = *d;
        v.x = add2(o.x, v.x);
        v.y = add2(o.y, v.y);
      }
      *d = v;
    }
  }

  template <int D>
  static __host__ __device__ constexpr int items() {
    return (D == 0 ? TT * TZ : (D == 1 ? TR * TZ : TR * TT)) * pow2ceil((D == 0 ? TR : (D == 1 ? TT : TZ)) + 2);
  }
  static constexpr int BITS = 10;  // chunks of a warp and sweep at most
  template <int D, class P>
  __device__ __forceinline__ void resweep(const PertArgs<float>& a, float* sm, unsigned left, unsigned& status,
                                          unsigned& nfallback) const {
    unsigned bit = 1u << (BITS * D);
#pragma unroll 1
    for (int base = threadIdx.x & ~31; base < items<D>(); base += blockDim.x, bit <<= 1)
      if (__any_sync(0xffffffffu, left & bit)) chunk<D, P, true>(a, sm, base, left & bit, status, nfallback);
    __syncthreads();
  }

  // The faces for the general solver (near a strong wave or in the sonic band)
  // and those of cells whose reconstruction is not physical, of all three sweeps,
  // for blocks that have any; sweep by sweep, so that every sum has one order.
  // Out of line and after the sweeps: with no call in their loops the kernel takes
  // 80 registers and 24 warps share an SM; with the solver called from the loops
  // it took 128 (16 warps), and spilled at fewer.  The solver is in line here, as
  // every face takes it: around a call the faces' states go to local memory.  A step
  // of 280 x 180 x 48 bi-fluid cells with jumps of 10 % at all faces, the most that
  // this can cost: 1.51 ms, 1.66 with a call, 1.58 with 16 warps and an FP32 Newton
  // iteration on every face.
  struct Word2 {
    unsigned status, nfallback;
  };
  template <class P>
  static __device__ __noinline__ Word2 redo(const PertArgs<float>& a, float* sm, unsigned left) {
    const F32Lines t(a, blockIdx.x);
    Word2 w{0, 0};
    t.template resweep<0, P>(a, sm, left, w.status, w.nfallback);
    t.template resweep<1, P>(a, sm, left, w.status, w.nfallback);
    t.template resweep<2, P>(a, sm, left, w.status, w.nfallback);
    return w;
  }
};

template <int NF, int TR, int TT, int TZ, int NT, int RC>
struct F32Tile : F32Lines<NF, TR, TT, TZ, RC> {
  using Base = F32Lines<NF, TR, TT, TZ, RC>;
  using M = typename Base::M;
  using Base::i0, Base::j0, Base::k0;
  using Base::Base;

  // The tile and its halo as deviations: the gas as conservative departures (or,
  // with RC = RECON_PRIM, primitive ones), the dust as primitives, converted
  // once here.  Each thread owns one (r, theta) position of the box and walks
  // its z planes (half of them where the block has two threads per position),
  // so that an index costs one addition; the loads of a batch of planes are all
  // in flight before the first is used.  Equilibrium ghosts are zero departures.
  __device__ __forceinline__ void stage(const PertArgs<float>& a, float* sm) const {
    constexpr int COLS = M::BX * M::BY, HALVES = NT >= 2 * COLS ? 2 : 1, NB = NF <= 9 ? 5 : 2;
    static_assert(COLS <= NT && M::BZ % 2 == 0, "a thread per (r, theta) position of the box");
    const DevGrid& g = a.g;
    if (threadIdx.x >= HALVES * COLS) return;
    const int half = HALVES == 2 && threadIdx.x >= COLS ? 1 : 0, pos = (int)threadIdx.x - half * COLS;
    const int x = pos % M::BX - 2, y = pos / M::BX - 2;
    const bool side = x < 0 || x >= TR, end = y < 0 || y >= TT;
    if (side && end) return;  // no sweep reads the box's edges and corners
    int ci = i0 + x, cj = j0 + y;
    const bool in = resolve_axis(g, 0, ci) && resolve_axis(g, 1, cj);
    const int first = side || end ? 2 : 0, last = side || end ? TZ + 2 : M::BZ;
    const int z0 = HALVES == 2 && half ? M::BZ / 2 : 0, z1 = HALVES == 2 && !half ? M::BZ / 2 : M::BZ;
    const size_t plane = (size_t)g.nth * g.nr, row = (size_t)cj * g.nr + ci;
    const int at = (y + 2) * M::ROW + (x + 2);
#pragma unroll 1
    for (int zb = z0; zb < z1; zb += NB) {
      float v[NB][NF], eq[NB][2];
      bool use[NB], inside[NB];
#pragma unroll
      for (int u = 0; u < NB; ++u) {
        const int z = zb + u;
        int ck = k0 + z - 2;
        use[u] = z < z1 && z >= first && z < last;
        inside[u] = use[u] && resolve_axis(g, 2, ck) && in;
        if (inside[u]) {
          const size_t lin = (size_t)ck * plane + row;
#pragma unroll
          for (int f = 0; f < NF; ++f) v[u][f] = a.in[f][lin];
          if (RC == RECON_PRIM) {
            const float* c = a.t.cen + 8 * ((size_t)ck * g.nr + ci);
            eq[u][0] = g.has_eq ? c[0] : 0.0f;
            eq[u][1] = g.has_eq ? c[1] : 0.0f;
          }
        } else {
#pragma unroll
          for (int f = 0; f < NF; ++f) v[u][f] = 0.0f;
        }
      }
#pragma unroll
      for (int u = 0; u < NB; ++u) {
        if (!use[u]) continue;
        const int s = (zb + u) * M::PLANE + at;
        if (RC == RECON_PRIM && inside[u]) {
          float w[5];
          face_prim(a.gm1, eq[u][1], v[u], recip(eq[u][0] + v[u][RHO]), w);
#pragma unroll
          for (int f = 0; f < 4; ++f) v[u][f] = w[f];
        }
        reinterpret_cast<float4*>(sm)[s] = make_float4(v[u][0], v[u][1], v[u][2], v[u][3]);
        sm[M::rho + (zb + u) * M::RPLANE + (y + 2) * M::RROW + (x + 2)] = v[u][RHO];
#pragma unroll
        for (int b = 5; b < NF; b += 4) {
          const float rd = v[u][b + 3], id = has_mass(rd) ? recip_normal(rd) : 0.0f;
          reinterpret_cast<float4*>(sm + M::quad((b - 1) / 4))[s] =
              make_float4(v[u][b] * id, v[u][b + 1] * id, v[u][b + 2] * id, rd);
        }
      }
    }
  }

  // The tables of the tile's faces and cells, indices clamped to the grid, by
  // asynchronous copies (in flight while the box is staged).
  __device__ __forceinline__ void tables(const PertArgs<float>& a, float* sm) const {
    const DevGrid& g = a.g;
    constexpr int N0 = (TR + 3) * TZ, N1 = N0 + TR * TZ, N2 = N1 + TR * (TZ + 3);
    for (int q = threadIdx.x; q < N2; q += NT) {
      const int at = q < N1 ? q : N1 + (q - N1) / TR * M::ZROW + (q - N1) % TR;
      float4* dst = reinterpret_cast<float4*>(sm + M::face0) + at;
      if (!g.has_eq) {
        *dst = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      } else {
        size_t o;
        const float* t;
        if (q < N0) {
          const int f = clampi(i0 - 1 + q % (TR + 3), 0, g.nr), k = clampi(k0 + q / (TR + 3), 0, g.nz - 1);
          t = a.t.face[0];
          o = (size_t)k * (g.nr + 1) + f;
        } else if (q < N1) {
          const int c = q - N0, i = clampi(i0 + c % TR, 0, g.nr - 1), k = clampi(k0 + c / TR, 0, g.nz - 1);
          t = a.t.face[1];
          o = (size_t)k * g.nr + i;
        } else {
          const int c = q - N1, i = clampi(i0 + c % TR, 0, g.nr - 1), f = clampi(k0 - 1 + c / TR, 0, g.nz);
          t = a.t.face[2];
          o = (size_t)f * g.nr + i;
        }
        copy_async<16>(dst, t + 4 * o);
      }
    }
    constexpr int W = RCW / 4 * (TR + 2);  // 16-byte pieces of the weights, then the areas one by one
    for (int q = threadIdx.x; q < W + 3 * TR + 1; q += NT) {
      if (q < W) {
        const int c = i0 - 1 + q / (RCW / 4);  // weights of cells -1 .. nr are tabulated
        copy_async<16>(sm + M::wgt + 4 * (q % (RCW / 4) * (TR + 2) + q / (RCW / 4)), a.t.rcoef + (size_t)((c > g.nr ? g.nr : c) + 1) * RCW + 4 * (q % (RCW / 4)));
      } else {
        const int n = q - W;
        const float* t = n < TR + 1 ? a.t.area_r + clampi(i0 + n, 0, g.nr)
                                    : (n < 2 * TR + 1 ? a.t.area_t + clampi(i0 + n - TR - 1, 0, g.nr - 1)
                                                      : a.t.area_z + clampi(i0 + n - 2 * TR - 1, 0, g.nr - 1));
        copy_async<4>(sm + M::area + n, t);
      }
    }
  }

  // The sweep along axis D, chunks spread over the warps; sets bit BITS D + n of
  // `left` where the lane's face of the warp's n-th chunk is left to redo().
  template <int D, class P>
  __device__ __forceinline__ void sweep(const PertArgs<float>& a, float* sm, unsigned& left) const {
    static_assert((Base::template items<D>() + NT - 1) / NT <= Base::BITS, "a bit per chunk");
    unsigned bit = 1u << (Base::BITS * D), status = 0, nfallback = 0;
#pragma unroll 1
    for (int base = threadIdx.x & ~31; base < Base::template items<D>(); base += NT, bit <<= 1)
      if (this->template chunk<D, P, false>(a, sm, base, false, status, nfallback)) left |= bit;
  }
  // The update of a cell.  THIN: with reciprocals of any density; the others are
  // cheaper and right for normal ones, so a cell below 2^-120 (which no stage takes
  // from there to a subnormal density) goes through an out-of-line copy.
  struct Updated {
    float rate;
    unsigned status;
  };
  template <bool XT>
  static __device__ __noinline__ Updated update_thin(const PertArgs<float>& a, const float* sm, int cidx, float tau) {
    Updated u{0.0f, 0};
    F32Tile(a, blockIdx.x).template update<XT, true>(a, sm, cidx, tau, u.rate, u.status);
    return u;
  }
  template <bool XT, bool THIN = false>
  __device__ __forceinline__ void update(const PertArgs<float>& a, const float* sm, int cidx, float tau, float& rate,
                                         unsigned& status) const {
    const int x = cidx % TR, y = (cidx / TR) % TT, z = cidx / (TR * TT);
    const int gi = i0 + x, gj = j0 + y, gk = k0 + z;
    if (gi >= a.g.nr || gj >= a.g.nth || gk >= a.g.nz) return;
    const int s = (z + 2) * M::PLANE + (y + 2) * M::ROW + (x + 2), core = z * M::CPLANE + y * M::CROW + x;
    const PCell<float> ce = cell_eq(a.t, a.g, gi, gk);
    float e[5], dust[NF > 5 ? M::ND : 1][4], G[NF];
    e[RHO] = sm[M::rho + (z + 2) * M::RPLANE + (y + 2) * M::RROW + (x + 2)];
    if constexpr (!THIN) {
      if (!(ce.rho0 + e[RHO] >= 0x1p-120f)) {
        const Updated u = update_thin<XT>(a, sm, cidx, tau);
        rate = fmaxf(rate, u.rate);
        status |= u.status;
        return;
      }
    }
    auto quad = [&](int at, float* q) {
      const float4 v = reinterpret_cast<const float4*>(sm)[at];
      q[0] = v.x;
      q[1] = v.y;
      q[2] = v.z;
      q[3] = v.w;
    };
    quad(s, e);
    quad(M::acc(0) / 4 + core, G);
    G[RHO] = sm[M::acc_rho + z * M::CRPLANE + y * M::CRROW + x];
#pragma unroll
    for (int q = 1; q < M::NQ; ++q) {
      quad(M::quad(q) / 4 + s, dust[q - 1]);
      quad(M::acc(q) / 4 + core, G + 1 + 4 * q);
    }
    pert_update<float, NF, RC, XT>(a, ce, gi, gj, gk, e, dust, G, tau, rate, status,
                                   [](float x) { return THIN ? recip(x) : recip_normal(x); });
  }
};

// One RK stage of one tile per block.
template <int NF, int TR, int TT, int TZ, int NT, int MINB, class P, bool XT, int RC>
__global__ void __launch_bounds__(NT, MINB) stage_f32_kernel(const __grid_constant__ PertArgs<float> a) {
  extern __shared__ __align__(16) float sm[];
  using Tile = F32Tile<NF, TR, TT, TZ, NT, RC>;
  const Tile t(a, blockIdx.x);
  unsigned status = 0, left = 0;
  __shared__ double s_tau;
  publish_tau(&s_tau, a.tau_frac, a.dt_host, a.rate_in, a.g.cfl);
  if (!a.stage2) clear_rate(a.rate_out);
  t.tables(a, sm);
  t.stage(a, sm);
  copy_async_wait();
  __syncthreads();
  t.template sweep<0, P>(a, sm, left);
  __syncthreads();
  t.template sweep<1, P>(a, sm, left);
  __syncthreads();
  t.template sweep<2, P>(a, sm, left);
  if (__syncthreads_or(left)) {
    const typename Tile::Word2 w = Tile::template redo<P>(a, sm, left);
    status = w.status;
    if (w.nfallback) atomicAdd(a.t.fallbacks, (unsigned long long)w.nfallback);
  }
  float rate = 0.0f;
  for (int cidx = threadIdx.x; cidx < TR * TT * TZ; cidx += NT)
    t.template update<XT>(a, sm, cidx, (float)s_tau, rate, status);
  if (a.stage2) raise_rate(a.rate_out, rate);
  if (status) atomicOr(a.status, status);
}

}  // namespace rossbi
