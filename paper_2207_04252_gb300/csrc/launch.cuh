// Kernel launchers of the stage and adjoint-flux kernels, one translation
// unit per kernel family (compiled in parallel), called by the host runtime.
// Each dispatches on the field count, the optional-term switch and the gas
// reconstruction mode to one instantiation of its kernel template.
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

#include "adjoint.cuh"
#include "stage_pert.cuh"

namespace rossbi {

// Tiles of the float stage kernel: 14 x 6 x 6 cells, lines of 16 / 8 / 8 lanes.
constexpr int P32_TR = 14, P32_TT = 6, P32_TZ = 6, P32_NT = 384, P32_MINB = 2, P32_WIDE_NT = 768;

// Tiles of the double stage kernels (both forms), with threads per block and
// blocks per SM.  TILE_MAIN wastes the fewest lanes on halos (1.27 of the
// cells); the thinner ones spread a small grid over the SMs; the flat ones,
// without a z halo or z sweep, are for full-state grids one z cell thick whose z
// boundaries are periodic or outflow (the cell's two z faces then carry the same
// flux): the cylindrical explosion of Sect. 4.1.
template <int R, int T, int Z, int N, int B>
struct Tile {
  static constexpr int TR = R, TT = T, TZ = Z, NT = N, MINB = B;
};
using TileMain = Tile<14, 6, 6, 192, 2>;
using TileMid = Tile<6, 6, 2, 128, 4>;
using TileSmall = Tile<6, 2, 2, 128, 4>;
using TileFlat = Tile<14, 30, 1, 160, 3>;
using TileFlatSmall = Tile<14, 6, 1, 128, 4>;
enum { TILE_MAIN = 0, TILE_MID = 1, TILE_SMALL = 2, TILE_FLAT = 3, TILE_FLAT_SMALL = 4 };

// Calls f(Tile{}) for tile number t.
template <class F>
auto by_tile(int t, F&& f) {
  switch (t) {
    case TILE_MID: return f(TileMid{});
    case TILE_SMALL: return f(TileSmall{});
    case TILE_FLAT: return f(TileFlat{});
    case TILE_FLAT_SMALL: return f(TileFlatSmall{});
    default: return f(TileMain{});
  }
}

// The tile of a double grid: the one with the least work on the busiest SM,
// in 32-lane chunks of its sweeps (60 for a main tile, whose sweeps have 18, 21
// and 21), as the FP64 pipe, which bounds these kernels, takes chunks at one
// rate.  Grids of some thousand main tiles keep the main tile; at 19 main
// tiles (the Sod tube, 256 x 4 x 4) an eighth of the SMs had all the work: 240 us per
// step against 92 with the small tile.  More than one dust species: the main
// tile only (the others are not instantiated).
template <class T>
constexpr long tile_chunks() {
  auto sweep = [](int lines, int cells) { return (long)(lines * pow2ceil(cells + 2) + 31) / 32; };
  return sweep(T::TT * T::TZ, T::TR) + sweep(T::TR * T::TZ, T::TT) + (T::TZ > 1 ? sweep(T::TR * T::TT, T::TZ) : 0);
}
inline int choose_tile(int nr, int nth, int nz, bool flat, int nf, int sms) {
  if (nf > 9) return TILE_MAIN;
  const int from = flat ? TILE_FLAT : TILE_MAIN, to = flat ? TILE_FLAT_SMALL : TILE_SMALL;
  int best = from;
  long least = 0;
  for (int t = from; t <= to; ++t) {
    const long work = by_tile(t, [&](auto tile) {
      using T = decltype(tile);
      const long n = (long)((nr + T::TR - 1) / T::TR) * ((nth + T::TT - 1) / T::TT) * ((nz + T::TZ - 1) / T::TZ);
      return (n + sms - 1) / sms * tile_chunks<T>();
    });
    if (t == from || work < least) {
      best = t;
      least = work;
    }
  }
  return best;
}
inline bool flat_grid(int nz, int bc_lo_z, int bc_hi_z, int nf) {
  return nz == 1 && bc_lo_z != BC_EQUILIBRIUM && bc_hi_z != BC_EQUILIBRIUM && nf <= 9;
}

// Calls f(std::integral_constant<int, NF>) for the field count nf (5 + 4 x
// the number of dust species, 0 .. 4).
template <class F>
cudaError_t by_nf(int nf, F&& f) {
  switch (nf) {
    case 5: return f(std::integral_constant<int, 5>{});
    case 9: return f(std::integral_constant<int, 9>{});
    case 13: return f(std::integral_constant<int, 13>{});
    case 17: return f(std::integral_constant<int, 17>{});
    case 21: return f(std::integral_constant<int, 21>{});
  }
  return cudaErrorInvalidValue;
}
// Adjoint flux kernel: lines of 16 lanes (12 owned cells), 12 lines per block,
// or of 32 lanes (28 owned cells), 6 lines per block; 192 threads either way,
// two blocks per SM.  The FP64 pipe bounds it, so an axis takes the lines that
// cover its n cells with fewer lanes: 128 and 256 cells take 160 and 320 lanes
// in wide lines, 176 and 352 in narrow ones (flux kernels of both axes 7 %
// faster, a gradient on 128 x 256 x 32 bi-fluid cells 41.7 -> 41.0 ms), 32
// cells take 48 in narrow lines and 64 in wide ones.
constexpr int ADJ_L = 16, ADJ_NL = 12, ADJ_L_WIDE = 32, ADJ_NL_WIDE = 6;
inline int adj_line(long n) {
  const long narrow = (n + ADJ_L - 5) / (ADJ_L - 4) * ADJ_L, wide = (n + ADJ_L_WIDE - 5) / (ADJ_L_WIDE - 4) * ADJ_L_WIDE;
  return wide < narrow ? ADJ_L_WIDE : ADJ_L;
}

// Raises a kernel's dynamic shared-memory limit once per device (the
// attribute belongs to the current device's context); `done` is the calling
// site's own flag word, one bit per device id < 64.
template <class K>
cudaError_t set_smem_once(K kern, size_t smem, unsigned long long& done) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
  if (bit && (done & bit)) return cudaSuccess;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) done |= bit;
  return e;
}

// Each launcher is instantiated per gas reconstruction mode RC (and power form
// P) in a translation unit of its own, which compile in parallel; the host
// runtime selects one.  (A selecting inline function here would make every
// such unit instantiate all of them.)
// One launch of a stage kernel over nblocks tiles; xt selects the
// instantiation with the optional terms (indirect gravity, damping zones,
// Stokes drag regime).
template <int RC>
cudaError_t run_stage_full_rc(const StageArgs& a, int nblocks, cudaStream_t s, bool xt);
template <class P, int RC>
cudaError_t run_stage_pert_f32_rc(const PertArgs<float>& a, int nblocks, cudaStream_t s, bool xt);
template <int RC>
cudaError_t run_stage_pert_f64_rc(const PertArgs<double>& a, int nblocks, cudaStream_t s, bool xt);
// One launch of the adjoint flux kernel along axis 0, 1 or 2.
cudaError_t run_adj_flux(const AdjFluxArgs& a, int axis, cudaStream_t s);

}  // namespace rossbi
