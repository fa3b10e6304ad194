// Launcher of the FP64 stage kernel (stage_full.cuh) for one gas
// reconstruction mode: ROSSBI_RC, the conservative one unless the including
// translation unit chose another.
#include "launch.cuh"

#ifndef ROSSBI_RC
#define ROSSBI_RC RECON_CONS
#endif

namespace rossbi {
namespace {

template <int NF, class T, bool XT, int RC>
cudaError_t launch(const StageArgs& a, int nblocks, cudaStream_t s) {
  constexpr size_t smem = (size_t)(5 * SweepLane<T::TR, T::TT, T::TZ, 0>::BOX + NF * T::TR * T::TT * T::TZ) * sizeof(double);
  auto kern = stage_full_kernel<NF, T::TR, T::TT, T::TZ, T::NT, T::MINB, XT, RC>;
  static unsigned long long done = 0;
  cudaError_t e = set_smem_once(kern, smem, done);
  if (e != cudaSuccess) return e;
  kern<<<nblocks, T::NT, smem, s>>>(a);
  return cudaGetLastError();
}

template <int NF, int RC>
cudaError_t launch_x(const StageArgs& a, int nblocks, cudaStream_t s, bool xt) {
  auto go = [&](auto tile) {
    using T = decltype(tile);
    return xt ? launch<NF, T, true, RC>(a, nblocks, s) : launch<NF, T, false, RC>(a, nblocks, s);
  };
  if constexpr (NF <= 9) return by_tile(a.tile, go);
  else return go(TileMain{});
}

}  // namespace

template <int RC>
cudaError_t run_stage_full_rc(const StageArgs& a, int nblocks, cudaStream_t s, bool xt) {
  return by_nf(a.g.nf, [&](auto nf) { return launch_x<decltype(nf)::value, RC>(a, nblocks, s, xt); });
}

template cudaError_t run_stage_full_rc<ROSSBI_RC>(const StageArgs&, int, cudaStream_t, bool);

}  // namespace rossbi
