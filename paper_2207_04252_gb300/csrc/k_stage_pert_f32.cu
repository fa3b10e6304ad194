// Launcher of the FP32 perturbation-form stage kernel (stage_f32.cuh) for
// one power form of the solver (ROSSBI_POW: the gamma = 7/5 integer powers
// unless the including translation unit chose the general ones) and one gas
// reconstruction mode (ROSSBI_RC, conservative unless chosen otherwise).
#include "launch.cuh"
#include "stage_f32.cuh"

#ifndef ROSSBI_RC
#define ROSSBI_RC RECON_CONS
#endif
#ifndef ROSSBI_POW
#define ROSSBI_POW PowG75
#endif

namespace rossbi {
namespace {

template <int NF, int NT, int MINB, class P, bool XT, int RC>
cudaError_t launch_nt(const PertArgs<float>& a, int nblocks, cudaStream_t s) {
  constexpr size_t smem = F32Smem<NF, P32_TR, P32_TT, P32_TZ>::bytes;
  auto kern = stage_f32_kernel<NF, P32_TR, P32_TT, P32_TZ, NT, MINB, P, XT, RC>;
  static unsigned long long done = 0;
  cudaError_t e = set_smem_once(kern, smem, done);
  if (e != cudaSuccess) return e;
  kern<<<nblocks, NT, smem, s>>>(a);
  return cudaGetLastError();
}

// Two blocks of 12 warps share an SM where their shared memory allows it (up to
// nine fields) and there are tiles for them; otherwise one block of 24 warps
// takes the SM: more fields (133 KB and up), or a grid of few tiles, where a
// tile's latency counts more than the overlap of one block's staging with
// another's sweeps.  Four steps with dust, two narrow blocks against a wide one:
// 152 tiles 223 / 165 us, 300 230 / 214, 456 308 / 281, 512 319 / 307, 600
// 346 / 333 (without dust 281 / 288), 760 404 / 409, 912 436 / 484, 4800
// 1808 / 2254: the lines cross between three and four tiles per SM of 152 without
// dust and between four and five with it.  One rule at three for both: beyond it
// the narrow blocks lose 4 % at most.
template <int NF, class P, bool XT, int RC>
cudaError_t launch(const PertArgs<float>& a, int nblocks, cudaStream_t s) {
  if constexpr (NF <= 9) {
    if (nblocks > 3 * a.sms) return launch_nt<NF, P32_NT, P32_MINB, P, XT, RC>(a, nblocks, s);
  }
  return launch_nt<NF, P32_WIDE_NT, 1, P, XT, RC>(a, nblocks, s);
}

}  // namespace

template <class P, int RC>
cudaError_t run_stage_pert_f32_rc(const PertArgs<float>& a, int nblocks, cudaStream_t s, bool xt) {
  return by_nf(a.g.nf, [&](auto nf) {
    constexpr int NF = decltype(nf)::value;
    return xt ? launch<NF, P, true, RC>(a, nblocks, s) : launch<NF, P, false, RC>(a, nblocks, s);
  });
}

template cudaError_t run_stage_pert_f32_rc<ROSSBI_POW, ROSSBI_RC>(const PertArgs<float>&, int, cudaStream_t, bool);

}  // namespace rossbi
