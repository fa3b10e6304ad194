// Host runtime and C ABI of the GB300 RoSSBi3D hot-path library.
//
// Owns the mesh tables, the equilibrium tables and balanced residual, the
// reduction slots and the optional scratch state; launches the fused stage
// kernels.  The C ABI is declared (and documented) in include/rossbi.h.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/rossbi.h"
#include "launch.cuh"

using namespace rossbi;

namespace {

constexpr int CFL_NT = 256;

}  // namespace

struct rossbi_grid {
  rossbi_grid_desc desc{};
  cudaStream_t stream = nullptr;
  int device = -1;                     // the device current at rossbi_init_grid
  int sms = 1;                         // its SM count
  int nf = 5;
  size_t ncell = 0;
  DevGrid dg{};
  bool eq_set = false;
  bool has_disc = false;
  rossbi_disc_params disc{};
  // device tables
  double *d_rcoef = nullptr, *d_rslope = nullptr, *d_vol = nullptr, *d_ivol = nullptr;
  double *d_area_r = nullptr, *d_area_t = nullptr, *d_area_z = nullptr, *d_aov = nullptr;
  double *d_ir = nullptr, *d_omk = nullptr, *d_grav = nullptr;
  double *d_e0c = nullptr, *d_e0r = nullptr, *d_e0z = nullptr, *d_r0 = nullptr;
  double* d_w0 = nullptr;              // primitive equilibrium tables (centres, r faces, z faces)
  std::vector<double> h_e0c;
  // reductions and status
  unsigned long long* d_dt = nullptr;  // [2]: ping-pong slots of the largest CFL rate (the step is N_CFL over it)
  int dt_slot = 0;                     // slot holding the rate of the next step
  bool dt_on_device = false;
  double* d_partials = nullptr;
  size_t partials_cap = 0;
  double* d_sums = nullptr;
  unsigned* d_status = nullptr;
  double* h_pinned = nullptr;          // [32] readback area: [0..20] values, [28] status word
  // library-owned buffers
  void* d_scratch = nullptr;           // E* when the caller passes none
  void* d_hoststate = nullptr;         // device copy for rossbi_step_host
  cudaStream_t s_in = nullptr, s_out = nullptr;  // its copies, one stream per direction
  cudaEvent_t host_ev[17] = {};        // slabs copied in [0..7], slabs stepped [8..15], start
  int tiles_r = 0, tiles_t = 0, tiles_z = 0;
  int tile_tt = 6, tile_tz = 6;        // theta and z extents of a stage-kernel tile
  int tile = TILE_MAIN;                // double forms: which tile
  // perturbation forms: equilibrium and metric tables in the state precision
  void* d_ptab = nullptr;              // one allocation holding every table below
  PertTables<float> pt_f{};
  PertTables<double> pt_d{};
  unsigned long long* d_fallbacks = nullptr;
  double eq_sums[5] = {0, 0, 0, 0, 0}; // sum_cells V E0_f (FP64)
  // adjoint: five FP64 states (Y1, E*, Y2, mu', cotangent of E*), d/dSt partials and slots
  double* d_adj = nullptr;
  double* d_adj_part = nullptr;
  double* d_adj_slots = nullptr;       // [0] this call's d/dSt, [1] running total
  // indirect gravity: [2] disc moments A, B; [2][nth] cos / sin of the
  // azimuthal centres; [nz][nr] V r / R^3; [2][IND_BLOCKS] block partials
  double* d_ind = nullptr;
  double* d_adj_ind = nullptr;         // adjoint of the indirect term: [2 stages][2][adj_blocks] partials,
                                       // [2 stages][2] reduced, [2][nth] stage-1 gradient table
  double* d_damp = nullptr;            // relaxation rates of the damping zones per cell centre [nz][nr]
                                       // in double, then [nz][nr] in float
  bool damp_r = false, damp_z = false; // radial wave-killing zones; vertical sheared damped boundary
  rossbi_damping_params damp_rp{};
  rossbi_vertical_damping_params damp_zp{};
  int adj_blocks = 0;
  // stage-kernel timing (rossbi_profile_*)
  bool profiling = false;
  std::vector<cudaEvent_t> ev;         // start/stop pairs
  int ev_used = 0;
  double prof_ms = 0.0;
  int prof_launches = 0;
};

namespace {

size_t elem_size(const rossbi_grid* g) { return g->desc.precision == ROSSBI_FP32_PERT ? 4 : 8; }

#define CK(call)                                            \
  do {                                                      \
    cudaError_t e_ = (call);                                \
    if (e_ != cudaSuccess) {                                \
      return e_ == cudaErrorMemoryAllocation ? ROSSBI_ERR_OOM : ROSSBI_ERR_CUDA; \
    }                                                       \
  } while (0)

template <class T>
rossbi_status upload(T** dst, const std::vector<T>& src, cudaStream_t s) {
  if (*dst) cudaFree(*dst);
  *dst = nullptr;
  CK(cudaMalloc(dst, src.size() * sizeof(T)));
  CK(cudaMemcpyAsync(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice, s));
  return ROSSBI_OK;
}

// ---------------------------------------------------------------- mesh (Sect. 2.3)
double axis0_face(const rossbi_grid_desc& d, int i) {
  if (d.geometry == ROSSBI_GEOM_CYL) return d.x0[0] * std::pow(d.x1[0] / d.x0[0], (double)i / d.nr);
  return d.x0[0] + (d.x1[0] - d.x0[0]) * i / d.nr;
}
double axis0_centre(const rossbi_grid_desc& d, int i) {
  if (d.geometry == ROSSBI_GEOM_CYL) return std::sqrt(axis0_face(d, i) * axis0_face(d, i + 1));
  return 0.5 * (axis0_face(d, i) + axis0_face(d, i + 1));
}

// ---------------------------------------------------------------- equilibrium (App. A)
void equilibrium_prim(const rossbi_grid_desc& d, const rossbi_disc_params& p, double r, double z, double& rho,
                      double& vth, double& pres, double* dlnp_out = nullptr) {
  const double cs2 = p.T0 * std::pow(r, p.beta_T);
  const double omk = std::sqrt(d.gm / (r * r * r));
  const double H = std::sqrt(2.0 * cs2) / omk;
  const double R = std::sqrt(r * r + z * z);
  const double gpot = 1.0 / R - 1.0 / r;
  rho = p.sigma0 * std::pow(r, p.beta_sigma) / (std::sqrt(M_PI) * H) * std::exp(d.gm / cs2 * gpot);
  pres = cs2 * rho;
  double dlnp = (p.beta_T + p.beta_sigma - 0.5 * (p.beta_T + 3.0)) / r +
                d.gm / cs2 * (-p.beta_T * gpot / r - r / (R * R * R) + 1.0 / (r * r));
  if (p.bump_delta != 0.0) {  // Sect. 4.3: rho, P x (1 + delta G) at the same T; d ln P / dr gains its log-derivative
    const double x = (r - p.bump_r0) / p.bump_width;
    const double G = std::exp(-0.5 * x * x);
    const double s = 1.0 + p.bump_delta * G;
    rho *= s;
    pres *= s;
    dlnp -= p.bump_delta * G * x / (p.bump_width * s);
  }
  vth = std::sqrt(d.gm * r * r / (R * R * R) + r * cs2 * dlnp);
  if (dlnp_out) *dlnp_out = dlnp;
}

void equilibrium_cons(const rossbi_grid_desc& d, const rossbi_disc_params& p, double r, double z, double* U,
                      size_t stride) {
  double rho, vth, pres;
  equilibrium_prim(d, p, r, z, rho, vth, pres);
  const double v = vth - d.omega_frame * r;
  U[MU * stride] = 0.0;
  U[MV * stride] = rho * v;
  U[MW * stride] = 0.0;
  U[EN * stride] = 0.5 * rho * v * v + pres / (d.gamma - 1.0);
  U[RHO * stride] = rho;
}

rossbi_status check_desc(const rossbi_grid_desc& d) {
  if (d.nr < 1 || d.nth < 1 || d.nz < 1) return ROSSBI_ERR_ARG;
  if (d.geometry != ROSSBI_GEOM_BOX && d.geometry != ROSSBI_GEOM_CYL) return ROSSBI_ERR_ARG;
  if (!(d.gamma > 1.0) || !(d.cfl > 0.0)) return ROSSBI_ERR_ARG;
  if (d.n_dust < 0 || d.n_dust > ND_MAX) return ROSSBI_ERR_UNSUPPORTED;
  for (int a = 0; a < 3; ++a) {
    if (!(d.x1[a] > d.x0[a])) return ROSSBI_ERR_ARG;
    for (int bc : {d.bc_lo[a], d.bc_hi[a]})
      if (bc < ROSSBI_BC_PERIODIC || bc > ROSSBI_BC_EQUILIBRIUM) return ROSSBI_ERR_ARG;
    if ((d.bc_lo[a] == ROSSBI_BC_PERIODIC) != (d.bc_hi[a] == ROSSBI_BC_PERIODIC)) return ROSSBI_ERR_ARG;
  }
  if (d.geometry == ROSSBI_GEOM_CYL) {
    if (!(d.x0[0] > 0.0) || !(d.gm >= 0.0) || !std::isfinite(d.gm)) return ROSSBI_ERR_ARG;
    if (d.bc_lo[1] != ROSSBI_BC_PERIODIC) return ROSSBI_ERR_ARG;
    if (d.bc_lo[0] == ROSSBI_BC_PERIODIC) return ROSSBI_ERR_ARG;
  }
  if (d.precision != ROSSBI_FP64 && d.precision != ROSSBI_FP32_PERT && d.precision != ROSSBI_FP64_PERT)
    return ROSSBI_ERR_ARG;
  if (d.recon != ROSSBI_RECON_CONSERVATIVE && d.recon != ROSSBI_RECON_PRIMITIVE) return ROSSBI_ERR_ARG;
  return ROSSBI_OK;
}

rossbi_status status_from_word(unsigned w) {
  if (w & STATUS_NONPHYSICAL) return ROSSBI_ERR_NONPHYSICAL;
  if (w & STATUS_RIEMANN) return ROSSBI_ERR_RIEMANN;
  return ROSSBI_OK;
}

rossbi_status sync_and_status(rossbi_grid* g) {
  CK(cudaMemcpyAsync(g->h_pinned + 28, g->d_status, sizeof(unsigned), cudaMemcpyDeviceToHost, g->stream));
  CK(cudaMemsetAsync(g->d_status, 0, sizeof(unsigned), g->stream));
  CK(cudaStreamSynchronize(g->stream));
  unsigned w;
  std::memcpy(&w, g->h_pinned + 28, sizeof(unsigned));
  return status_from_word(w);
}

// The step length N_CFL / rate of a rate slot, on the host (no cell with a
// rate: infinite).  Synchronises.
rossbi_status read_dt(rossbi_grid* g, int slot, double* dt) {
  CK(cudaMemcpyAsync(g->h_pinned, g->d_dt + slot, sizeof(double), cudaMemcpyDeviceToHost, g->stream));
  const rossbi_status st = sync_and_status(g);
  *dt = g->desc.cfl / g->h_pinned[0];
  return st;
}

// ---------------------------------------------------------------- kernels
template <int NF>
__global__ void cfl_kernel(DevGrid g, StageArgs a, unsigned long long* slot) {
  const size_t ncell = (size_t)g.nr * g.nth * g.nz;
  double rate = 0.0;
  unsigned status = 0;
  for (size_t lin = blockIdx.x * (size_t)CFL_NT + threadIdx.x; lin < ncell; lin += (size_t)gridDim.x * CFL_NT) {
    double U[NF], id[NF > 5 ? (NF - 5) / 4 : 1];
#pragma unroll
    for (int f = 0; f < NF; ++f) U[f] = a.in[f][lin];
#pragma unroll
    for (int b = 5; b < NF; b += 4) id[(b - 5) / 4] = recip(U[b + 3]);
    bool bad = false;
    const double c = cell_rate<NF>(g, (int)(lin % g.nr), U, recip(U[RHO]), id, bad);
    if (bad) status |= STATUS_NONPHYSICAL;
    if (positive(c) && mag_less(rate, c)) rate = c;
  }
  raise_rate(slot, rate);
  if (status) atomicOr(a.status, status);
}

// Primitive equilibrium table from a conservative one ([5][n] each), with the
// conversion the stage kernels apply to the state, so that the deviations of
// an equilibrium state are exactly zero.
__global__ void eq_prim_kernel(double gamma, const double* e, double* w, size_t n) {
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n; q += (size_t)gridDim.x * blockDim.x) {
    double U[5], W[5];
    for (int f = 0; f < 5; ++f) U[f] = e[f * n + q];
    cell_prim_rounded(gamma, U, W);
    for (int f = 0; f < 5; ++f) w[f * n + q] = W[f];
  }
}

// Per-block FP64 partial sums of V * E_f, fixed order.
__global__ void sums_kernel(DevGrid g, StageArgs a, double* partials) {
  __shared__ double red[CFL_NT / 32];
  const size_t ncell = (size_t)g.nr * g.nth * g.nz;
  double s[NF_MAX] = {};
  for (size_t lin = blockIdx.x * (size_t)CFL_NT + threadIdx.x; lin < ncell; lin += (size_t)gridDim.x * CFL_NT) {
    const double V = g.vol[lin % g.nr];
    for (int f = 0; f < g.nf; ++f) s[f] += V * a.in[f][lin];
  }
  for (int f = 0; f < g.nf; ++f) {
    const double t = block_sum<CFL_NT>(s[f], red);
    if (threadIdx.x == 0) partials[(size_t)f * gridDim.x + blockIdx.x] = t;
  }
}

// Sums the per-block partials row by row in a fixed order (so the result
// does not depend on scheduling) into sums[].
constexpr int RED_NT = 512;
__global__ void __launch_bounds__(RED_NT) reduce_partials_kernel(const double* partials, int nblocks, double* sums) {
  __shared__ double red[RED_NT / 32];
  const int row = blockIdx.x;
  const double* p = partials + (size_t)row * nblocks;
  double v = 0.0;
  for (int b = threadIdx.x; b < nblocks; b += RED_NT) v += p[b];
  v = block_sum<RED_NT>(v, red);
  if (threadIdx.x == 0) sums[row] = v;
}

// Dust densities of every species (null beyond n).
template <class T>
struct DustRho {
  const T* p[ND_MAX];
  int n;
};

// Disc moments of the indirect gravity (Sect. 2.10): per-block FP64 partial
// sums of w (rho - rho_0 + sum rho_d) cos(theta) and ... sin(theta), with
// w = V r / R^3 of the cell centre; `full` states carry rho itself, the
// perturbation forms rho' already.  A warp takes one azimuthal row (nr cells)
// at a time; each lane sums its cells of the row in the state's precision
// (FP32: against a float copy of w, so that GB300's narrow FP64 pipe sees
// three operations per lane and row instead of several per cell), then the
// row sums are weighted by cos / sin and accumulated in FP64.  Rows go to
// warps in a fixed order, so the sums are reproducible.
constexpr int IND_NT = 256, IND_BLOCKS = 152 * 4;
template <class T, int ND>
__global__ void __launch_bounds__(IND_NT) indirect_moments_kernel(DevGrid g, const T* rho, const DustRho<T> dr,
                                                                  int full, const double* w, const float* wf,
                                                                  double* partials) {
  __shared__ double red[IND_NT / 32];
  constexpr int NW = IND_NT / 32;
  const int lane = threadIdx.x & 31;
  double A = 0.0, B = 0.0;
  const int rows = g.nth * g.nz;
  for (int row = blockIdx.x * NW + (threadIdx.x >> 5); row < rows; row += gridDim.x * NW) {
    const int j = row % g.nth, k = row / g.nth;
    const size_t base = (size_t)row * g.nr;
    T m = T(0);
    if constexpr (sizeof(T) == 4) {
      const float* wk = wf + (size_t)k * g.nr;
      for (int i = lane; i < g.nr; i += 32) {
        float x = rho[base + i];
#pragma unroll
        for (int s = 0; s < ND; ++s) x += dr.p[s][base + i];  // static indices: the pointers stay in the parameter bank
        m += x * wk[i];
      }
    } else {
      const double* wk = w + (size_t)k * g.nr;
      const double* e0 = full && g.has_eq ? g.e0c + ((size_t)RHO * g.nz + k) * g.nr : nullptr;
      for (int i = lane; i < g.nr; i += 32) {
        double dm = rho[base + i];
        if (e0) dm -= e0[i];
#pragma unroll
        for (int s = 0; s < ND; ++s) dm += dr.p[s][base + i];
        m += dm * wk[i];
      }
    }
    A += (double)m * g.ind_cs[j];
    B += (double)m * g.ind_cs[g.nth + j];
  }
  A = block_sum<IND_NT>(A, red);
  B = block_sum<IND_NT>(B, red);
  if (threadIdx.x == 0) {
    partials[blockIdx.x] = A;
    partials[gridDim.x + blockIdx.x] = B;
  }
}

// Fixed-order reduction of the moment partials into (A_disc, B_disc), as
// reduce_partials_kernel does it, then the gradient of the indirect
// potential at every axis-1 index, X_ref (A cos + B sin, -A sin + B cos), in
// double and in float (the stage epilogues read it per cell).
__global__ void __launch_bounds__(RED_NT) indirect_reduce_kernel(const double* partials, int nblocks, int nth,
                                                                 double x_ref, const double* cs, double* ab,
                                                                 double* gtab, float* gtabf) {
  __shared__ double red[RED_NT / 32];
  __shared__ double AB[2];
  for (int row = 0; row < 2; ++row) {
    const double* p = partials + (size_t)row * nblocks;
    double v = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += RED_NT) v += p[b];
    v = block_sum<RED_NT>(v, red);
    if (threadIdx.x == 0) AB[row] = v;
  }
  __syncthreads();
  const double A = AB[0], B = AB[1];
  if (threadIdx.x == 0) {
    ab[0] = A;
    ab[1] = B;
  }
  for (int j = threadIdx.x; j < nth; j += RED_NT) {
    const double c = cs[j], s = cs[nth + j];
    const double gr = x_ref * (A * c + B * s), gt = x_ref * (-A * s + B * c);
    gtab[j] = gr;
    gtab[nth + j] = gt;
    gtabf[j] = (float)gr;
    gtabf[nth + j] = (float)gt;
  }
}

// Halo rows of a decomposition in theta (Sect. 3.1 splits the grid into
// blocks of cells): copies rows j0 .. j0 + rows - 1 of every field between
// the state (SoA, index (k nth + j) nr + i) and a contiguous buffer laid out
// [f][k][jj][i].  One thread per element, consecutive threads along r, so
// both sides are read and written in coalesced runs of nr elements.
template <class T>
struct FieldPtrs {
  T* p[NF_MAX];
};
template <class T>
__global__ void theta_rows_kernel(FieldPtrs<T> st, T* buf, int nr, int nth, int nz, int nf, int j0, int rows,
                                  int unpack) {
  const size_t per_field = (size_t)nz * rows * nr, n = per_field * nf;
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n; q += (size_t)gridDim.x * blockDim.x) {
    const int f = (int)(q / per_field);
    const size_t r = q - (size_t)f * per_field;
    const int i = (int)(r % nr);
    const size_t kj = r / nr;
    const int jj = (int)(kj % rows), k = (int)(kj / rows);
    const size_t lin = ((size_t)k * nth + (j0 + jj)) * nr + i;
    if (unpack) st.p[f][lin] = buf[q];
    else buf[q] = st.p[f][lin];
  }
}

constexpr int PROFILE_PAIRS = 1024;

rossbi_status profile_drain(rossbi_grid* g) {
  if (g->ev_used == 0) return ROSSBI_OK;
  CK(cudaStreamSynchronize(g->stream));
  for (int q = 0; q < g->ev_used; ++q) {
    float ms = 0.f;
    CK(cudaEventElapsedTime(&ms, g->ev[2 * q], g->ev[2 * q + 1]));
    g->prof_ms += ms;
  }
  g->prof_launches += g->ev_used;
  g->ev_used = 0;
  return ROSSBI_OK;
}

// The launcher of a grid's reconstruction mode and, for the float form, of
// the gamma = 7/5 integer powers or the general ones.
cudaError_t run_stage_full(const StageArgs& a, int nblocks, cudaStream_t s, bool xt) {
  return a.g.recon == RECON_PRIM ? run_stage_full_rc<RECON_PRIM>(a, nblocks, s, xt)
                                 : run_stage_full_rc<RECON_CONS>(a, nblocks, s, xt);
}
cudaError_t run_stage_pert(const PertArgs<float>& a, int nblocks, cudaStream_t s, bool xt) {
  const bool g75 = a.g.gamma == 1.4;
  if (a.g.recon == RECON_PRIM)
    return g75 ? run_stage_pert_f32_rc<PowG75, RECON_PRIM>(a, nblocks, s, xt)
               : run_stage_pert_f32_rc<PowGeneric<float>, RECON_PRIM>(a, nblocks, s, xt);
  return g75 ? run_stage_pert_f32_rc<PowG75, RECON_CONS>(a, nblocks, s, xt)
             : run_stage_pert_f32_rc<PowGeneric<float>, RECON_CONS>(a, nblocks, s, xt);
}
cudaError_t run_stage_pert(const PertArgs<double>& a, int nblocks, cudaStream_t s, bool xt) {
  return a.g.recon == RECON_PRIM ? run_stage_pert_f64_rc<RECON_PRIM>(a, nblocks, s, xt)
                                 : run_stage_pert_f64_rc<RECON_CONS>(a, nblocks, s, xt);
}

cudaError_t run_stage(const StageArgs& a, int nblocks, cudaStream_t s, bool xt) {
  return run_stage_full(a, nblocks, s, xt);
}
template <class T>
cudaError_t run_stage(const PertArgs<T>& a, int nblocks, cudaStream_t s, bool xt) {
  return run_stage_pert(a, nblocks, s, xt);
}

// One launch of the form's stage kernel over nblocks tiles, timed where asked.
template <class Args>
rossbi_status launch_stage(rossbi_grid* g, const Args& a, int nblocks, bool timed = true) {
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (g->profiling && timed) {
    if (g->ev_used == PROFILE_PAIRS) {
      rossbi_status st = profile_drain(g);
      if (st != ROSSBI_OK) return st;
    }
    e0 = g->ev[2 * g->ev_used];
    e1 = g->ev[2 * g->ev_used + 1];
    CK(cudaEventRecord(e0, g->stream));
  }
  const bool xt = a.g.x_ind != 0.0 || a.g.damp_k != nullptr || a.drag.law == 2;  // optional terms on
  CK(run_stage(a, nblocks, g->stream, xt));
  if (e0) {
    CK(cudaEventRecord(e1, g->stream));
    g->ev_used++;
  }
  return ROSSBI_OK;
}

int n_tiles(const rossbi_grid* g) { return g->tiles_r * g->tiles_t * g->tiles_z; }

rossbi_status ensure_partials(rossbi_grid* g, size_t nblocks) {
  if (g->partials_cap >= nblocks) return ROSSBI_OK;
  if (g->d_partials) cudaFree(g->d_partials);
  g->d_partials = nullptr;
  g->partials_cap = 0;
  CK(cudaMalloc(&g->d_partials, nblocks * (NF_MAX + 1) * sizeof(double)));
  g->partials_cap = nblocks;
  return ROSSBI_OK;
}

StageArgs base_args(rossbi_grid* g) {
  StageArgs a;
  std::memset(&a, 0, sizeof(a));
  a.g = g->dg;
  a.status = g->d_status;
  a.order = TileOrder{fast_div(g->tiles_r), fast_div(g->tiles_z), 0};
  a.tile = g->tile;
  return a;
}

// The empty run of Sect. 2.8 on a one-tile-thick azimuthal slab of the grid
// (same dtheta, so the same arithmetic as every column of the full grid).
rossbi_status empty_run(rossbi_grid* g) {
  const rossbi_grid_desc& d = g->desc;
  const int nth_s = std::min(d.nth, g->tile_tt);
  const size_t nslab = (size_t)d.nr * nth_s * d.nz;
  std::vector<double> E0(nslab * g->nf, 0.0);
  for (int f = 0; f < 5; ++f)
    for (int k = 0; k < d.nz; ++k)
      for (int j = 0; j < nth_s; ++j)
        for (int i = 0; i < d.nr; ++i)
          E0[f * nslab + ((size_t)k * nth_s + j) * d.nr + i] = g->h_e0c[((size_t)f * d.nz + k) * d.nr + i];
  double *dE = nullptr, *dG = nullptr;
  CK(cudaMalloc(&dE, E0.size() * sizeof(double)));
  cudaError_t e = cudaMalloc(&dG, E0.size() * sizeof(double));
  if (e != cudaSuccess) { cudaFree(dE); return ROSSBI_ERR_OOM; }
  rossbi_status st = ROSSBI_OK;
  do {
    if (cudaMemcpyAsync(dE, E0.data(), E0.size() * sizeof(double), cudaMemcpyHostToDevice, g->stream) !=
        cudaSuccess) { st = ROSSBI_ERR_CUDA; break; }
    StageArgs a = base_args(g);
    a.g.nth = nth_s;
    a.g.r0 = nullptr;
    a.g.x_ind = 0.0;  // the equilibrium's residual carries no indirect term
    a.g.damp_k = nullptr;  // nor a relaxation (E' = 0 there)
    for (int f = 0; f < g->nf; ++f) a.in[f] = dE + f * nslab;
    a.gout = dG;
    a.mode = 1;
    const int nblocks = g->tiles_r * 1 * g->tiles_z;  // one tile along theta
    st = launch_stage(g, a, nblocks, false);
    if (st != ROSSBI_OK) break;
    std::vector<double> G(E0.size());
    if (cudaMemcpyAsync(G.data(), dG, G.size() * sizeof(double), cudaMemcpyDeviceToHost, g->stream) !=
        cudaSuccess) { st = ROSSBI_ERR_CUDA; break; }
    if (cudaStreamSynchronize(g->stream) != cudaSuccess) { st = ROSSBI_ERR_CUDA; break; }
    std::vector<double> R0((size_t)5 * d.nz * d.nr);
    for (int f = 0; f < 5; ++f)
      for (int k = 0; k < d.nz; ++k)
        for (int i = 0; i < d.nr; ++i)
          R0[((size_t)f * d.nz + k) * d.nr + i] = G[f * nslab + ((size_t)k * nth_s) * d.nr + i];
    st = upload(&g->d_r0, R0, g->stream);
    if (st != ROSSBI_OK) break;
    if (cudaStreamSynchronize(g->stream) != cudaSuccess) { st = ROSSBI_ERR_CUDA; break; }
  } while (false);
  cudaFree(dE);
  cudaFree(dG);
  return st;
}

rossbi_status ensure_scratch(rossbi_grid* g, void** buf) {
  if (*buf) return ROSSBI_OK;
  CK(cudaMalloc(buf, g->ncell * g->nf * elem_size(g)));
  return ROSSBI_OK;
}

// Tables of the perturbation forms in the state precision T, built from FP64.
template <class T>
rossbi_status build_pert_tables(rossbi_grid* g, PertTables<T>& pt) {
  const rossbi_grid_desc& d = g->desc;
  const int nr = d.nr, nz = d.nz;
  const size_t ncen = (size_t)nz * nr, nfr = (size_t)nz * (nr + 1), nfz = (size_t)(nz + 1) * nr;
  // offsets in elements, each a multiple of 8 (the kernels load 16 bytes at a time)
  size_t total = 0;
  auto room = [&](size_t n) {
    const size_t at = total;
    total += (n + 7) & ~(size_t)7;
    return at;
  };
  const size_t off_cen = room(8 * ncen);
  const size_t nface[3] = {nfr, ncen, nfz};
  size_t off_face[3], off_wave[3];
  for (int q = 0; q < 3; ++q) {
    off_face[q] = room(4 * nface[q]);
    off_wave[q] = room(4 * nface[q]);
  }
  const size_t off_rc = room((size_t)(nr + 2) * RCW), off_vol = room(nr), off_ivol = room(nr), off_ar = room(nr + 1);
  const size_t off_at = room(nr), off_az = room(nr), off_ma = room(nr), off_om = room(nr);
  std::vector<double> h(total, 0.0);
  std::vector<double> v(nr), rcoef((size_t)(nr + 2) * RCW), ar(nr + 1), at(nr), az(nr), ma(nr), iv(nr);
  if (cudaMemcpy(v.data(), g->d_vol, nr * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess ||
      cudaMemcpy(iv.data(), g->d_ivol, nr * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess ||
      cudaMemcpy(rcoef.data(), g->d_rcoef, rcoef.size() * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess ||
      cudaMemcpy(ar.data(), g->d_area_r, ar.size() * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess ||
      cudaMemcpy(at.data(), g->d_area_t, nr * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess ||
      cudaMemcpy(az.data(), g->d_area_z, nr * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess ||
      cudaMemcpy(ma.data(), g->d_aov, nr * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess)
    return ROSSBI_ERR_CUDA;
  for (size_t q = 0; q < rcoef.size(); ++q) h[off_rc + q] = rcoef[q];
  for (int i = 0; i < nr; ++i) {
    h[off_vol + i] = v[i];
    h[off_ivol + i] = iv[i];
    h[off_at + i] = at[i];
    h[off_az + i] = az[i];
    h[off_ma + i] = ma[i];
    const double r = axis0_centre(d, i);
    h[off_om + i] = d.geometry == ROSSBI_GEOM_CYL ? std::sqrt(d.gm / (r * r * r)) : 1.0;
  }
  for (int i = 0; i <= nr; ++i) h[off_ar + i] = ar[i];
  if (g->has_disc) {
    const double dz = (d.x1[2] - d.x0[2]) / nz, Om = d.omega_frame, gam = d.gamma;
    auto prim = [&](int axis, size_t at, double r, double z) {
      double rho, vth, p, dlnp;
      equilibrium_prim(d, g->disc, r, z, rho, vth, p, &dlnp);
      const double v0 = vth - Om * r, c0 = std::sqrt(gam * p / rho), un = axis == 1 ? v0 : 0.0;
      const double f[4] = {rho, v0, p, 0.5 * rho * v0 * v0 + gam * p / (gam - 1.0)};
      const double w[4] = {c0, un - c0, un + c0, 0.0};
      for (int q = 0; q < 4; ++q) {
        h[off_face[axis] + 4 * at + q] = f[q];
        h[off_wave[axis] + 4 * at + q] = w[q];
      }
    };
    for (int k = 0; k < nz; ++k) {
      const double z = d.x0[2] + (k + 0.5) * dz;
      for (int i = 0; i < nr; ++i) {
        const double r = axis0_centre(d, i);
        double rho, vth, p, dlnp;
        equilibrium_prim(d, g->disc, r, z, rho, vth, p, &dlnp);
        const double v0 = vth - Om * r, R2 = r * r + z * z, R3 = R2 * std::sqrt(R2);
        const double cs2 = g->disc.T0 * std::pow(r, g->disc.beta_T);
        double* c = &h[off_cen + 8 * ((size_t)k * nr + i)];
        c[0] = rho;
        c[1] = v0;
        c[2] = p;
        c[3] = cs2 * dlnp;                       // (1/rho0) dP0/dr
        c[4] = -d.gm * z / R3;                   // f_z
        c[5] = -d.gm * r / R3 + Om * Om * r;     // f_r + Omega^2 r
        c[6] = 2.0 * v0 / r + 2.0 * Om;
        c[7] = 1.0 / r;
        prim(1, (size_t)k * nr + i, r, z);
      }
      for (int i = 0; i <= nr; ++i) prim(0, (size_t)k * (nr + 1) + i, axis0_face(d, i), z);
    }
    for (int k = 0; k <= nz; ++k) {
      const double z = d.x0[2] + k * dz;
      for (int i = 0; i < nr; ++i) prim(2, (size_t)k * nr + i, axis0_centre(d, i), z);
    }
  }
  std::vector<T> ht(total);
  for (size_t q = 0; q < total; ++q) ht[q] = (T)h[q];
  if (g->d_ptab) cudaFree(g->d_ptab);
  g->d_ptab = nullptr;
  CK(cudaMalloc(&g->d_ptab, total * sizeof(T)));
  CK(cudaMemcpy(g->d_ptab, ht.data(), total * sizeof(T), cudaMemcpyHostToDevice));
  const T* b = (const T*)g->d_ptab;
  pt.cen = b + off_cen;
  for (int q = 0; q < 3; ++q) {
    pt.face[q] = b + off_face[q];
    pt.wave[q] = b + off_wave[q];
  }
  pt.rcoef = b + off_rc;
  pt.vol = b + off_vol;
  pt.ivol = b + off_ivol;
  pt.area_r = b + off_ar;
  pt.area_t = b + off_at;
  pt.area_z = b + off_az;
  pt.aov = b + off_ma;
  pt.omk = b + off_om;
  if (!g->d_fallbacks) {
    CK(cudaMalloc(&g->d_fallbacks, sizeof(unsigned long long)));
    CK(cudaMemset(g->d_fallbacks, 0, sizeof(unsigned long long)));
  }
  pt.fallbacks = g->d_fallbacks;
  for (int f = 0; f < 5; ++f) {
    double sum = 0.0;
    for (int k = 0; k < nz; ++k)
      for (int i = 0; i < nr; ++i) sum += v[i] * g->h_e0c[((size_t)f * nz + k) * nr + i];
    g->eq_sums[f] = sum * d.nth;
  }
  return ROSSBI_OK;
}

template <class T>
PertArgs<T> pert_args(rossbi_grid* g) {
  PertArgs<T> a;
  std::memset(&a, 0, sizeof(a));
  a.g = g->dg;
  if constexpr (sizeof(T) == 4) a.t = g->pt_f;
  else a.t = g->pt_d;
  a.status = g->d_status;
  a.order = TileOrder{fast_div(g->tiles_r), fast_div(g->tiles_z), 0};
  a.sms = g->sms;
  a.tile = g->tile;
  a.gam = (T)g->dg.gamma;
  a.om = (T)g->dg.omega;
  a.gm1 = (T)(g->dg.gamma - 1.0);
  a.g_gm1 = (T)g->dg.near.g_gm1;
  return a;
}

// The drag parameters of a step in the state precision.
template <class T>
void set_pert_drag(PertArgs<T>& a, const DragArgs& drag) {
  a.drag = drag;
  a.kappa = (T)drag.kappa;
  for (int sp = 0; sp < ND_MAX; ++sp) {
    a.ist[sp] = (T)drag.ist[sp];
    a.irr[sp] = (T)drag.irr[sp];
  }
}

// Drag parameters of a step (Sect. 2.9 drag law; Epstein constant fixed so
// that the Stokes number holds at r = 1, z = 0).
rossbi_status drag_args(rossbi_grid* g, const rossbi_dust_params* dust, DragArgs& drag) {
  drag = DragArgs{};
  double unit = 0.0;  // rho_s r_p of St = 1
  if (g->nf > 5) {
    drag.stokes = dust->stokes;
    drag.law = dust->drag_law;
    if (!(dust->stokes > 0.0)) return ROSSBI_ERR_ARG;
    if (dust->drag_law == 0 && g->desc.geometry == ROSSBI_GEOM_CYL && !(g->desc.gm > 0.0))
      return ROSSBI_ERR_ARG;  // t_s = St / Omega_K needs a star
    if (dust->drag_law == 2) {  // Epstein constant as for law 1, plus the Stokes regime
      if (!(dust->kappa >= 0.0) || !std::isfinite(dust->kappa)) return ROSSBI_ERR_ARG;
      drag.kappa = dust->kappa;
    }
    if (dust->drag_law == 1 || dust->drag_law == 2) {
      if (!g->has_disc) return ROSSBI_ERR_ARG;
      double rho1, vth1, p1;
      equilibrium_prim(g->desc, g->disc, 1.0, 0.0, rho1, vth1, p1);
      const double cs1 = std::sqrt(g->desc.gamma * p1 / rho1), om1 = std::sqrt(g->desc.gm);
      drag.rhos_rp = dust->stokes * rho1 * cs1 / om1;
      unit = rho1 * cs1 / om1;
    } else if (dust->drag_law != 0) {
      return ROSSBI_ERR_ARG;
    }
    // A Stokes number below `least` stops the dust to a part in 10^14 (of the
    // state's 10^7) or 10^190 in any step worth taking: it is taken as `least`,
    // whose inverse is a number in the state's precision.
    const double least = g->desc.precision == ROSSBI_FP32_PERT ? 0x1p-66 : 0x1p-660;
    for (int s = 0; s < ND_MAX; ++s) {
      const double f = g->dg.st_factor[s], st = drag.stokes * f;
      drag.ist[s] = 1.0 / std::max(st, least);
      drag.irr[s] = 1.0 / (st > least ? drag.rhos_rp * f : least * unit);
    }
  }
  return ROSSBI_OK;
}

rossbi_status prepare_step(rossbi_grid* g, void* const* state, void* const* scratch, double dt,
                           const rossbi_dust_params* dust, void** sc, DragArgs& drag) {
  if (!g->eq_set) return ROSSBI_ERR_ARG;
  if (!state) return ROSSBI_ERR_ARG;
  for (int f = 0; f < g->nf; ++f)
    if (!state[f]) return ROSSBI_ERR_ARG;
  if (g->nf > 5 && !dust) return ROSSBI_ERR_ARG;
  if (dt < 0.0 || !std::isfinite(dt)) return ROSSBI_ERR_ARG;
  if (dt == 0.0 && !g->dt_on_device) return ROSSBI_ERR_ARG;
  if (scratch) {
    for (int f = 0; f < g->nf; ++f) {
      if (!scratch[f]) return ROSSBI_ERR_ARG;
      for (int h = 0; h < g->nf; ++h)
        if (scratch[f] == state[h]) return ROSSBI_ERR_ARG;  // E* must not overwrite E^n
      sc[f] = scratch[f];
    }
  } else {
    rossbi_status st = ensure_scratch(g, &g->d_scratch);
    if (st != ROSSBI_OK) return st;
    for (int f = 0; f < g->nf; ++f) sc[f] = (char*)g->d_scratch + (size_t)f * g->ncell * elem_size(g);
  }
  return drag_args(g, dust, drag);
}

// Layout of the indirect-gravity tables, offsets in doubles: [2] the moments
// A, B; [2][nth] cos / sin of the azimuthal centres; [nz][nr] the weights
// V r / R^3 of the cell centres; [2][IND_BLOCKS] block partials; [2][nth]
// the gradient of the indirect potential; the same as floats; the weights as
// floats (for the FP32 form).
struct IndLayout {
  size_t cs, w, part, g, gf, wf, total;
};
IndLayout ind_layout(const rossbi_grid_desc& d) {
  const size_t nw = (size_t)d.nz * d.nr, nth = d.nth;
  IndLayout L;
  L.cs = 2;
  L.w = L.cs + 2 * nth;
  L.part = L.w + nw;
  L.g = L.part + 2 * (size_t)IND_BLOCKS;
  L.gf = L.g + 2 * nth;
  L.wf = L.gf + nth;  // 2 nth floats
  L.total = L.wf + (nw + 1) / 2;
  return L;
}

// Device tables of the indirect gravity (allocated once, layout above).
rossbi_status ensure_ind_tables(rossbi_grid* g) {
  if (g->d_ind) return ROSSBI_OK;
  const rossbi_grid_desc& d = g->desc;
  const double dy = (d.x1[1] - d.x0[1]) / d.nth, dz = (d.x1[2] - d.x0[2]) / d.nz;
  const IndLayout L = ind_layout(d);
  const size_t nw = (size_t)d.nz * d.nr, wf_at = L.wf;
  std::vector<double> h(L.total, 0.0);
  for (int j = 0; j < d.nth; ++j) {
    const double th = d.x0[1] + (j + 0.5) * dy;
    h[2 + j] = std::cos(th);
    h[2 + d.nth + j] = std::sin(th);
  }
  double* w = h.data() + 2 + 2 * (size_t)d.nth;
  for (int k = 0; k < d.nz; ++k) {
    const double z = d.x0[2] + (k + 0.5) * dz;
    for (int i = 0; i < d.nr; ++i) {
      const double r = axis0_centre(d, i), rm = axis0_face(d, i), rp = axis0_face(d, i + 1);
      const double V = 0.5 * (rp * rp - rm * rm) * dy * dz, R2 = r * r + z * z;
      w[(size_t)k * d.nr + i] = V * r / (R2 * std::sqrt(R2));
    }
  }
  std::vector<float> wf(nw);
  for (size_t q = 0; q < nw; ++q) wf[q] = (float)w[q];
  std::memcpy(h.data() + wf_at, wf.data(), nw * sizeof(float));
  rossbi_status st = upload(&g->d_ind, h, g->stream);
  if (st == ROSSBI_OK && cudaStreamSynchronize(g->stream) != cudaSuccess) st = ROSSBI_ERR_CUDA;
  if (st != ROSSBI_OK) {
    if (g->d_ind) cudaFree(g->d_ind);
    g->d_ind = nullptr;
    return st;
  }
  g->dg.ind_cs = g->d_ind + L.cs;
  g->dg.ind_g = g->d_ind + L.g;
  g->dg.ind_gf = reinterpret_cast<const float*>(g->d_ind + L.gf);
  return ROSSBI_OK;
}

// X_ref-free disc moments (A_disc, B_disc) of a state into d_ind[0..1].
rossbi_status indirect_moments(rossbi_grid* g, void* const* state) {
  const rossbi_grid_desc& d = g->desc;
  const IndLayout L = ind_layout(d);
  const double* w = g->d_ind + L.w;
  double* part = g->d_ind + L.part;
  const float* wf = reinterpret_cast<const float*>(g->d_ind + L.wf);
  // one instantiation per dust-species count
  auto launch = [&](auto tag, auto nd) {
    using T = decltype(tag);
    constexpr int ND = decltype(nd)::value;
    DustRho<T> dr{};
    for (int b = 5; b < g->nf; b += 4) dr.p[dr.n++] = (const T*)state[b + 3];
    indirect_moments_kernel<T, ND><<<IND_BLOCKS, IND_NT, 0, g->stream>>>(
        g->dg, (const T*)state[RHO], dr, d.precision == ROSSBI_FP64, w, wf, part);
  };
  auto by_species = [&](auto tag) {
    switch ((g->nf - 5) / 4) {
      case 0: launch(tag, std::integral_constant<int, 0>{}); break;
      case 1: launch(tag, std::integral_constant<int, 1>{}); break;
      case 2: launch(tag, std::integral_constant<int, 2>{}); break;
      case 3: launch(tag, std::integral_constant<int, 3>{}); break;
      default: launch(tag, std::integral_constant<int, 4>{}); break;
    }
  };
  if (d.precision == ROSSBI_FP32_PERT) by_species(float{});
  else by_species(double{});
  CK(cudaGetLastError());
  indirect_reduce_kernel<<<1, RED_NT, 0, g->stream>>>(part, IND_BLOCKS, d.nth, g->dg.x_ind, g->d_ind + L.cs,
                                                      g->d_ind, g->d_ind + L.g,
                                                      reinterpret_cast<float*>(g->d_ind + L.gf));
  CK(cudaGetLastError());
  return ROSSBI_OK;
}

rossbi_status finish_step(rossbi_grid* g, int nxt, double* next_dt) {
  g->dt_slot = nxt;
  g->dt_on_device = true;
  return next_dt ? read_dt(g, nxt, next_dt) : ROSSBI_OK;
}

// The arguments of stage `stage2` of a step from `state` in place with E* in
// sc: stage 1 E* = E^n + dt/2 (G(E^n) - R0)/V, stage 2 E^{n+1} = E^n +
// dt (G(E*) - R0)/V with the CFL rate fused, each followed by the drag.
template <class T, class Args>
void set_stage(rossbi_grid* g, Args& a, void* const* state, void* const* sc, double dt, bool stage2) {
  a.dt_host = dt;
  a.rate_in = dt == 0.0 ? g->d_dt + g->dt_slot : nullptr;
  a.rate_out = g->d_dt + (1 - g->dt_slot);
  for (int f = 0; f < g->nf; ++f) {
    a.in[f] = (const T*)(stage2 ? sc[f] : state[f]);
    a.base[f] = (const T*)state[f];
    a.out[f] = (T*)(stage2 ? state[f] : sc[f]);
  }
  a.tau_frac = stage2 ? 1.0 : 0.5;
  a.stage2 = stage2;
}

// Host copies of a step on host buffers.
struct HostState {
  void* const* host;
  void* const* dev;
};

// The two stages of one step (Sect. 2.5); with the indirect gravity on, the
// disc moments of each stage's input are summed before it.  Allocates nothing.
template <class Args>
rossbi_status run_stages(rossbi_grid* g, const Args& a1, const Args& a2, void* const* state, void* const* sc) {
  const bool ind = g->dg.x_ind != 0.0;
  rossbi_status st = ind ? indirect_moments(g, state) : ROSSBI_OK;
  if (st == ROSSBI_OK) st = launch_stage(g, a1, n_tiles(g));
  if (st == ROSSBI_OK && ind) st = indirect_moments(g, sc);
  if (st == ROSSBI_OK) st = launch_stage(g, a2, n_tiles(g));
  return st;
}

// Slabs of whole tile layers along z that a host step is cut into: at most 8,
// each of at least four tiles per SM (fewer leave the last wave of every launch
// too empty): 192 x 384 x 48 bi-fluid cells in float take six slabs, and 1.40 ms
// where one piece took 2.04.  One where the layers depend on one another otherwise (periodic
// in z, the moments of the indirect gravity) or launches are timed, and where
// the host buffers are pageable: their copies hold the calling thread, so that
// nothing overlaps and the more of them take longer (3.59 ms of that grid in six
// slabs, 2.26 in one).
int host_slabs(const rossbi_grid* g, void* const* host) {
  if (g->desc.bc_lo[2] == ROSSBI_BC_PERIODIC || g->dg.x_ind != 0.0 || g->profiling) return 1;
  const int slabs = std::max(1, std::min({8, g->tiles_z, n_tiles(g) / (4 * g->sms)}));
  for (int f = 0; slabs > 1 && f < g->nf; ++f) {
    cudaPointerAttributes at{};
    if (cudaPointerGetAttributes(&at, host[f]) != cudaSuccess || at.type != cudaMemoryTypeHost) {
      cudaGetLastError();
      return 1;
    }
  }
  return slabs;
}

rossbi_status ensure_host_streams(rossbi_grid* g) {
  if (g->s_in) return ROSSBI_OK;
  for (cudaEvent_t& e : g->host_ev) CK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
  CK(cudaStreamCreateWithFlags(&g->s_out, cudaStreamNonBlocking));
  CK(cudaStreamCreateWithFlags(&g->s_in, cudaStreamNonBlocking));
  return ROSSBI_OK;
}

// The same in slabs along z, each copied in, stepped and copied out on three
// streams, so that the two directions of the link and the kernels work at the
// same time (one after the other the copies of a 127 MB state took 1.3 of 2.0
// ms).  Stage 1 of a slab waits for the next slab's planes (its halo), stage 2
// of a slab follows stage 1 of the next one, which is also the last to read E^n
// of this slab.
template <class Args>
rossbi_status run_slabs(rossbi_grid* g, const Args& a1, const Args& a2, const HostState& h, int slabs) {
  const int tz = g->tile_tz, nz = g->desc.nz;
  const size_t plane = (size_t)g->desc.nr * g->desc.nth * elem_size(g);
  auto layer = [&](int s) { return (int)((long)g->tiles_z * s / slabs); };
  auto copy = [&](int s, bool in) -> rossbi_status {
    const size_t k0 = (size_t)layer(s) * tz, k1 = std::min<size_t>((size_t)layer(s + 1) * tz, nz);
    for (int f = 0; f < g->nf; ++f) {
      char* d = (char*)h.dev[f] + k0 * plane;
      char* c = (char*)h.host[f] + k0 * plane;
      CK(in ? cudaMemcpyAsync(d, c, (k1 - k0) * plane, cudaMemcpyHostToDevice, g->s_in)
            : cudaMemcpyAsync(c, d, (k1 - k0) * plane, cudaMemcpyDeviceToHost, g->s_out));
    }
    return ROSSBI_OK;
  };
  auto stage = [&](Args a, int s) -> rossbi_status {
    const int layers = layer(s + 1) - layer(s);
    a.order.z = fast_div(layers);
    a.order.k_first = layer(s) * tz;
    if (!a.stage2 && s > 0) a.rate_out = nullptr;  // cleared once
    return launch_stage(g, a, g->tiles_r * g->tiles_t * layers);
  };
  auto finish = [&](int s) -> rossbi_status {  // stage 2 of a slab and its way home
    rossbi_status st = stage(a2, s);
    if (st != ROSSBI_OK) return st;
    CK(cudaEventRecord(g->host_ev[8 + s], g->stream));
    CK(cudaStreamWaitEvent(g->s_out, g->host_ev[8 + s], 0));
    return copy(s, false);
  };
  CK(cudaEventRecord(g->host_ev[16], g->stream));  // after what the caller's stream holds
  CK(cudaStreamWaitEvent(g->s_in, g->host_ev[16], 0));
  rossbi_status st = ROSSBI_OK;
  for (int s = 0; s < slabs && st == ROSSBI_OK; ++s) {
    st = copy(s, true);
    if (st == ROSSBI_OK) CK(cudaEventRecord(g->host_ev[s], g->s_in));
  }
  for (int s = 0; s < slabs && st == ROSSBI_OK; ++s) {
    CK(cudaStreamWaitEvent(g->stream, g->host_ev[std::min(s + 1, slabs - 1)], 0));
    st = stage(a1, s);
    if (st == ROSSBI_OK && s > 0) st = finish(s - 1);
  }
  if (st == ROSSBI_OK) st = finish(slabs - 1);
  return st;
}

// One step of the grid's form; h: the state's host copies, to be read before
// and written after it, or null.
rossbi_status step_form(rossbi_grid* g, void* const* state, void* const* sc, double dt, const DragArgs& drag,
                        double* next_dt, const HostState* h = nullptr, int slabs = 1) {
  const int nxt = 1 - g->dt_slot;
  auto run = [&](auto a1, auto tag) {
    using T = decltype(tag);
    auto a2 = a1;
    set_stage<T>(g, a1, state, sc, dt, false);
    set_stage<T>(g, a2, state, sc, dt, true);
    return h ? run_slabs(g, a1, a2, *h, slabs) : run_stages(g, a1, a2, state, sc);
  };
  auto pert = [&](auto tag) {
    PertArgs<decltype(tag)> a = pert_args<decltype(tag)>(g);
    set_pert_drag(a, drag);
    return run(a, tag);
  };
  rossbi_status st;
  if (g->desc.precision == ROSSBI_FP64) {
    StageArgs a = base_args(g);
    a.drag = drag;
    st = run(a, double{});
  } else if (g->desc.precision == ROSSBI_FP32_PERT) {
    st = pert(float{});
  } else {
    st = pert(double{});
  }
  return st == ROSSBI_OK ? finish_step(g, nxt, next_dt) : st;
}

// ---------------------------------------------------------------- adjoint
rossbi_status launch_adj_flux3(rossbi_grid* g, const AdjFluxArgs& a) {
  for (int axis = 0; axis < 3; ++axis) CK(run_adj_flux(a, axis, g->stream));
  return ROSSBI_OK;
}

template <int NF>
rossbi_status adjoint_reverse(rossbi_grid* g, void* const* state, double dt, const DragArgs& drag,
                              const void* const* lam_np1, void* const* lam_n, double* const* Y1, double* const* Es,
                              double* const* Y2, double* const* Mu, double* const* LamS) {
  const int nb = g->adj_blocks;
  AdjPointArgs p;
  std::memset(&p, 0, sizeof(p));
  p.g = g->dg;
  p.drag = drag;
  AdjFluxArgs fa;
  std::memset(&fa, 0, sizeof(fa));
  fa.g = g->dg;
  fa.status = g->d_status;
  // stage 2: E^{n+1} = D(Y2), Y2 = E^n + dt (G(E*) - R0) / V
  for (int f = 0; f < NF; ++f) {
    p.Y[f] = Y2[f];
    p.lout[f] = (const double*)lam_np1[f];
    p.Ein[f] = Es[f];
    p.M[f] = Mu[f];
    p.lam_n[f] = (double*)lam_n[f];
    p.lam_in[f] = LamS[f];
    fa.E[f] = Es[f];
    fa.M[f] = Mu[f];
    fa.lam[f] = LamS[f];
  }
  p.tau = dt;
  p.stage2 = 1;
  p.partials = g->d_adj_part;
  // indirect gravity: the stage's gradient tables (stage 2: those of E*, left
  // in the grid's tables by the recompute; stage 1: the saved copy), block
  // partials of dJ/dA, dJ/dB, their reduction, and the broadcast through the
  // moments into the cotangent of the stage input
  const bool ind = g->dg.x_ind != 0.0;
  const IndLayout L = ind_layout(g->desc);
  double* ind_part = g->d_adj_ind;
  double* ind_dab = g->d_adj_ind + 4 * (size_t)nb;
  const double* ind_g1 = g->d_adj_ind + 4 * (size_t)nb + 4;
  p.ind_partials = ind_part;
  adj_point_kernel<NF><<<nb, ADJ_PT_NT, 0, g->stream>>>(p);
  CK(cudaGetLastError());
  if (ind) {
    reduce_partials_kernel<<<2, RED_NT, 0, g->stream>>>(ind_part, nb, ind_dab);
    CK(cudaGetLastError());
    adj_indirect_bcast_kernel<<<nb, ADJ_PT_NT, 0, g->stream>>>(g->dg, g->d_ind + L.w, ind_dab, LamS[RHO],
                                                                NF == 9 ? LamS[DRHO] : nullptr);
    CK(cudaGetLastError());
  }
  rossbi_status st = launch_adj_flux3(g, fa);
  if (st != ROSSBI_OK) return st;
  // stage 1: E* = D(Y1), Y1 = E^n + dt/2 (G(E^n) - R0) / V
  for (int f = 0; f < NF; ++f) {
    p.Y[f] = Y1[f];
    p.lout[f] = LamS[f];
    p.Ein[f] = (const double*)state[f];
    fa.E[f] = (const double*)state[f];
    fa.lam[f] = (double*)lam_n[f];
  }
  p.tau = 0.5 * dt;
  p.stage2 = 0;
  p.partials = g->d_adj_part + nb;
  if (ind) {
    p.g.ind_g = ind_g1;
    p.ind_partials = ind_part + 2 * (size_t)nb;
  }
  adj_point_kernel<NF><<<nb, ADJ_PT_NT, 0, g->stream>>>(p);
  CK(cudaGetLastError());
  if (ind) {
    reduce_partials_kernel<<<2, RED_NT, 0, g->stream>>>(ind_part + 2 * (size_t)nb, nb, ind_dab + 2);
    CK(cudaGetLastError());
    adj_indirect_bcast_kernel<<<nb, ADJ_PT_NT, 0, g->stream>>>(g->dg, g->d_ind + L.w, ind_dab + 2,
                                                                (double*)lam_n[RHO],
                                                                NF == 9 ? (double*)lam_n[DRHO] : nullptr);
    CK(cudaGetLastError());
  }
  st = launch_adj_flux3(g, fa);
  if (st != ROSSBI_OK) return st;
  adj_dst_reduce_kernel<<<1, 512, 0, g->stream>>>(g->d_adj_part, 2 * nb, g->d_adj_slots);
  CK(cudaGetLastError());
  return ROSSBI_OK;
}

rossbi_status adjoint_step(rossbi_grid* g, void* const* state, double dt, const rossbi_dust_params* dust,
                           const void* const* lam_np1, void* const* lam_n, double* dparam) {
  if (!g->eq_set || !state || !lam_np1 || !lam_n) return ROSSBI_ERR_ARG;
  if (g->desc.precision != ROSSBI_FP64) return ROSSBI_ERR_UNSUPPORTED;
  if (!(dt > 0.0) || !std::isfinite(dt)) return ROSSBI_ERR_ARG;
  for (int f = 0; f < g->nf; ++f) {
    if (!state[f] || !lam_np1[f] || !lam_n[f]) return ROSSBI_ERR_ARG;
    for (int h = 0; h < g->nf; ++h)  // the cotangents must not overwrite E^n (lam_n may be lam_np1)
      if (lam_np1[f] == state[h] || lam_n[f] == state[h]) return ROSSBI_ERR_ARG;
  }
  if (g->nf > 9) return ROSSBI_ERR_UNSUPPORTED;  // the adjoint carries one dust species
  if (g->nf == 9 && !dust) return ROSSBI_ERR_ARG;
  DragArgs drag;
  rossbi_status st = drag_args(g, dust, drag);
  if (st != ROSSBI_OK) return st;
  const size_t nfc = (size_t)g->nf * g->ncell;
  if (!g->d_adj) {
    // all three buffers or none, so that a failed allocation leaves no half state
    const int nb = (int)std::min<size_t>((g->ncell + ADJ_PT_NT - 1) / ADJ_PT_NT, 2048);
    double *adj = nullptr, *part = nullptr, *slots = nullptr;
    cudaError_t e = cudaMalloc(&adj, 5 * nfc * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&part, 2 * (size_t)nb * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&slots, 2 * sizeof(double));
    if (e == cudaSuccess) e = cudaMemsetAsync(slots, 0, 2 * sizeof(double), g->stream);
    if (e != cudaSuccess) {
      cudaFree(adj);
      cudaFree(part);
      cudaFree(slots);
      return e == cudaErrorMemoryAllocation ? ROSSBI_ERR_OOM : ROSSBI_ERR_CUDA;
    }
    g->d_adj = adj;
    g->d_adj_part = part;
    g->d_adj_slots = slots;
    g->adj_blocks = nb;
  }
  const bool ind = g->dg.x_ind != 0.0;
  if (ind && !g->d_adj_ind) {
    const size_t n = 4 * (size_t)g->adj_blocks + 4 + 2 * (size_t)g->desc.nth;
    CK(cudaMalloc(&g->d_adj_ind, n * sizeof(double)));
  }
  double *Y1[9], *Es[9], *Y2[9], *Mu[9], *LamS[9];
  for (int f = 0; f < g->nf; ++f) {
    Y1[f] = g->d_adj + f * g->ncell;
    Es[f] = g->d_adj + nfc + f * g->ncell;
    Y2[f] = g->d_adj + 2 * nfc + f * g->ncell;
    Mu[f] = g->d_adj + 3 * nfc + f * g->ncell;
    LamS[f] = g->d_adj + 4 * nfc + f * g->ncell;
  }
  // forward recompute from E^n: the stage kernels with the drag switched off
  // (1 / t_s = 0 makes apply_drag the identity) give the pre-drag states
  const int nblocks = n_tiles(g);
  StageArgs a = base_args(g);
  a.drag = drag;
  for (int sp = 0; sp < ND_MAX; ++sp) a.drag.ist[sp] = a.drag.irr[sp] = 0.0;
  a.dt_host = dt;
  for (int f = 0; f < g->nf; ++f) {
    a.in[f] = (const double*)state[f];
    a.base[f] = (const double*)state[f];
    a.out[f] = Y1[f];
  }
  a.tau_frac = 0.5;
  if (ind) {  // the moments of E^n; stage 1's gradient table is kept for the reverse sweep
    st = indirect_moments(g, state);
    if (st != ROSSBI_OK) return st;
    const IndLayout L = ind_layout(g->desc);
    CK(cudaMemcpyAsync(g->d_adj_ind + 4 * (size_t)g->adj_blocks + 4, g->d_ind + L.g,
                       2 * (size_t)g->desc.nth * sizeof(double), cudaMemcpyDeviceToDevice, g->stream));
  }
  st = launch_stage(g, a, nblocks);
  if (st != ROSSBI_OK) return st;
  double* const* Estar = Y1;
  if (g->nf == 9) {
    Fields9 y, o;
    for (int f = 0; f < 9; ++f) {
      y.p[f] = Y1[f];
      o.p[f] = Es[f];
    }
    drag_only_kernel<<<g->adj_blocks, ADJ_PT_NT, 0, g->stream>>>(g->dg, y, o, 0.5 * dt, drag);
    CK(cudaGetLastError());
    Estar = Es;
  }
  for (int f = 0; f < g->nf; ++f) {
    a.in[f] = Estar[f];
    a.base[f] = (const double*)state[f];
    a.out[f] = Y2[f];
  }
  a.tau_frac = 1.0;
  if (ind && (st = indirect_moments(g, (void* const*)Estar)) != ROSSBI_OK) return st;
  st = launch_stage(g, a, nblocks);
  if (st != ROSSBI_OK) return st;
  st = g->nf == 9 ? adjoint_reverse<9>(g, state, dt, drag, lam_np1, lam_n, Y1, Estar, Y2, Mu, LamS)
                  : adjoint_reverse<5>(g, state, dt, drag, lam_np1, lam_n, Y1, Estar, Y2, Mu, LamS);
  if (st != ROSSBI_OK) return st;
  if (dparam) {
    CK(cudaMemcpyAsync(g->h_pinned, g->d_adj_slots, sizeof(double), cudaMemcpyDeviceToHost, g->stream));
    st = sync_and_status(g);
    *dparam += g->h_pinned[0];
    return st;
  }
  return ROSSBI_OK;
}

rossbi_status step_device(rossbi_grid* g, void* const* state, void* const* scratch, double dt,
                          const rossbi_dust_params* dust, double* next_dt) {
  void* sc[NF_MAX];
  DragArgs drag;
  rossbi_status st = prepare_step(g, state, scratch, dt, dust, sc, drag);
  if (st != ROSSBI_OK) return st;
  return step_form(g, state, sc, dt, drag, next_dt);
}

}  // namespace

namespace {
// Eight independent FMA chains per thread; the result is stored so that
// nothing is eliminated.
template <class T>
__global__ void fma_peak_kernel(T* out, int iters) {
  T a[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) a[c] = T(threadIdx.x + c) * T(1e-7);
  const T m = T(0.9999999), k = T(1e-9);
  for (int i = 0; i < iters; ++i) {
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      if constexpr (sizeof(T) == 4) a[c] = fmaf(a[c], m, k);
      else a[c] = fma(a[c], m, k);
    }
  }
  T s = T(0);
#pragma unroll
  for (int c = 0; c < 8; ++c) s += a[c];
  out[(size_t)blockIdx.x * blockDim.x + threadIdx.x] = s;
}

template <class T>
rossbi_status fma_peak(cudaStream_t st, int iters, double* flops) {
  int dev = 0, sms = 0;
  CK(cudaGetDevice(&dev));
  CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int blocks = 8 * sms, threads = 256;
  T* out = nullptr;
  if (cudaMalloc(&out, (size_t)blocks * threads * sizeof(T)) != cudaSuccess) return ROSSBI_ERR_OOM;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  rossbi_status r = ROSSBI_OK;
  float ms = 0.0f;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) r = ROSSBI_ERR_CUDA;
  if (r == ROSSBI_OK) {
    fma_peak_kernel<T><<<blocks, threads, 0, st>>>(out, iters);  // warm-up
    cudaEventRecord(e0, st);
    fma_peak_kernel<T><<<blocks, threads, 0, st>>>(out, iters);
    cudaEventRecord(e1, st);
    if (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess ||
        cudaGetLastError() != cudaSuccess)
      r = ROSSBI_ERR_CUDA;
  }
  if (r == ROSSBI_OK) *flops = 2.0 * 8.0 * iters * (double)blocks * threads / (ms * 1e-3);
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  cudaFree(out);
  return r;
}
}  // namespace

extern "C" {

const char* rossbi_status_string(rossbi_status s) {
  switch (s) {
    case ROSSBI_OK: return "ok";
    case ROSSBI_ERR_ARG: return "invalid argument";
    case ROSSBI_ERR_CUDA: return "CUDA error";
    case ROSSBI_ERR_OOM: return "out of device memory";
    case ROSSBI_ERR_NONPHYSICAL: return "non-physical state (rho <= 0, P <= 0 or NaN)";
    case ROSSBI_ERR_RIEMANN: return "Riemann solver did not converge";
    case ROSSBI_ERR_UNSUPPORTED: return "unsupported configuration";
  }
  return "unknown status";
}

int rossbi_nfields(const rossbi_grid* g) { return g ? g->nf : 0; }
int rossbi_precision(const rossbi_grid* g) { return g ? g->desc.precision : -1; }

void rossbi_destroy(rossbi_grid* g) {
  if (!g) return;
  double* tabs[] = {g->d_rcoef, g->d_rslope, g->d_vol, g->d_ivol, g->d_area_r, g->d_area_t,
                    g->d_area_z, g->d_aov, g->d_ir, g->d_omk, g->d_grav, g->d_e0c, g->d_e0r, g->d_e0z, g->d_r0, g->d_partials, g->d_sums};
  for (double* p : tabs)
    if (p) cudaFree(p);
  if (g->d_dt) cudaFree(g->d_dt);
  if (g->d_status) cudaFree(g->d_status);
  if (g->d_scratch) cudaFree(g->d_scratch);
  if (g->d_hoststate) cudaFree(g->d_hoststate);
  if (g->d_ptab) cudaFree(g->d_ptab);
  if (g->d_fallbacks) cudaFree(g->d_fallbacks);
  if (g->d_w0) cudaFree(g->d_w0);
  if (g->d_adj) cudaFree(g->d_adj);
  if (g->d_adj_part) cudaFree(g->d_adj_part);
  if (g->d_adj_slots) cudaFree(g->d_adj_slots);
  if (g->d_ind) cudaFree(g->d_ind);
  if (g->d_adj_ind) cudaFree(g->d_adj_ind);
  if (g->d_damp) cudaFree(g->d_damp);
  if (g->h_pinned) cudaFreeHost(g->h_pinned);
  for (cudaEvent_t e : g->ev) cudaEventDestroy(e);
  for (cudaEvent_t e : g->host_ev)
    if (e) cudaEventDestroy(e);
  if (g->s_in) cudaStreamDestroy(g->s_in);
  if (g->s_out) cudaStreamDestroy(g->s_out);
  delete g;
}

rossbi_status rossbi_init_grid(const rossbi_grid_desc* desc, void* cuda_stream, rossbi_grid** out) {
  if (!desc || !out) return ROSSBI_ERR_ARG;
  *out = nullptr;
  const rossbi_status chk = check_desc(*desc);
  if (chk != ROSSBI_OK) return chk;
  rossbi_grid* g = new (std::nothrow) rossbi_grid();
  if (!g) return ROSSBI_ERR_OOM;
  g->desc = *desc;
  g->stream = (cudaStream_t)cuda_stream;
  if (cudaGetDevice(&g->device) != cudaSuccess ||
      cudaDeviceGetAttribute(&g->sms, cudaDevAttrMultiProcessorCount, g->device) != cudaSuccess) {
    delete g;
    return ROSSBI_ERR_CUDA;
  }
  g->nf = 5 + 4 * desc->n_dust;
  g->ncell = (size_t)desc->nr * desc->nth * desc->nz;
  // the tile of the form's stage kernel
  auto set_tiles = [&](int tr, int tt, int tz) {
    g->tile_tt = tt;
    g->tile_tz = tz;
    g->tiles_r = (desc->nr + tr - 1) / tr;
    g->tiles_t = (desc->nth + tt - 1) / tt;
    g->tiles_z = (desc->nz + tz - 1) / tz;
  };
  if (desc->precision == ROSSBI_FP32_PERT) {
    set_tiles(P32_TR, P32_TT, P32_TZ);
  } else {
    const bool flat = desc->precision == ROSSBI_FP64 && flat_grid(desc->nz, desc->bc_lo[2], desc->bc_hi[2], g->nf);
    g->tile = choose_tile(desc->nr, desc->nth, desc->nz, flat, g->nf, g->sms);
    by_tile(g->tile, [&](auto t) {
      using T = decltype(t);
      set_tiles(T::TR, T::TT, T::TZ);
      return 0;
    });
  }
  const rossbi_grid_desc& d = *desc;
  const int nr = d.nr;
  const double dy = (d.x1[1] - d.x0[1]) / d.nth;
  const double dz = (d.x1[2] - d.x0[2]) / d.nz;
  constexpr int GH = 2;  // ghosts of the axis-0 coordinates
  std::vector<double> rc(nr + 2 * GH), rf(nr + 2 * GH + 1), rcoef((size_t)(nr + 2) * RCW, 0.0), rslope((size_t)(nr + 2) * 9);
  for (int i = -GH; i < nr + GH; ++i) rc[i + GH] = axis0_centre(d, i);
  for (int i = -GH; i <= nr + GH; ++i) rf[i + GH] = axis0_face(d, i);
  for (int i = -1; i <= nr; ++i) {  // parabola weights (Sect. 2.7)
    const double xm = rc[i - 1 + GH], x0 = rc[i + GH], xp = rc[i + 1 + GH];
    const double fm = rf[i + GH], fp = rf[i + 1 + GH];
    double* w = &rcoef[(size_t)(i + 1) * RCW];
    // The parabola through the three centres at the face distances hm, hp from
    // x0, in the differences dm = e0 - em, dp = ep - e0:
    // q(x0 - hm) = e0 - (w2 dm + w3 dp), q(x0 + hp) = e0 + (w4 dm + w5 dp)
    const double hm = x0 - fm, hp = fp - x0, dl = x0 - xm, dr = xp - x0, dx = xp - xm;
    const double lo = std::min(2.0 * hm, dl), up = std::min(2.0 * hp, dr);  // limiter reaches
    w[0] = lo / dl;  // lower limit min(w0 dm, w1 dp), upper limit w6 times that
    w[1] = lo / dr;
    w[2] = hm * (dr + hm) / (dl * dx);
    w[3] = hm * (dl - hm) / (dr * dx);
    w[4] = hp * (dr - hp) / (dl * dx);
    w[5] = hp * (dl + hp) / (dr * dx);
    w[6] = up / lo;
    double* v = &rslope[(size_t)(i + 1) * 9];
    v[0] = 1.0 / (x0 - xm);
    v[1] = 1.0 / (xp - x0);
    v[2] = 1.0 / (xp - xm);
    v[3] = x0 - xm;
    v[4] = xp - x0;
    v[5] = fm - x0;
    v[6] = fp - x0;
    v[7] = -std::min(2.0 * (x0 - fm), x0 - xm);
    v[8] = std::min(2.0 * (fp - x0), xp - x0);
  }
  std::vector<double> vol(nr), ivol(nr), ar(nr + 1), at(nr), az(nr), maxA(nr);
  if (d.geometry == ROSSBI_GEOM_CYL) {  // Sect. 2.2 finite volumes of the cylindrical mesh
    for (int i = 0; i <= nr; ++i) ar[i] = rf[i + GH] * dy * dz;
    for (int i = 0; i < nr; ++i) {
      const double rm = rf[i + GH], rp = rf[i + 1 + GH];
      vol[i] = 0.5 * (rp * rp - rm * rm) * dy * dz;
      at[i] = (rp - rm) * dz;
      az[i] = 0.5 * (rp * rp - rm * rm) * dy;
      maxA[i] = std::max(ar[i + 1], std::max(at[i], az[i]));
    }
  } else {
    const double dx = (d.x1[0] - d.x0[0]) / nr;
    for (int i = 0; i <= nr; ++i) ar[i] = dy * dz;
    for (int i = 0; i < nr; ++i) {
      vol[i] = dx * dy * dz;
      at[i] = dx * dz;
      az[i] = dx * dy;
      maxA[i] = std::max(ar[i], std::max(at[i], az[i]));
    }
  }
  std::vector<double> ir(nr, 0.0), omk(nr, 1.0), grav((size_t)2 * d.nz * nr, 0.0);
  for (int i = 0; i < nr; ++i) {
    ivol[i] = 1.0 / vol[i];
    maxA[i] /= vol[i];
    if (d.geometry != ROSSBI_GEOM_CYL) continue;
    const double r = rc[i + GH];
    ir[i] = 1.0 / r;
    omk[i] = std::sqrt(d.gm / (r * r * r));
    for (int k = 0; k < d.nz; ++k) {  // stellar gravity and the frame's centrifugal term at the cell centres
      const double z = d.x0[2] + (k + 0.5) * dz, R2 = r * r + z * z, R3 = R2 * std::sqrt(R2);
      grav[(size_t)k * nr + i] = -d.gm * r / R3 + d.omega_frame * d.omega_frame * r;
      grav[(size_t)(d.nz + k) * nr + i] = -d.gm * z / R3;
    }
  }
  rossbi_status st = ROSSBI_OK;
  do {
    if ((st = upload(&g->d_rcoef, rcoef, g->stream)) != ROSSBI_OK) break;
    if ((st = upload(&g->d_rslope, rslope, g->stream)) != ROSSBI_OK) break;
    if ((st = upload(&g->d_vol, vol, g->stream)) != ROSSBI_OK) break;
    if ((st = upload(&g->d_ivol, ivol, g->stream)) != ROSSBI_OK) break;
    if ((st = upload(&g->d_area_r, ar, g->stream)) != ROSSBI_OK) break;
    if ((st = upload(&g->d_area_t, at, g->stream)) != ROSSBI_OK) break;
    if ((st = upload(&g->d_area_z, az, g->stream)) != ROSSBI_OK) break;
    if ((st = upload(&g->d_aov, maxA, g->stream)) != ROSSBI_OK) break;
    if ((st = upload(&g->d_ir, ir, g->stream)) != ROSSBI_OK) break;
    if ((st = upload(&g->d_omk, omk, g->stream)) != ROSSBI_OK) break;
    if ((st = upload(&g->d_grav, grav, g->stream)) != ROSSBI_OK) break;
    if (cudaMalloc(&g->d_dt, 2 * sizeof(unsigned long long)) != cudaSuccess) { st = ROSSBI_ERR_OOM; break; }
    if (cudaMalloc(&g->d_sums, NF_MAX * sizeof(double)) != cudaSuccess) { st = ROSSBI_ERR_OOM; break; }
    if (cudaMalloc(&g->d_status, sizeof(unsigned)) != cudaSuccess) { st = ROSSBI_ERR_OOM; break; }
    if (cudaMemsetAsync(g->d_status, 0, sizeof(unsigned), g->stream) != cudaSuccess) { st = ROSSBI_ERR_CUDA; break; }
    if (cudaMallocHost(&g->h_pinned, 32 * sizeof(double)) != cudaSuccess) { st = ROSSBI_ERR_OOM; break; }
    if (cudaStreamSynchronize(g->stream) != cudaSuccess) { st = ROSSBI_ERR_CUDA; break; }
  } while (false);
  if (st != ROSSBI_OK) {
    rossbi_destroy(g);
    return st;
  }
  DevGrid& dg = g->dg;
  dg.geom = d.geometry;
  dg.nr = d.nr;
  dg.nth = d.nth;
  dg.nz = d.nz;
  dg.nf = g->nf;
  dg.has_eq = 0;
  dg.recon = d.recon == ROSSBI_RECON_PRIMITIVE ? RECON_PRIM : RECON_CONS;
  for (int sp = 0; sp < ND_MAX; ++sp) dg.st_factor[sp] = 1.0;
  for (int a = 0; a < 3; ++a) {
    dg.bc_lo[a] = d.bc_lo[a];
    dg.bc_hi[a] = d.bc_hi[a];
    dg.dx[a] = (d.x1[a] - d.x0[a]) / (a == 0 ? d.nr : (a == 1 ? d.nth : d.nz));
  }
  dg.gamma = d.gamma;
  dg.gm = d.gm;
  dg.omega = d.geometry == ROSSBI_GEOM_CYL ? d.omega_frame : 0.0;
  dg.cfl = d.cfl;
  dg.rcoef = g->d_rcoef;
  dg.rslope = g->d_rslope;
  dg.vol = g->d_vol;
  dg.ivol = g->d_ivol;
  dg.area_r = g->d_area_r;
  dg.area_t = g->d_area_t;
  dg.area_z = g->d_area_z;
  dg.aov = g->d_aov;
  dg.ir = g->d_ir;
  dg.omk = g->d_omk;
  dg.grav = g->d_grav;
  dg.near = near_coef(d.gamma);
  *out = g;
  return ROSSBI_OK;
}

rossbi_status rossbi_set_equilibrium(rossbi_grid* g, const rossbi_disc_params* disc) {
  if (!g) return ROSSBI_ERR_ARG;
  const rossbi_grid_desc& d = g->desc;
  // a cylindrical grid without a disc (E0 = 0, e.g. the explosion test of
  // Sect. 4.1) runs in the FP64 form; the perturbation forms' source
  // coefficients are tabulated from a disc equilibrium
  if (d.geometry == ROSSBI_GEOM_CYL && !disc && d.precision != ROSSBI_FP64) return ROSSBI_ERR_UNSUPPORTED;
  if (d.geometry == ROSSBI_GEOM_CYL && disc && !(d.gm > 0.0)) return ROSSBI_ERR_ARG;  // Keplerian disc
  if (disc && disc->bump_delta != 0.0 &&
      (!(disc->bump_delta > -1.0) || !(disc->bump_width > 0.0) || !std::isfinite(disc->bump_delta) ||
       !std::isfinite(disc->bump_width) || !std::isfinite(disc->bump_r0)))
    return ROSSBI_ERR_ARG;
  g->eq_set = false;
  g->dg.has_eq = 0;
  g->dg.e0c = g->dg.e0r = g->dg.e0z = g->dg.r0 = nullptr;
  g->dg.w0c = g->dg.w0r = g->dg.w0z = nullptr;
  g->has_disc = disc != nullptr;
  if (!disc) {
    g->h_e0c.assign((size_t)5 * d.nz * d.nr, 0.0);
    rossbi_status st = ROSSBI_OK;
    if (d.precision == ROSSBI_FP32_PERT) st = build_pert_tables<float>(g, g->pt_f);
    else if (d.precision == ROSSBI_FP64_PERT) st = build_pert_tables<double>(g, g->pt_d);
    if (st != ROSSBI_OK) return st;
    g->eq_set = true;
    return ROSSBI_OK;
  }
  g->disc = *disc;
  const int nr = d.nr, nz = d.nz;
  const double dz = (d.x1[2] - d.x0[2]) / nz;
  std::vector<double> e0c((size_t)5 * nz * nr), e0r((size_t)5 * nz * (nr + 1)), e0z((size_t)5 * (nz + 1) * nr);
  for (int k = 0; k < nz; ++k) {
    const double z = d.x0[2] + (k + 0.5) * dz;
    for (int i = 0; i < nr; ++i)
      equilibrium_cons(d, *disc, axis0_centre(d, i), z, &e0c[(size_t)k * nr + i], (size_t)nz * nr);
    for (int i = 0; i <= nr; ++i)
      equilibrium_cons(d, *disc, axis0_face(d, i), z, &e0r[(size_t)k * (nr + 1) + i], (size_t)nz * (nr + 1));
  }
  for (int k = 0; k <= nz; ++k) {
    const double z = d.x0[2] + k * dz;
    for (int i = 0; i < nr; ++i)
      equilibrium_cons(d, *disc, axis0_centre(d, i), z, &e0z[(size_t)k * nr + i], (size_t)(nz + 1) * nr);
  }
  for (double v : e0c)
    if (!std::isfinite(v)) return ROSSBI_ERR_ARG;
  rossbi_status st;
  if ((st = upload(&g->d_e0c, e0c, g->stream)) != ROSSBI_OK) return st;
  if ((st = upload(&g->d_e0r, e0r, g->stream)) != ROSSBI_OK) return st;
  if ((st = upload(&g->d_e0z, e0z, g->stream)) != ROSSBI_OK) return st;
  g->h_e0c = e0c;
  g->dg.has_eq = 1;
  g->dg.e0c = g->d_e0c;
  g->dg.e0r = g->d_e0r;
  g->dg.e0z = g->d_e0z;
  {
    const size_t nc = (size_t)nz * nr, nrf = (size_t)nz * (nr + 1), nzf = (size_t)(nz + 1) * nr;
    if (g->d_w0) cudaFree(g->d_w0);
    g->d_w0 = nullptr;
    CK(cudaMalloc(&g->d_w0, 5 * (nc + nrf + nzf) * sizeof(double)));
    eq_prim_kernel<<<64, 256, 0, g->stream>>>(d.gamma, g->d_e0c, g->d_w0, nc);
    eq_prim_kernel<<<64, 256, 0, g->stream>>>(d.gamma, g->d_e0r, g->d_w0 + 5 * nc, nrf);
    eq_prim_kernel<<<64, 256, 0, g->stream>>>(d.gamma, g->d_e0z, g->d_w0 + 5 * (nc + nrf), nzf);
    CK(cudaGetLastError());
    g->dg.w0c = g->d_w0;
    g->dg.w0r = g->d_w0 + 5 * nc;
    g->dg.w0z = g->d_w0 + 5 * (nc + nrf);
  }
  if (d.precision == ROSSBI_FP64) {
    if ((st = empty_run(g)) != ROSSBI_OK) return st;
    g->dg.r0 = g->d_r0;
  } else if (d.precision == ROSSBI_FP32_PERT) {
    if ((st = build_pert_tables<float>(g, g->pt_f)) != ROSSBI_OK) return st;
  } else {
    if ((st = build_pert_tables<double>(g, g->pt_d)) != ROSSBI_OK) return st;
  }
  g->eq_set = true;
  return sync_and_status(g);
}

rossbi_status rossbi_get_equilibrium(rossbi_grid* g, double* host_out) {
  if (!g || !host_out || !g->eq_set) return ROSSBI_ERR_ARG;
  std::memcpy(host_out, g->h_e0c.data(), g->h_e0c.size() * sizeof(double));
  return ROSSBI_OK;
}

rossbi_status rossbi_cfl_dt(rossbi_grid* g, const void* const* state, double* dt_out) {
  if (!g || !state || !dt_out || !g->eq_set) return ROSSBI_ERR_ARG;
  for (int f = 0; f < g->nf; ++f)
    if (!state[f]) return ROSSBI_ERR_ARG;
  unsigned long long* slot = g->d_dt + g->dt_slot;
  CK(cudaMemsetAsync(slot, 0, sizeof(*slot), g->stream));
  const int blocks = (int)std::min<size_t>((g->ncell + CFL_NT - 1) / CFL_NT, 152 * 8);
  const int prec = g->desc.precision;
  if (prec == ROSSBI_FP64) {
    StageArgs a = base_args(g);
    for (int f = 0; f < g->nf; ++f) a.in[f] = (const double*)state[f];
    CK(by_nf(g->nf, [&](auto nf) {
      cfl_kernel<decltype(nf)::value><<<blocks, CFL_NT, 0, g->stream>>>(g->dg, a, slot);
      return cudaGetLastError();
    }));
  } else if (prec == ROSSBI_FP32_PERT) {
    PertArgs<float> a = pert_args<float>(g);
    for (int f = 0; f < g->nf; ++f) a.in[f] = (const float*)state[f];
    CK(by_nf(g->nf, [&](auto nf) {
      pert_cfl_kernel<float, decltype(nf)::value><<<blocks, 256, 0, g->stream>>>(a, slot);
      return cudaGetLastError();
    }));
  } else {
    PertArgs<double> a = pert_args<double>(g);
    for (int f = 0; f < g->nf; ++f) a.in[f] = (const double*)state[f];
    CK(by_nf(g->nf, [&](auto nf) {
      pert_cfl_kernel<double, decltype(nf)::value><<<blocks, 256, 0, g->stream>>>(a, slot);
      return cudaGetLastError();
    }));
  }
  CK(cudaGetLastError());
  g->dt_on_device = true;
  return read_dt(g, g->dt_slot, dt_out);
}

rossbi_status rossbi_step(rossbi_grid* g, void* const* state, void* const* scratch, double dt,
                          const rossbi_dust_params* dust, double* next_dt) {
  if (!g) return ROSSBI_ERR_ARG;
  return step_device(g, state, scratch, dt, dust, next_dt);
}

rossbi_status rossbi_step_host(rossbi_grid* g, void* const* host_state, double dt, const rossbi_dust_params* dust,
                               double* next_dt) {
  if (!g || !host_state) return ROSSBI_ERR_ARG;
  for (int f = 0; f < g->nf; ++f)
    if (!host_state[f]) return ROSSBI_ERR_ARG;
  rossbi_status st = ensure_scratch(g, &g->d_hoststate);
  if (st != ROSSBI_OK) return st;
  const size_t bytes = g->ncell * elem_size(g);
  void* dev[NF_MAX];
  for (int f = 0; f < g->nf; ++f) dev[f] = (char*)g->d_hoststate + (size_t)f * bytes;
  double ndt = 0.0;
  const int slabs = host_slabs(g, host_state);
  if (slabs > 1) {
    void* sc[NF_MAX];
    DragArgs drag;
    st = prepare_step(g, dev, nullptr, dt, dust, sc, drag);
    if (st == ROSSBI_OK) st = ensure_host_streams(g);
    if (st != ROSSBI_OK) return st;
    const HostState h{host_state, dev};
    st = step_form(g, dev, sc, dt, drag, &ndt, &h, slabs);
    // the host buffers are the caller's again, whatever happened
    const cudaError_t e1 = cudaStreamSynchronize(g->s_in), e2 = cudaStreamSynchronize(g->s_out);
    CK(e1);
    CK(e2);
    if (next_dt) *next_dt = ndt;
    return st;
  }
  for (int f = 0; f < g->nf; ++f)
    CK(cudaMemcpyAsync(dev[f], host_state[f], bytes, cudaMemcpyHostToDevice, g->stream));
  st = step_device(g, dev, nullptr, dt, dust, &ndt);
  for (int f = 0; f < g->nf; ++f)
    CK(cudaMemcpyAsync(host_state[f], dev[f], bytes, cudaMemcpyDeviceToHost, g->stream));
  CK(cudaStreamSynchronize(g->stream));
  if (next_dt) *next_dt = ndt;
  return st;
}

rossbi_status rossbi_conservation_sums(rossbi_grid* g, const void* const* state, double* sums) {
  if (!g || !state || !sums || !g->eq_set) return ROSSBI_ERR_ARG;
  for (int f = 0; f < g->nf; ++f)
    if (!state[f]) return ROSSBI_ERR_ARG;
  const int blocks = (int)std::min<size_t>((g->ncell + CFL_NT - 1) / CFL_NT, 152 * 8);
  rossbi_status st = ensure_partials(g, blocks);
  if (st != ROSSBI_OK) return st;
  const int prec = g->desc.precision;
  if (prec == ROSSBI_FP64) {
    StageArgs a = base_args(g);
    for (int f = 0; f < g->nf; ++f) a.in[f] = (const double*)state[f];
    sums_kernel<<<blocks, CFL_NT, 0, g->stream>>>(g->dg, a, g->d_partials);
  } else if (prec == ROSSBI_FP32_PERT) {
    PertArgs<float> a = pert_args<float>(g);
    for (int f = 0; f < g->nf; ++f) a.in[f] = (const float*)state[f];
    CK(by_nf(g->nf, [&](auto nf) {
      pert_sums_kernel<float, decltype(nf)::value><<<blocks, 256, 0, g->stream>>>(a, g->d_partials);
      return cudaGetLastError();
    }));
  } else {
    PertArgs<double> a = pert_args<double>(g);
    for (int f = 0; f < g->nf; ++f) a.in[f] = (const double*)state[f];
    CK(by_nf(g->nf, [&](auto nf) {
      pert_sums_kernel<double, decltype(nf)::value><<<blocks, 256, 0, g->stream>>>(a, g->d_partials);
      return cudaGetLastError();
    }));
  }
  CK(cudaGetLastError());
  reduce_partials_kernel<<<g->nf, RED_NT, 0, g->stream>>>(g->d_partials, blocks, g->d_sums);
  CK(cudaGetLastError());
  CK(cudaMemcpyAsync(g->h_pinned, g->d_sums, g->nf * sizeof(double), cudaMemcpyDeviceToHost, g->stream));
  st = sync_and_status(g);
  for (int f = 0; f < g->nf; ++f) sums[f] = g->h_pinned[f];
  if (prec != ROSSBI_FP64)
    for (int f = 0; f < 5; ++f) sums[f] += g->eq_sums[f];
  return st;
}

rossbi_status rossbi_fallback_count(rossbi_grid* g, unsigned long long* count) {
  if (!g || !count) return ROSSBI_ERR_ARG;
  *count = 0;
  if (!g->d_fallbacks) return ROSSBI_OK;
  CK(cudaStreamSynchronize(g->stream));
  CK(cudaMemcpy(count, g->d_fallbacks, sizeof(unsigned long long), cudaMemcpyDeviceToHost));
  return ROSSBI_OK;
}

rossbi_status rossbi_measure_fma_peak(int fp64, void* cuda_stream, double* flops_per_s) {
  if (!flops_per_s) return ROSSBI_ERR_ARG;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  return fp64 ? fma_peak<double>(st, 1 << 13, flops_per_s) : fma_peak<float>(st, 1 << 19, flops_per_s);
}

rossbi_status rossbi_profile_enable(rossbi_grid* g, int enable) {
  if (!g) return ROSSBI_ERR_ARG;
  if (enable && g->ev.empty()) {
    g->ev.resize(2 * PROFILE_PAIRS, nullptr);
    for (auto& e : g->ev) CK(cudaEventCreate(&e));
  }
  g->profiling = enable != 0;
  return ROSSBI_OK;
}

rossbi_status rossbi_profile_read(rossbi_grid* g, double* stage_ms, int* stage_launches) {
  if (!g || !stage_ms || !stage_launches) return ROSSBI_ERR_ARG;
  const rossbi_status st = profile_drain(g);
  if (st != ROSSBI_OK) return st;
  *stage_ms = g->prof_ms;
  *stage_launches = g->prof_launches;
  g->prof_ms = 0.0;
  g->prof_launches = 0;
  return ROSSBI_OK;
}

rossbi_status rossbi_set_indirect(rossbi_grid* g, double x_ref) {
  if (!g || !std::isfinite(x_ref)) return ROSSBI_ERR_ARG;
  if (x_ref != 0.0 && g->desc.geometry != ROSSBI_GEOM_CYL) return ROSSBI_ERR_ARG;
  if (x_ref != 0.0) {
    const rossbi_status st = ensure_ind_tables(g);
    if (st != ROSSBI_OK) return st;
  }
  g->dg.x_ind = x_ref;
  return ROSSBI_OK;
}

}  // extern "C"

namespace {

// The rate table of the damping zones, per cell centre (nz, nr): the radial
// wave-killing zones (a parabola in r, 1 / tau at the boundary, 0 with zero
// slope at the zone edge, tau = f x the orbital period at that boundary)
// plus the vertical damped boundary (the same parabola in |z|, tau = f x the
// orbital period at the cell's radius).  Both off: no table.
rossbi_status build_damping(rossbi_grid* g) {
  const rossbi_grid_desc& d = g->desc;
  g->dg.damp_k = nullptr;
  g->dg.damp_kf = nullptr;
  if (!g->damp_r && !g->damp_z) return ROSSBI_OK;
  const double pi = 3.14159265358979323846;
  const double rin = d.x0[0], rout = d.x1[0], zmax = d.x1[2], dz = (d.x1[2] - d.x0[2]) / d.nz;
  const size_t n = (size_t)d.nz * d.nr;
  std::vector<double> k(n + (n + 1) / 2, 0.0);  // rates, then the same as floats
  const rossbi_damping_params& p = g->damp_rp;
  const double tau_in = p.period_factor * 2.0 * pi / std::sqrt(d.gm / (rin * rin * rin));
  const double tau_out = p.period_factor * 2.0 * pi / std::sqrt(d.gm / (rout * rout * rout));
  for (int kk = 0; kk < d.nz; ++kk) {
    const double az = std::fabs(d.x0[2] + (kk + 0.5) * dz);
    for (int i = 0; i < d.nr; ++i) {
      const double r = axis0_centre(d, i);
      double rate = 0.0;
      if (g->damp_r) {
        if (r < p.r_edge_in) {
          const double x = (p.r_edge_in - r) / (p.r_edge_in - rin);
          rate = x * x / tau_in;
        } else if (r > p.r_edge_out) {
          const double x = (r - p.r_edge_out) / (rout - p.r_edge_out);
          rate = x * x / tau_out;
        }
      }
      if (g->damp_z && az > g->damp_zp.z_edge) {
        const double x = (az - g->damp_zp.z_edge) / (zmax - g->damp_zp.z_edge);
        rate += x * x / (g->damp_zp.period_factor * 2.0 * pi / std::sqrt(d.gm / (r * r * r)));
      }
      k[(size_t)kk * d.nr + i] = rate;
    }
  }
  std::vector<float> kf(n);
  for (size_t q = 0; q < n; ++q) kf[q] = (float)k[q];
  std::memcpy(k.data() + n, kf.data(), n * sizeof(float));
  rossbi_status st = upload(&g->d_damp, k, g->stream);
  if (st == ROSSBI_OK && cudaStreamSynchronize(g->stream) != cudaSuccess) st = ROSSBI_ERR_CUDA;
  if (st != ROSSBI_OK) return st;
  g->dg.damp_k = g->d_damp;
  g->dg.damp_kf = reinterpret_cast<const float*>(g->d_damp + n);
  return ROSSBI_OK;
}

}  // namespace

extern "C" {

rossbi_status rossbi_set_damping(rossbi_grid* g, const rossbi_damping_params* p) {
  if (!g) return ROSSBI_ERR_ARG;
  if (!p) {
    g->damp_r = false;
    return build_damping(g);
  }
  const rossbi_grid_desc& d = g->desc;
  const double rin = d.x0[0], rout = d.x1[0];
  if (d.geometry != ROSSBI_GEOM_CYL || !g->eq_set || !g->has_disc) return ROSSBI_ERR_ARG;
  if (!(p->r_edge_in > rin) || !(p->r_edge_out < rout) || !(p->r_edge_in <= p->r_edge_out)) return ROSSBI_ERR_ARG;
  if (!(p->period_factor > 0.0) || !std::isfinite(p->period_factor)) return ROSSBI_ERR_ARG;
  g->damp_r = true;
  g->damp_rp = *p;
  return build_damping(g);
}

rossbi_status rossbi_set_vertical_damping(rossbi_grid* g, const rossbi_vertical_damping_params* p) {
  if (!g) return ROSSBI_ERR_ARG;
  if (!p) {
    g->damp_z = false;
    return build_damping(g);
  }
  const rossbi_grid_desc& d = g->desc;
  if (d.geometry != ROSSBI_GEOM_CYL || !g->eq_set || !g->has_disc || !(d.x0[2] == -d.x1[2])) return ROSSBI_ERR_ARG;
  if (!(p->z_edge >= 0.0) || !(p->z_edge < d.x1[2])) return ROSSBI_ERR_ARG;
  if (!(p->period_factor > 0.0) || !std::isfinite(p->period_factor)) return ROSSBI_ERR_ARG;
  g->damp_z = true;
  g->damp_zp = *p;
  return build_damping(g);
}

rossbi_status theta_rows(rossbi_grid* g, void* const* state, int j0, int rows, void* buf, int unpack) {
  if (!g || !state || !buf || rows < 1 || j0 < 0 || j0 + rows > g->desc.nth) return ROSSBI_ERR_ARG;
  for (int f = 0; f < g->nf; ++f)
    if (!state[f]) return ROSSBI_ERR_ARG;
  const rossbi_grid_desc& d = g->desc;
  const size_t n = (size_t)g->nf * d.nz * rows * d.nr;
  const int blocks = (int)std::min<size_t>((n + 255) / 256, 152 * 8);
  if (d.precision == ROSSBI_FP32_PERT) {
    FieldPtrs<float> p{};
    for (int f = 0; f < g->nf; ++f) p.p[f] = (float*)state[f];
    theta_rows_kernel<float><<<blocks, 256, 0, g->stream>>>(p, (float*)buf, d.nr, d.nth, d.nz, g->nf, j0, rows,
                                                             unpack);
  } else {
    FieldPtrs<double> p{};
    for (int f = 0; f < g->nf; ++f) p.p[f] = (double*)state[f];
    theta_rows_kernel<double><<<blocks, 256, 0, g->stream>>>(p, (double*)buf, d.nr, d.nth, d.nz, g->nf, j0, rows,
                                                              unpack);
  }
  CK(cudaGetLastError());
  return ROSSBI_OK;
}

rossbi_status rossbi_pack_theta_rows(rossbi_grid* g, const void* const* state, int j0, int rows, void* buf) {
  return theta_rows(g, (void* const*)state, j0, rows, buf, 0);
}

rossbi_status rossbi_unpack_theta_rows(rossbi_grid* g, void* const* state, int j0, int rows, const void* buf) {
  return theta_rows(g, state, j0, rows, (void*)buf, 1);
}

rossbi_status rossbi_set_dust_species(rossbi_grid* g, const double* stokes_factor, int n) {
  if (!g || !stokes_factor) return ROSSBI_ERR_ARG;
  const int nd = (g->nf - 5) / 4;
  if (n != nd || nd < 1) return ROSSBI_ERR_ARG;
  if (stokes_factor[0] != 1.0) return ROSSBI_ERR_ARG;  // species 0 has the Stokes number itself
  for (int sp = 1; sp < n; ++sp)
    if (!(stokes_factor[sp] > 0.0) || !std::isfinite(stokes_factor[sp])) return ROSSBI_ERR_ARG;
  for (int sp = 0; sp < n; ++sp) g->dg.st_factor[sp] = stokes_factor[sp];
  return ROSSBI_OK;
}

rossbi_status rossbi_indirect_moments(rossbi_grid* g, const void* const* state, double* ab) {
  if (!g || !state || !ab || !g->eq_set || g->desc.geometry != ROSSBI_GEOM_CYL) return ROSSBI_ERR_ARG;
  if (!state[RHO]) return ROSSBI_ERR_ARG;
  for (int b = 5; b < g->nf; b += 4)
    if (!state[b + 3]) return ROSSBI_ERR_ARG;
  rossbi_status st = ensure_ind_tables(g);
  if (st == ROSSBI_OK) st = indirect_moments(g, (void* const*)state);
  if (st != ROSSBI_OK) return st;
  CK(cudaMemcpyAsync(g->h_pinned, g->d_ind, 2 * sizeof(double), cudaMemcpyDeviceToHost, g->stream));
  st = sync_and_status(g);
  ab[0] = g->h_pinned[0];
  ab[1] = g->h_pinned[1];
  return st;
}

rossbi_status rossbi_adjoint_step(rossbi_grid* g, const void* const* state_n, double dt,
                                  const rossbi_dust_params* dust, const void* const* lam_np1, void* const* lam_n,
                                  double* dparam) {
  if (!g) return ROSSBI_ERR_ARG;
  return adjoint_step(g, (void* const*)state_n, dt, dust, lam_np1, lam_n, dparam);
}

rossbi_status rossbi_adjoint_dstokes(rossbi_grid* g, double* total, int reset) {
  if (!g || !total) return ROSSBI_ERR_ARG;
  *total = 0.0;
  if (!g->d_adj_slots) return ROSSBI_OK;
  CK(cudaMemcpyAsync(g->h_pinned, g->d_adj_slots + 1, sizeof(double), cudaMemcpyDeviceToHost, g->stream));
  const rossbi_status st = sync_and_status(g);
  *total = g->h_pinned[0];
  if (reset) {
    CK(cudaMemsetAsync(g->d_adj_slots, 0, 2 * sizeof(double), g->stream));
    CK(cudaStreamSynchronize(g->stream));
  }
  return st;
}

rossbi_status rossbi_take_status(rossbi_grid* g) {
  if (!g) return ROSSBI_ERR_ARG;
  return sync_and_status(g);
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Step without device allocation.
//
// rossbi_step takes its stage scratch (the intermediate state E*) from a
// buffer it cudaMallocs on first use, or from caller-passed buffers.  Some callers can allocate neither: host codes
// that hand all device memory to their own pool at start-up and forbid any
// later cudaMalloc, or loops that cannot afford the implicit device
// synchronisation a cudaMalloc/cudaFree may cause.  rossbi_step_noalloc runs
// the same kernels with that scratch placed in the fixed array below instead.
//
// The array is a file-scope __device__ variable: every GPU that loads this
// library holds NOALLOC_SCRATCH_BYTES of it until the process exits.  Host code
// must not use `noalloc_scratch` as a pointer (in host code the name is a host
// stand-in, not a device address); its device address is looked up once per
// device with cudaGetSymbolAddress, with that device current, on the first
// rossbi_step_noalloc call made on that device.  That first call should
// therefore come before any stream capture.  All calls share the array and it
// keeps the last call's contents; nothing in it needs to start at zero
// (stage 1 writes every E* cell stage 2 reads).  Calls whose work overlaps on the GPU (other streams,
// other grids, other threads) race on the array and must be serialised by the
// caller.
// ---------------------------------------------------------------------------
namespace {

constexpr size_t NOALLOC_SCRATCH_BYTES = (size_t)64 << 20;  // 64 MiB
static __device__ __align__(256) unsigned char noalloc_scratch[NOALLOC_SCRATCH_BYTES];

constexpr int NOALLOC_MAX_DEVICES = 64;
void* noalloc_ptr[NOALLOC_MAX_DEVICES] = {nullptr};

size_t align256(size_t n) { return (n + 255) & ~(size_t)255; }

rossbi_status noalloc_scratch_ptr(void** out) {
  int dev = -1;
  CK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) return ROSSBI_ERR_ARG;
  if (!noalloc_ptr[dev]) {
    void* p = nullptr;
    CK(cudaGetSymbolAddress(&p, noalloc_scratch));
    noalloc_ptr[dev] = p;
  }
  *out = noalloc_ptr[dev];
  return ROSSBI_OK;
}

}  // namespace

extern "C" rossbi_status rossbi_step_noalloc(rossbi_grid* g, void* const* state, double dt,
                                             const rossbi_dust_params* dust, double* next_dt) {
  if (!g || !g->eq_set || !state) return ROSSBI_ERR_ARG;
  for (int f = 0; f < g->nf; ++f)
    if (!state[f]) return ROSSBI_ERR_ARG;
  if (g->nf > 5 && !dust) return ROSSBI_ERR_ARG;
  if (g->nf > 5 && dust->drag_law == 2) return ROSSBI_ERR_ARG;
  if (dt < 0.0 || !std::isfinite(dt)) return ROSSBI_ERR_ARG;
  if (dt == 0.0 && !g->dt_on_device) return ROSSBI_ERR_ARG;
  // the array's address is per device: only the grid's own device may be current
  int dev = -1;
  CK(cudaGetDevice(&dev));
  if (dev != g->device) return ROSSBI_ERR_ARG;
  const size_t field_bytes = align256(g->ncell * elem_size(g));
  // the documented limit: beside the fields, nf + 1 doubles per tile (14 x 6 x 6
  // cells; two z cells in the FP64-state forms of two and more species, 14 x 30 x
  // 1 on a flat FP64 grid), whatever the launches use
  const rossbi_grid_desc& d = g->desc;
  const bool f64 = d.precision != ROSSBI_FP32_PERT;
  const bool flat = d.precision == ROSSBI_FP64 && flat_grid(d.nz, d.bc_lo[2], d.bc_hi[2], g->nf);
  auto tiles = [](int n, int t) { return (size_t)((n + t - 1) / t); };
  const size_t ntiles = tiles(d.nr, 14) * tiles(d.nth, flat ? 30 : 6) * tiles(d.nz, flat ? 1 : (f64 && g->nf > 9 ? 2 : 6));
  const size_t partial_bytes = (size_t)(g->nf + 1) * ntiles * sizeof(double);
  if ((size_t)g->nf * field_bytes + partial_bytes > NOALLOC_SCRATCH_BYTES) return ROSSBI_ERR_ARG;
  DragArgs drag;
  rossbi_status st = drag_args(g, dust, drag);
  if (st != ROSSBI_OK) return st;
  void* base = nullptr;
  st = noalloc_scratch_ptr(&base);
  if (st != ROSSBI_OK) return st;
  void* sc[NF_MAX];
  for (int f = 0; f < g->nf; ++f) sc[f] = (char*)base + (size_t)f * field_bytes;
  // the same two stages as rossbi_step (with the indirect gravity's moments
  // in the grid's own tables, set up by rossbi_set_indirect)
  return step_form(g, state, sc, dt, drag, next_dt);
}
