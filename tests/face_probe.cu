// Entry points around device functions of the library's headers, for the
// tests of their rounding (test_gpu_face_numerics.py).  Pointers are device
// arrays; every thread beyond n returns.
#include "../paper_2207_04252_gb300/csrc/stage_full.cuh"

using namespace rossbi;

__global__ void scalar_kernel(int op, int n, const double* x, double* y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  switch (op) {
    case 0: y[i] = recip(x[i]); break;
    case 1: y[i] = recip_sqrt(x[i]); break;
    case 2: y[i] = root(x[i]); break;
    case 3: y[i] = narrow(x[i]); break;
    case 4: y[i] = widen((float)x[i]); break;
    case 5: y[i] = (positive(x[i]) ? 1 : 0) + (non_negative(x[i]) ? 2 : 0) + (sign_bit(x[i]) ? 4 : 0); break;
    case 6: y[i] = scale_down<3>(x[i]); break;
    case 7: y[i] = recip((float)x[i]); break;
    case 8: y[i] = root((float)x[i]); break;
    case 9: y[i] = recip_sqrt((float)x[i]); break;
    default: y[i] = recip_normal((float)x[i]);
  }
}

// in: [8][n] rho, u, p of the left side, then of the right, p_R - p_L, u_R - u_L; out: [6][n] kind, p* - p_L, u*,
// rho* - rho_K, f_L, f_R
__global__ void near_kernel(NearCoef C, int n, const double* in, double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double v[8];
  for (int q = 0; q < 8; ++q) v[q] = in[(size_t)q * n + i];
  NearStar<double> s{};
  const int kind = near_riemann<NEAR_DEPARTURES>(C, v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7], 0.0, false, v[1], v[4], s);
  const double o[6] = {(double)kind, s.d, s.us, s.drho, s.fl, s.fr};
  for (int q = 0; q < 6; ++q) out[(size_t)q * n + i] = o[q];
}

extern "C" int probe_scalar(int op, int n, const double* x, double* y) {
  scalar_kernel<<<(n + 255) / 256, 256>>>(op, n, x, y);
  return (int)cudaDeviceSynchronize();
}
extern "C" int probe_near(double gamma, int n, const double* in, double* out) {
  near_kernel<<<(n + 255) / 256, 256>>>(near_coef(gamma), n, in, out);
  return (int)cudaDeviceSynchronize();
}
