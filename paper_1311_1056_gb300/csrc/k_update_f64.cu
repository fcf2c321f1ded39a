// k_update_f64.cu -- the CL-step kernels of the FP64 form, the dispatch over the
// forms and the step's bookkeeping.
#include <cmath>

#include "ensemble.cuh"
#include "k_update_fx_launch.cuh"
#include "launch.h"

namespace clgc {

template struct StepFx<double>;
extern template struct StepFx<df64>;  // k_update_df64.cu

// k_update_f32.cu
cudaError_t launch_plaq_f32(const GeoH&, const void*, void*, void*, cudaStream_t);
cudaError_t launch_clover_rot_f32(const GeoH&, const void*, const void*, void*, double, double, cudaStream_t);
cudaError_t launch_plaq_force_f32(bool, const GeoH&, const void*, const void*, const void*, const void*, void*, double,
                                  cudaStream_t);
cudaError_t launch_update_gather_f32(int, const GeoH&, const void*, const void*, void*, double,
                                     uint64_t, StepDev*, bool, cudaStream_t);

// The smallest e with beta/6 2^-e <= 1/4 and |s| 2^-e <= 1/128 for the clover
// scale's parts: the contributions C 2^-e then stay below 1.4 in fixed point.
int drift_exponent(double beta, double sre, double sim) {
  const double m = fmax(4.0 * fabs(beta / 6.0), 128.0 * fmax(fabs(sre), fabs(sim)));
  int e = 0;
  if (!(m > 0.0) || !std::isfinite(m)) return 0;
  frexp(m, &e);
  return e < -300 ? -300 : e > 300 ? 300 : e;
}

cudaError_t launch_link_inverse(int prec, const GeoH& h, const void* U, void* Ux, void* Ui, cudaStream_t st) {
  if (prec == 1) return cudaSuccess;
  return prec == 0 ? StepFx<double>::links(h, U, Ux, Ui, st) : StepFx<df64>::links(h, U, Ux, Ui, st);
}
cudaError_t launch_plaq(int prec, const GeoH& h, const void* U, const void* Ux, const void* Ui, void* Pq, void* Dq,
                        cudaStream_t st) {
  if (prec == 1) return launch_plaq_f32(h, U, Pq, Dq, st);
  return prec == 0 ? StepFx<double>::plaq(h, U, Ux, Ui, Pq, Dq, st) : StepFx<df64>::plaq(h, U, Ux, Ui, Pq, Dq, st);
}
cudaError_t launch_clover_rot(int prec, const GeoH& h, const void* U, const void* Ux, const void* Ui, const void* Dq,
                              void* E, void* F, double sre, double sim, cudaStream_t st) {
  if (prec == 1) return launch_clover_rot_f32(h, U, Dq, F, sre, sim, st);
  return prec == 0 ? StepFx<double>::clover(h, U, Ux, Ui, Dq, E, F, sre, sim, st)
                   : StepFx<df64>::clover(h, U, Ux, Ui, Dq, E, F, sre, sim, st);
}
cudaError_t launch_plaq_force(int prec, bool theta, const GeoH& h, const void* U, const void* Ux, const void* Ui,
                              const void* Pq, const void* Dq, const void* F, void* Gq, void* C,
                              double beta, int cexp, cudaStream_t st) {
  if (prec == 1) return launch_plaq_force_f32(theta, h, U, Pq, Dq, F, C, beta, st);
  const double b6 = ldexp(beta / 6.0, -cexp);
  return prec == 0 ? StepFx<double>::force(theta, h, U, Ux, Ui, Pq, Dq, F, Gq, C, b6, st)
                   : StepFx<df64>::force(theta, h, U, Ux, Ui, Pq, Dq, F, Gq, C, b6, st);
}
cudaError_t launch_update_gather(int prec, int mode, const GeoH& h, const void* U, const void* C,
                                 void* out, double eps, uint64_t seed, StepDev* sd, bool adaptive,
                                 int cexp, cudaStream_t st) {
  if (prec == 1) return launch_update_gather_f32(mode, h, U, C, out, eps, seed, sd, adaptive, st);
  return prec == 0 ? StepFx<double>::update(mode, h, U, C, out, eps, seed, sd, adaptive, cexp, st)
                   : StepFx<df64>::update(mode, h, U, C, out, eps, seed, sd, adaptive, cexp, st);
}

// After an update: step += 1 and t += the step size taken (one thread).
__device__ __forceinline__ void step_bump(StepDev* sd, double eps, int adaptive) {
  sd->step += 1u;
  sd->t += adaptive ? sd->eps_n : eps;
}
__global__ void k_step_bump(StepDev* sd, double eps, int adaptive) { step_bump(sd, eps, adaptive); }

// Adaptive step size from the drift pass's max |K|^2: eps_n = eps min(1, k_ref / K_max);
// clears the running max for the next step.
__device__ __forceinline__ void step_eps(StepDev* sd, double eps, double k_ref) {
  const double kmax = sqrt(__longlong_as_double((long long)sd->kmax2_bits));
  const double e = kmax > k_ref ? eps * (k_ref / kmax) : eps;
  sd->eps_n = e;
  sd->sqrt_eps_n = sqrt(e);
  sd->kmax = kmax;
  sd->kmax2_bits = 0ull;
}
__global__ void k_step_eps(StepDev* sd, double eps, double k_ref) { step_eps(sd, eps, k_ref); }

// The same for the chains of a fused batch, one thread per listed chain.
__global__ void k_ens_step_eps(const ChainDesc* __restrict__ cd, const int* __restrict__ chains, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const ChainDesc& c = cd[chains[i]];
  step_eps(c.sd, c.eps, c.k_ref);
}
__global__ void k_ens_step_bump(const ChainDesc* __restrict__ cd, const int* __restrict__ chains,
                                const int* __restrict__ adaptive, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const ChainDesc& c = cd[chains[i]];
  step_bump(c.sd, c.eps, adaptive[i]);
}

cudaError_t launch_ens_step_eps(const ChainDesc* cd, const int* chains, int n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_ens_step_eps<<<(n + 127) / 128, 128, 0, st>>>(cd, chains, n);
  return cudaGetLastError();
}
cudaError_t launch_ens_step_bump(const ChainDesc* cd, const int* chains, const int* adaptive, int n,
                                 cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_ens_step_bump<<<(n + 127) / 128, 128, 0, st>>>(cd, chains, adaptive, n);
  return cudaGetLastError();
}

cudaError_t launch_step_bump(StepDev* sd, double eps, bool adaptive, cudaStream_t st) {
  k_step_bump<<<1, 1, 0, st>>>(sd, eps, adaptive ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_step_eps(StepDev* sd, double eps, double k_ref, cudaStream_t st) {
  k_step_eps<<<1, 1, 0, st>>>(sd, eps, k_ref);
  return cudaGetLastError();
}
cudaError_t launch_ens_step_f64(int fam, const ChainDesc* cd, const WorkItem* w, int nw, cudaStream_t st) {
  return launch_ens_step_family<double>(fam, cd, w, nw, st);
}

}  // namespace clgc
