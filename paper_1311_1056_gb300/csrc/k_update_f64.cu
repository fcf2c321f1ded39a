// k_update_f64.cu -- the CL-step kernels of the FP64 form, and the dispatch over
// the forms.
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
cudaError_t launch_update_gather_f32(int, const GeoH&, const void*, const void*, void*, double, double, uint64_t,
                                     StepDev*, cudaStream_t);

// The smallest e with beta/6 2^-e <= 1/2 and |s| 2^-e <= 1/32 for the clover
// scale's parts: the contributions C 2^-e then stay below 1.4 in fixed point for
// links near SU(3), and as large as that allows.
int drift_exponent(double beta, double sre, double sim) {
  const double m = fmax(2.0 * fabs(beta / 6.0), 32.0 * fmax(fabs(sre), fabs(sim)));
  int e = 0;
  if (!(m > 0.0) || !std::isfinite(m)) return 0;
  if (frexp(m, &e) == 0.5) --e;
  return e < -300 ? -300 : e > 300 ? 300 : e;
}

cudaError_t prepare_step_kernels(int prec) {
  if (prec == 1) return cudaSuccess;
  if (prec == 2) return StepFx<df64>::prepare();
  const cudaError_t e = StepFx<double>::prepare();
  return e == cudaSuccess ? prepare_ens_step<double>() : e;
}

cudaError_t launch_link_inverse(int prec, const GeoH& h, const void* U, void* Ux, void* Ui, StepDev* sd, cudaStream_t st) {
  if (prec == 1) return cudaSuccess;
  return prec == 0 ? StepFx<double>::links(h, U, Ux, Ui, sd, st) : StepFx<df64>::links(h, U, Ux, Ui, sd, st);
}
cudaError_t launch_plaq(int prec, const GeoH& h, const void* U, const void* Ux, const void* Ui, void* Pq, void* Dq,
                        StepDev* sd, cudaStream_t st) {
  if (prec == 1) return launch_plaq_f32(h, U, Pq, Dq, st);
  return prec == 0 ? StepFx<double>::plaq(h, U, Ux, Ui, Pq, Dq, sd, st) : StepFx<df64>::plaq(h, U, Ux, Ui, Pq, Dq, sd, st);
}
cudaError_t launch_clover_rot(int prec, const GeoH& h, const void* U, const void* Ux, const void* Ui, const void* Dq,
                              void* E, void* F, double sre, double sim, StepDev* sd, cudaStream_t st) {
  if (prec == 1) return launch_clover_rot_f32(h, U, Dq, F, sre, sim, st);
  return prec == 0 ? StepFx<double>::clover(h, U, Ux, Ui, Dq, E, F, sd, st)
                   : StepFx<df64>::clover(h, U, Ux, Ui, Dq, E, F, sd, st);
}
cudaError_t launch_plaq_force(int prec, bool theta, const GeoH& h, const void* U, const void* Ux, const void* Ui,
                              const void* Pq, const void* Dq, const void* F, void* Gq, void* C,
                              double beta, double sre, double sim, int cexp, StepDev* sd, cudaStream_t st) {
  if (prec == 1) return launch_plaq_force_f32(theta, h, U, Pq, Dq, F, C, beta, st);
  const double b6 = ldexp(beta / 6.0, -cexp);
  sre = ldexp(sre, -cexp);
  sim = ldexp(sim, -cexp);
  return prec == 0 ? StepFx<double>::force(theta, h, U, Ux, Ui, Pq, Dq, F, Gq, C, b6, sre, sim, sd, st)
                   : StepFx<df64>::force(theta, h, U, Ux, Ui, Pq, Dq, F, Gq, C, b6, sre, sim, sd, st);
}
cudaError_t launch_update_gather(int prec, int mode, const GeoH& h, const void* U, const void* C,
                                 void* out, double eps, double k_ref, uint64_t seed, StepDev* sd,
                                 int cexp, cudaStream_t st) {
  if (prec == 1) return launch_update_gather_f32(mode, h, U, C, out, eps, k_ref, seed, sd, st);
  return prec == 0 ? StepFx<double>::update(mode, h, U, C, out, eps, k_ref, seed, sd, cexp, st)
                   : StepFx<df64>::update(mode, h, U, C, out, eps, k_ref, seed, sd, cexp, st);
}

cudaError_t launch_ens_step_f64(int fam, const ChainDesc* cd, const WorkItem* w, int nw, cudaStream_t st) {
  return launch_ens_step_family<double>(fam, cd, w, nw, st);
}

}  // namespace clgc
