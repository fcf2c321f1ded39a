// k_update_df64.cu -- the CL-step kernels of the DF64 form: links stored as
// double-float pairs, everything between the links in fixed point as in the
// FP64 form (k_update_fx.cuh).  Double-float arithmetic on the FP32 pipe, with
// the matrices in a shared-memory workspace, took 20.8 ms per 32^4 step of ten
// sweeps (whose sweeps were in fixed point) against 18.2 (now 16.7), observables 8.9
// against 3.4 (3.0), and its error was thirteen times larger (1.1e-14 against
// 8.6e-16 of the links after a 16^4 step).
#include "k_update_fx_launch.cuh"

namespace clgc {
template struct StepFx<df64>;
}  // namespace clgc
