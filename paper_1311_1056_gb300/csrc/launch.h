// launch.h -- host-side launchers of the CL / gauge-cooling kernels (internal
// interface between the C-ABI runtime and the kernel translation units).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace clgc {

// Launch families whose block size is tunable (cl_autotune).  Every thread
// of these kernels owns one site (or one link), so the block size changes
// neither the arithmetic nor its order; the reductions keep a fixed shape.
enum { TUNE_CLOVER = 0, TUNE_FORCE = 1, TUNE_UPDATE = 2, TUNE_OMEGA = 3, TUNE_APPLY = 4, NTUNE = 5 };
const int TUNE_DEFAULT_BLOCK = 128;
const int TUNE_MAX_BLOCK = 256;  // the launch bound of the tunable kernels

struct GeoH {
  int L[4];
  int V;
  int blk[NTUNE];  // threads per block per family; 0 = TUNE_DEFAULT_BLOCK
};

inline int block_of(const GeoH& h, int fam) { return h.blk[fam] > 0 ? h.blk[fam] : TUNE_DEFAULT_BLOCK; }

// Per-lattice step state, resident on the device so that captured graphs
// replay with fresh noise and the adaptive step size is decided on the GPU.
struct StepDev {
  uint32_t step;                 // Philox step counter (the noise key's step word)
  uint32_t pad;                  // counter of finished blocks (last-block reductions), zero between launches
  double eps_n, sqrt_eps_n;      // step size of the current step (adaptive mode)
  double t;                      // Langevin time: sum of the step sizes taken
  double kmax;                   // K_max of the last adaptive step
  unsigned long long kmax2_bits; // running max of |K|^2 (non-negative doubles order as integers)
};

// Behind it in the same allocation: the largest entry of the plaquette pass's D / 2
// (the high limb's magnitude), from which the FP64 and DF64 forms take the power of
// two that their clover field is kept at.
__host__ __device__ inline unsigned* field_top(StepDev* sd) { return reinterpret_cast<unsigned*>(sd + 1); }
const size_t STEP_DEV_BYTES = sizeof(StepDev) + sizeof(unsigned);

// Packed results of the cooling rule, resident on the device.
struct CoolState {
  double alpha_ad;       // alpha / D of the sweep about to run
  double alpha_ad_last;  // of the last applied sweep
  double un_prev;        // unitarity norm before the last applied sweep
  double un_before, un_after, D;
  int sweeps, done, k, nonfinite;
};

struct CoolArgs {
  double inv_links;  // 1 / (4 V)
  double eps, alpha, tol_rel, d_floor, d_guard;
  int mode, n_min, n_max, forced_sweeps;
};

// Observables accumulated on the device (FP64), one record per call.
struct ObsOut {
  double plaq_re, plaq_im, un, q_re, q_im, sw_re, sw_im, s_re, s_im, max_det_dev;
  double nonfinite;
};

enum { NQ_OBS = 9, RED_THREADS = 128, RED_MAX_BLOCKS = 1216 };

// One chain of a fused batch (the ensemble kernels below): its geometry (the
// fields of lattice.cuh's Geo), device buffers and per-chain parameters.  U
// holds the links the step starts from; the update writes Un, and cooling
// then works on Un (the runtime swaps the two after the step).
struct ChainDesc {
  int L[4], stride[4], V;
  void *U, *Un, *Ui, *Pq, *Dq, *F, *C, *Gq, *f, *Om, *Omi;
  double* arec;             // the cooling kernels' block records
  CoolState* cs;
  StepDev* sd;
  double beta, sre, sim;    // coupling; clover scale -i theta kappa = sre + i sim (FP64: times 2^-cexp)
  int cexp;                 // drift_exponent (FP64)
  double eps, sqrt_eps, k_ref;
  uint64_t seed;
  CoolArgs ca;
};
// One block of a fused launch: chain index and the block index that a
// launch for that chain alone would have had.
struct WorkItem {
  int chain, vb;
};
// Fused kernel families (one launch over the work list's blocks of every
// chain; block size ENS_BLOCK, the reductions' RED_THREADS).
enum {
  ENS_INVERSE = 0,      // link inverses, 4 directions
  ENS_PLAQ = 1,         // plaquettes, 6 planes
  ENS_CLOVER = 2,       // clover field (theta != 0 chains; FP64: two kernels)
  ENS_FORCE_WILSON = 3, // drift contributions, theta = 0 chains
  ENS_FORCE_THETA = 4,  // drift contributions, theta != 0 chains (FP64: two kernels)
  ENS_UPDATE = 5,       // gather + update, fixed step size
  ENS_DRIFTMAX = 6,     // gather, drift into Ui, max |K|^2 (adaptive step size)
  ENS_UPDATE_X = 7,     // update from the drift in Ui (adaptive step size)
  ENS_COOL_GRAD = 8,    // gradient + rule
  ENS_COOL_OMEGA = 9,   // Omega, Omega^{-1}
  ENS_COOL_APPLY = 10,  // apply
  ENS_COOL_GRAD_OMEGA = 11, // single-pass sweeps (D_0 / D_1): gradient + Omega
  ENS_COOL_APPLY_UN = 12,   // single-pass sweeps: apply + rule
  ENS_NFAM = 13
};
const int ENS_BLOCK = 128;

int reduce_blocks(int V);  // number of per-block partial records for V sites

// prec: 0 = FP64 links, 1 = FP32 links.  All pointers are device pointers;
// link fields are SoA (see lattice.cuh), `partials` holds reduce_blocks(V)
// records of NQ_* doubles.
cudaError_t launch_cold(int prec, const GeoH& g, void* U, cudaStream_t st);
cudaError_t launch_hot(int prec, const GeoH& g, void* U, uint64_t seed, cudaStream_t st);
// Omega_x = exp(-sigma g_a lambda_a) per site (Philox stream 1) into Om/Omi.
cudaError_t launch_gauge_omega(int prec, const GeoH& g, void* Om, void* Omi, uint64_t seed,
                               double sigma, cudaStream_t st);
cudaError_t launch_aos_to_soa(int prec, const GeoH& g, const double* aos, void* U, int nplanes,
                              cudaStream_t st);
cudaError_t launch_soa_to_aos(int prec, const GeoH& g, const void* U, double* aos, int nplanes,
                              cudaStream_t st);
// The FP64 and DF64 forms run the step's link algebra in 64-bit fixed point
// (k_update_fx.cuh): Ux receives the links in fixed point (the update's target
// buffer, free until then), the contributions C carry the factor 2^-cexp, cexp =
// drift_exponent(beta, scale_re, scale_im).  FP32 storage ignores Ux and Ui and
// takes cexp = 0.
int drift_exponent(double beta, double sre, double sim);
cudaError_t prepare_step_kernels(int prec);  // before a device's first step of that form
// The CL step (k_update.cuh): link inverses Ui; plaquettes P and D = P - P^{-1}
// (six planes); the clover field F^ = scale * F_{mu nu}(x) built from the D's (fixed
// point: F_{mu nu} / 8 times the power of two of field_top, whatever the scale, which
// the force then applies);
// the per-plaquette drift contributions C (24 planes: 4 links x 6 planes);
// then per link the gather of its six contributions followed by the update
// (mode 0) or by storing the drift matrix X_S (mode 1).
cudaError_t launch_noise_sample(int prec, int site0, int n, uint64_t seed, uint32_t step, int mu, double* out,
                                cudaStream_t st);
cudaError_t launch_link_inverse(int prec, const GeoH& g, const void* U, void* Ux, void* Ui, StepDev* sd, cudaStream_t st);
cudaError_t launch_plaq(int prec, const GeoH& g, const void* U, const void* Ux, const void* Ui, void* Pq, void* Dq,
                        StepDev* sd, cudaStream_t st);
cudaError_t launch_clover_rot(int prec, const GeoH& g, const void* U, const void* Ux, const void* Ui, const void* Dq,
                              void* E, void* F, double scale_re, double scale_im, StepDev* sd, cudaStream_t st);
// The clover field of the fixed-point forms goes through E, six planes of
// scratch (the first of C).  Their theta force runs three kernels, parking the
// transported dual fields and partial sums of them in planes of C (Gq points at
// some of these).
cudaError_t launch_plaq_force(int prec, bool theta, const GeoH& g, const void* U, const void* Ux, const void* Ui,
                              const void* Pq, const void* Dq, const void* F, void* Gq, void* C,
                              double beta, double scale_re, double scale_im, int cexp, StepDev* sd, cudaStream_t st);
// mode 0: update from the gathered drift, step size eps; 1: write the drift X_S
// to out; 2: write X_S to out, max |K| and from it the device step size, eps
// min(1, k_ref / K_max); 3: update reading X_S from C (a mode-2 output), device
// step size.  Modes 0 and 3 count the step (sd->step, the Philox step word, and
// sd->t).
cudaError_t launch_update_gather(int prec, int mode, const GeoH& g, const void* U, const void* C, void* out,
                                 double eps, double k_ref, uint64_t seed, StepDev* sd, int cexp, cudaStream_t st);
// Cooling (cool_sweep.cuh).  What a call works on: the links U; the second link
// buffer Ux, which holds their fixed-point words during a call of the FP64 and
// DF64 forms (FP32 storage: Ux = U); f (8 FP64 values per site, [a][V]); the
// packed Omega, Omega^{-1}; records of 32 bytes, one per 32 sites, and 160 bytes;
// the rule's parameters and state.
struct CoolBufs {
  void *U, *Ux, *f, *Om, *Omi;
  double* rec;
  StepDev* sd;
  CoolState* cs;
  CoolArgs ca;
};
int ens_cool_blocks(int prec, int fam, int V);  // a chain's blocks in a fused launch of family ENS_COOL_*
// Gradient f and (rule) the adaptive rule in its last block; first: a call's
// first one, which reads U and writes Ux.
cudaError_t launch_cool_grad(int prec, const GeoH& g, const CoolBufs& b, bool first, bool rule, cudaStream_t st);
// Omega and its inverse from f.
cudaError_t launch_cool_omega(int prec, const GeoH& g, const CoolBufs& b, cudaStream_t st);
// Single-pass sweeps of the D_0 / D_1 rules: Omega and its inverse straight
// from the gradient with the strength the rule already set.
cudaError_t launch_cool_grad_omega(int prec, const GeoH& g, const CoolBufs& b, cudaStream_t st);
// Apply; rule: single-pass sweeps, the rule for the next sweep from the new
// links' norm.  last: the call's last enqueued sweep, after which U holds the
// links again (also when the rule has stopped the call before).  b.cs NULL:
// no rule state, always applied.
cudaError_t launch_cool_apply(int prec, const GeoH& g, const CoolBufs& b, bool rule, bool last, cudaStream_t st);
// Ux from U (FP64, DF64), for an apply without a gradient before it.
cudaError_t launch_cool_load(int prec, const GeoH& g, const void* U, void* Ux, cudaStream_t st);
// Observables: per-site pass over the links, the plaquette pass's fields and
// the clover field F (FP32 storage: of scale one), then the final fixed-order
// reduction into *out.
cudaError_t launch_obs(int prec, const GeoH& g, const void* U, const void* Ux, const void* Pq, const void* Dq,
                       const void* F, double* partials, double* q_site, StepDev* sd, cudaStream_t st);
cudaError_t launch_obs_final(const GeoH& g, const double* partials, double beta, double th_re,
                             double th_im, ObsOut* out, cudaStream_t st);
// Fused batch: one launch of family fam (ENS_*) over nw work items (device
// arrays cd, w); FP64 and FP32 storage only.  arg: ENS_COOL_GRAD's `first` flag (the call's first gradient runs whatever the rule state); the applies' sweep number.
cudaError_t launch_ens(int prec, int fam, const ChainDesc* cd, const WorkItem* w, int nw, int arg, cudaStream_t st);
// Integer-pipe float <-> double conversions (cvt.cuh) against the hardware
// ones on n generated cases; mismatch counts added into bad[0] (float ->
// double) and bad[1] (double -> float).
cudaError_t launch_selftest_convert(uint64_t seed, long long n, unsigned long long* bad, cudaStream_t st);
// The FP64 Box-Muller's table-driven ln and sincospi against CUDA's log and
// sincospi on n generated uniforms; the largest distances in ulp (rounded
// up) into worst[0] (ln) and worst[1] (sin, cos).
cudaError_t launch_selftest_box_muller(uint64_t seed, long long n, unsigned long long* worst, cudaStream_t st);

}  // namespace clgc
