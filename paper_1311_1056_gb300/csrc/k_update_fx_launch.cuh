// k_update_fx_launch.cuh -- kernels and launches of the CL step in fixed point
// (k_update_fx.cuh) for one link type, instantiated by k_update_f64.cu and
// k_update_df64.cu.
#pragma once
#include <algorithm>
#include <cmath>

#include "k_update_fx.cuh"
#include "launch.h"

namespace clgc {

// The step's launches for links of type L (k_update_fx_launch.cuh).
template <typename L>
struct StepFx {
  static cudaError_t prepare();  // once per device: shared memory of the theta force
  static cudaError_t links(const GeoH& h, const void* U, void* Ux, void* Ui, StepDev* sd, cudaStream_t st);
  static cudaError_t plaq(const GeoH& h, const void* U, const void* Ux, const void* Ui, void* Pq, void* Dq, StepDev* sd,
                          cudaStream_t st);
  static cudaError_t clover(const GeoH& h, const void* U, const void* Ux, const void* Ui, const void* Dq, void* E,
                            void* F, StepDev* sd, cudaStream_t st);
  static cudaError_t force(bool theta, const GeoH& h, const void* U, const void* Ux, const void* Ui, const void* Pq, const void* Dq, const void* F, void* Gq, void* C, double b6,
                           double sre, double sim, StepDev* sd, cudaStream_t st);
  static cudaError_t update(int mode, const GeoH& h, const void* U, const void* C, void* out, double eps, double k_ref,
                            uint64_t seed, StepDev* sd, int cexp, cudaStream_t st);
};

namespace {
// 1-D grid, plane (or direction) fastest: the blocks resident at one time
// cover every plane of a range of sites, so shared neighbours stay in cache.
inline dim3 grid(int V, int planes, int bs) { return dim3((unsigned)(((V + bs - 1) / bs) * planes)); }

// Resident blocks of 128 threads that the kernels are built for.  Three (168
// registers) for the plaquettes and the clover field, whose operands come
// through the pipe.  Two (255, next to nothing spilled) for the theta force's
// stages a and b: 5.68 ms per 32^4 step when this was chosen (with the transport pass; now,
// with the theta scale applied here, 6.17); three blocks
// spill ~470 bytes a thread and took 6.34 ms without the pipe, 6.98 ms with it
// (its slots are the spills' L1).  FP64 arithmetic took 26.0 ms, plaquettes and
// clover field 11.95 (now 2.59).
const int FX_BLOCKS_SM = 3, FX_BLOCKS_FORCE = 2;
template <typename L>
__global__ void __launch_bounds__(TUNE_MAX_BLOCK) k_fx_links(Geo g, const typename vec2_of<L>::type* __restrict__ U, int4* Ux, int4* Ui,
                                                             unsigned* top) {
  fx_links_body<L>(g, U, Ux, Ui, top, blockIdx.x);
}
template <typename L>
__global__ void __launch_bounds__(FX_BLOCK, FX_BLOCKS_SM) k_fx_plaq(Geo g, const typename vec2_of<L>::type* U, const int4* __restrict__ Ux,
                                                            const int4* __restrict__ Ui, int4* Pq, int4* Dq, unsigned* top) {
  __shared__ int4 sm[FX_PIPE];
  fx_plaq_body<L>(g, U, Ux, Ui, Pq, Dq, top, sm, blockIdx.x);
}
__global__ void __launch_bounds__(FX_BLOCK, FX_BLOCKS_SM) k_fx_clover_half(Geo g, const int4* __restrict__ Ux, const int4* __restrict__ Ui,
                                                         const int4* __restrict__ Dq, int4* E, const unsigned* top) {
  __shared__ int4 sm[FX_PIPE];
  fx_clover_half_body(g, Ux, Ui, Dq, E, top, sm, blockIdx.x);
}
template <typename L>
__global__ void __launch_bounds__(FX_BLOCK, FX_BLOCKS_SM) k_fx_clover(Geo g, const typename vec2_of<L>::type* U, const int4* __restrict__ Ux,
                                                    const int4* __restrict__ Ui, const int4* __restrict__ Dq,
                                                    const int4* __restrict__ E, int4* F, const unsigned* top) {
  __shared__ int4 sm[FX_PIPE];
  fx_clover_body<L>(g, U, Ux, Ui, Dq, E, F, top, sm, blockIdx.x);
}
template <typename L>
__global__ void __launch_bounds__(FX_BLOCK, FX_BLOCKS_FORCE) k_fx_force_wilson(Geo g, const typename vec2_of<L>::type* U,
                                                                    const int4* __restrict__ Ux,
                                                                    const int4* __restrict__ Ui,
                                                                    const int4* __restrict__ Dq, int4* C, double b6) {
  __shared__ int4 sm[FX_PIPE];
  fx_force_wilson_body<L>(g, U, Ux, Ui, Dq, C, b6, sm, blockIdx.x);
}
__global__ void __launch_bounds__(FX_BLOCK, FX_BLOCKS_SM) k_fx_force_t(Geo g, const int4* __restrict__ Ux, const int4* __restrict__ Ui,
                                                     const int4* __restrict__ F, int4* C) {
  __shared__ int4 sm[FX_PIPE];
  fx_force_t_body(g, Ux, Ui, F, C, sm, blockIdx.x);
}
__global__ void __launch_bounds__(FX_BLOCK, FX_BLOCKS_FORCE) k_fx_force_a(Geo g, const int4* __restrict__ Ux,
                                                               const int4* __restrict__ Ui,
                                                               const int4* __restrict__ Dq,
                                                               const int4* __restrict__ F, int4* Gq, int4* C,
                                                               double b6, double sre, double sim, const unsigned* top) {
  extern __shared__ int4 sm_park[];
  fx_force_a_body(g, Ux, Ui, Dq, F, Gq, C, b6, sre, sim, top, sm_park, blockIdx.x);
}
template <typename L>
__global__ void __launch_bounds__(FX_BLOCK, FX_BLOCKS_FORCE) k_fx_force_b(Geo g, const typename vec2_of<L>::type* U, const int4* __restrict__ Ux,
                                                               const int4* __restrict__ Ui, const int4* Pq,
                                                               const int4* Dq, const int4* F, const int4* Gq, int4* C,
                                                               double b6, double sre, double sim, const unsigned* top) {
  __shared__ int4 sm[FX_PIPE];
  fx_force_b_body<L>(g, U, Ux, Ui, Pq, Dq, F, Gq, C, b6, sre, sim, top, sm, blockIdx.x);
}
template <typename L, int MODE>
__global__ void __maxnreg__(UPDATE_MAXNREG) k_fx_update(Geo g, const typename vec2_of<L>::type* __restrict__ U,
                                                              const int4* __restrict__ C, void* __restrict__ out, UpdArgs a) {
  const uint32_t step = step_begin<MODE>(g, a);
  fx_update_body<L, MODE>(g, U, C, out, a, step, blockIdx.x);
  step_size<MODE>(g, a);
}
}  // namespace

template <typename L>
cudaError_t StepFx<L>::prepare() {
  return cudaFuncSetAttribute(k_fx_force_a, cudaFuncAttributeMaxDynamicSharedMemorySize, FX_PARK_BYTES);
}

template <typename L>
cudaError_t StepFx<L>::links(const GeoH& h, const void* U, void* Ux, void* Ui, StepDev* sd, cudaStream_t st) {
  Geo g = make_geo(h.L, h.V);
  const int bs = std::min(block_of(h, TUNE_CLOVER), FX_BLOCK);
  k_fx_links<L><<<grid(g.V, 4, bs), bs, 0, st>>>(g, (const typename vec2_of<L>::type*)U, (int4*)Ux, (int4*)Ui, field_top(sd));
  return cudaGetLastError();
}

template <typename L>
cudaError_t StepFx<L>::plaq(const GeoH& h, const void* U, const void* Ux, const void* Ui, void* Pq, void* Dq,
                            StepDev* sd, cudaStream_t st) {
  Geo g = make_geo(h.L, h.V);
  const int bs = std::min(block_of(h, TUNE_CLOVER), FX_BLOCK);
  k_fx_plaq<L><<<grid(g.V, 6, bs), bs, 0, st>>>(g, (const typename vec2_of<L>::type*)U, (const int4*)Ux, (const int4*)Ui, (int4*)Pq, (int4*)Dq, field_top(sd));
  return cudaGetLastError();
}

template <typename L>
cudaError_t StepFx<L>::clover(const GeoH& h, const void* U, const void* Ux, const void* Ui, const void* Dq,
                                  void* E, void* F, StepDev* sd, cudaStream_t st) {
  Geo g = make_geo(h.L, h.V);
  const int bs = std::min(block_of(h, TUNE_CLOVER), FX_BLOCK);
  k_fx_clover_half<<<grid(g.V, 6, bs), bs, 0, st>>>(g, (const int4*)Ux, (const int4*)Ui, (const int4*)Dq, (int4*)E, field_top(sd));
  k_fx_clover<L><<<grid(g.V, 6, bs), bs, 0, st>>>(g, (const typename vec2_of<L>::type*)U, (const int4*)Ux, (const int4*)Ui, (const int4*)Dq, (const int4*)E, (int4*)F, field_top(sd));
  return cudaGetLastError();
}

template <typename L>
cudaError_t StepFx<L>::force(bool theta, const GeoH& h, const void* U, const void* Ux, const void* Ui,
                                  const void* Pq, const void* Dq, const void* F, void* Gq, void* C, double b6,
                                  double sre, double sim, StepDev* sd, cudaStream_t st) {
  Geo g = make_geo(h.L, h.V);
  const int bs = std::min(block_of(h, TUNE_FORCE), FX_BLOCK);
  const dim3 gr = grid(g.V, 6, bs);
  if (!theta) {
    k_fx_force_wilson<L><<<gr, bs, 0, st>>>(g, (const typename vec2_of<L>::type*)U, (const int4*)Ux, (const int4*)Ui, (const int4*)Dq, (int4*)C, b6);
    return cudaGetLastError();
  }
  k_fx_force_t<<<gr, bs, 0, st>>>(g, (const int4*)Ux, (const int4*)Ui, (const int4*)F, (int4*)C);
  k_fx_force_a<<<gr, bs, FX_PARK_BYTES, st>>>(g, (const int4*)Ux, (const int4*)Ui, (const int4*)Dq, (const int4*)F, (int4*)Gq,
                                  (int4*)C, b6, sre, sim, field_top(sd));
  k_fx_force_b<L><<<gr, bs, 0, st>>>(g, (const typename vec2_of<L>::type*)U, (const int4*)Ux, (const int4*)Ui, (const int4*)Pq, (const int4*)Dq,
                                  (const int4*)F, (const int4*)Gq, (int4*)C, b6, sre, sim, field_top(sd));
  return cudaGetLastError();
}

template <typename L>
cudaError_t StepFx<L>::update(int mode, const GeoH& h, const void* U, const void* C, void* out, double eps, double k_ref,
                              uint64_t seed, StepDev* sd, int cexp, cudaStream_t st) {
  Geo g = make_geo(h.L, h.V);
  const UpdArgs a = update_args(mode, eps, k_ref, seed, sd, cexp);
  const int bs = block_of(h, TUNE_UPDATE);
  const dim3 gr = grid(g.V, 4, bs);
  const typename vec2_of<L>::type* u = (const typename vec2_of<L>::type*)U;
  const int4* c = (const int4*)C;
  switch (mode) {
    case MODE_DRIFT: k_fx_update<L, MODE_DRIFT><<<gr, bs, 0, st>>>(g, u, c, out, a); break;
    case MODE_DRIFTMAX: k_fx_update<L, MODE_DRIFTMAX><<<gr, bs, 0, st>>>(g, u, c, out, a); break;
    case MODE_UPDATE_X: k_fx_update<L, MODE_UPDATE_X><<<gr, bs, 0, st>>>(g, u, c, out, a); break;
    default: k_fx_update<L, MODE_UPDATE><<<gr, bs, 0, st>>>(g, u, c, out, a); break;
  }
  return cudaGetLastError();
}

}  // namespace clgc
