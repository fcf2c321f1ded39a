// ensemble.cuh -- fused-batch wrappers of the CL-step kernels (k_update.cuh):
// one launch runs the blocks of every chain of a batch.  Block i of a launch
// reads its work item (chain, block index the chain's own launch would have
// used) and the chain's descriptor, then runs the same kernel body with that
// chain's geometry, buffers and parameters, so each chain's arithmetic is
// exactly that of its own launches.  Included by k_update_f64.cu and
// k_update_f32.cu, which instantiate it for their link type.
#pragma once
#include "k_update.cuh"
#include "k_update_fx.cuh"
#include "launch.h"

namespace clgc {

__device__ __forceinline__ Geo geo_of(const ChainDesc& c) {
  Geo g;
#pragma unroll
  for (int mu = 0; mu < 4; ++mu) {
    g.L[mu] = c.L[mu];
    g.stride[mu] = c.stride[mu];
  }
  g.V = c.V;
  return g;
}

// Blocks per SM the link-algebra kernels are built for: the FP64 form's as its
// single-chain kernels (k_update_fx_launch.cuh); its force's kernels 2.
static_assert(ENS_BLOCK <= FX_BLOCK, "shared-memory slots of a block");
#define ENS_MIN_BLOCKS(T) (is_fx<T>() ? 3 : 1)

template <typename T>
__global__ void __launch_bounds__(TUNE_MAX_BLOCK) k_ens_inverse(const ChainDesc* __restrict__ cd,
                                                                const WorkItem* __restrict__ w) {
  typedef typename vec2_of<T>::type V2;
  const WorkItem it = w[blockIdx.x];
  const ChainDesc& c = cd[it.chain];
  fx_links_body<T>(geo_of(c), (const V2*)c.U, (int4*)c.Un, (int4*)c.Ui, field_top(c.sd), it.vb);
}

template <typename T>
__global__ void __launch_bounds__(ENS_BLOCK, ENS_MIN_BLOCKS(T)) k_ens_plaq(const ChainDesc* __restrict__ cd,
                                                             const WorkItem* __restrict__ w) {
  typedef typename vec2_of<T>::type V2;
  __shared__ int4 sm[is_fx<T>() ? FX_PIPE : 1];
  const WorkItem it = w[blockIdx.x];
  const ChainDesc& c = cd[it.chain];
  if constexpr (is_fx<T>())
    fx_plaq_body<T>(geo_of(c), (const V2*)c.U, (const int4*)c.Un, (const int4*)c.Ui, (int4*)c.Pq, (int4*)c.Dq, field_top(c.sd),
                    sm, it.vb);
  else
    k_plaq_body<T>(geo_of(c), (const V2*)c.U, (V2*)c.Pq, (V2*)c.Dq, it.vb);
}

// FP64: the clover field's first kernel and the theta force's
template <typename T>
__global__ void __launch_bounds__(ENS_BLOCK, ENS_MIN_BLOCKS(T)) k_ens_clover_half(const ChainDesc* __restrict__ cd,
                                                                    const WorkItem* __restrict__ w) {
  __shared__ int4 sm[FX_PIPE];
  const WorkItem it = w[blockIdx.x];
  const ChainDesc& c = cd[it.chain];
  fx_clover_half_body(geo_of(c), (const int4*)c.Un, (const int4*)c.Ui, (const int4*)c.Dq, (int4*)c.C, field_top(c.sd), sm, it.vb);
}
template <typename T>
__global__ void __launch_bounds__(ENS_BLOCK, ENS_MIN_BLOCKS(T)) k_ens_force_t(const ChainDesc* __restrict__ cd,
                                                                const WorkItem* __restrict__ w) {
  __shared__ int4 sm[FX_PIPE];
  const WorkItem it = w[blockIdx.x];
  const ChainDesc& c = cd[it.chain];
  fx_force_t_body(geo_of(c), (const int4*)c.Un, (const int4*)c.Ui, (const int4*)c.F, (int4*)c.C, sm, it.vb);
}

template <typename T>
__global__ void __launch_bounds__(ENS_BLOCK, ENS_MIN_BLOCKS(T)) k_ens_clover(const ChainDesc* __restrict__ cd,
                                                               const WorkItem* __restrict__ w) {
  typedef typename vec2_of<T>::type V2;
  __shared__ int4 sm[is_fx<T>() ? FX_PIPE : 1];
  const WorkItem it = w[blockIdx.x];
  const ChainDesc& c = cd[it.chain];
  if constexpr (is_fx<T>())
    fx_clover_body<T>(geo_of(c), (const V2*)c.U, (const int4*)c.Un, (const int4*)c.Ui, (const int4*)c.Dq,
                      (const int4*)c.C, (int4*)c.F, field_top(c.sd), sm, it.vb);
  else
    k_clover_rot_body<T>(geo_of(c), (const V2*)c.U, (const V2*)c.Dq, (V2*)c.F, c.sre, c.sim, it.vb);
}

template <typename T>
__global__ void __launch_bounds__(ENS_BLOCK, is_fx<T>() ? 2 : 1) k_ens_force_wilson(const ChainDesc* __restrict__ cd,
                                                                     const WorkItem* __restrict__ w) {
  typedef typename vec2_of<T>::type V2;
  __shared__ int4 sm[is_fx<T>() ? FX_PIPE : 1];
  const WorkItem it = w[blockIdx.x];
  const ChainDesc& c = cd[it.chain];
  if constexpr (is_fx<T>())
    fx_force_wilson_body<T>(geo_of(c), (const V2*)c.U, (const int4*)c.Un, (const int4*)c.Ui, (const int4*)c.Dq, (int4*)c.C,
                         ldexp(c.beta / 6.0, -c.cexp), sm, it.vb);
  else
    k_plaq_force_wilson_body<T>(geo_of(c), (const V2*)c.U, (const V2*)c.Dq, (V2*)c.C,
                              (T)(c.beta / 6.0), it.vb);
}

template <typename T>
__global__ void __launch_bounds__(ENS_BLOCK, 2) k_ens_force_a(const ChainDesc* __restrict__ cd,
                                                                const WorkItem* __restrict__ w) {
  const WorkItem it = w[blockIdx.x];
  const ChainDesc& c = cd[it.chain];
  extern __shared__ int4 sm_park[];
  fx_force_a_body(geo_of(c), (const int4*)c.Un, (const int4*)c.Ui, (const int4*)c.Dq, (const int4*)c.F, (int4*)c.Gq,
                  (int4*)c.C, ldexp(c.beta / 6.0, -c.cexp), c.sre, c.sim, field_top(c.sd), sm_park, it.vb);
}

template <typename T>
__global__ void __launch_bounds__(ENS_BLOCK, 2) k_ens_force_b(const ChainDesc* __restrict__ cd,
                                                                const WorkItem* __restrict__ w) {
  const WorkItem it = w[blockIdx.x];
  const ChainDesc& c = cd[it.chain];
  __shared__ int4 sm[FX_PIPE];
  fx_force_b_body<T>(geo_of(c), (const typename vec2_of<T>::type*)c.U, (const int4*)c.Un, (const int4*)c.Ui, (const int4*)c.Pq,
                  (const int4*)c.Dq, (const int4*)c.F, (const int4*)c.Gq, (int4*)c.C, ldexp(c.beta / 6.0, -c.cexp), c.sre,
                  c.sim, field_top(c.sd), sm, it.vb);
}

template <typename T>
__global__ void __maxnreg__(FORCE_AB_MAXNREG) k_ens_force_ab(const ChainDesc* __restrict__ cd,
                                                                 const WorkItem* __restrict__ w) {
  typedef typename vec2_of<T>::type V2;
  const WorkItem it = w[blockIdx.x];
  const ChainDesc& c = cd[it.chain];
  k_plaq_force_ab_body<T>(geo_of(c), (const V2*)c.U, (const V2*)c.Pq, (const V2*)c.Dq,
                          (const V2*)c.F, (V2*)c.C, (T)(c.beta / 6.0), it.vb);
}

// The update modes as the runtime runs them: MODE_UPDATE reads C and writes
// Un at the fixed step size; MODE_DRIFTMAX writes the drift into Pq (dead
// after the force); MODE_UPDATE_X reads it back and writes Un at the device
// step size.
template <typename T, int MODE>
__global__ void __launch_bounds__(ENS_BLOCK, 3) k_ens_update(const ChainDesc* __restrict__ cd,
                                                               const WorkItem* __restrict__ w) {
  typedef typename vec2_of<T>::type V2;
  const WorkItem it = w[blockIdx.x];
  const ChainDesc& c = cd[it.chain];
  const UpdArgs a = {c.eps, c.sqrt_eps, c.k_ref, c.seed, c.sd, MODE == MODE_UPDATE_X ? 1 : 0, c.cexp};
  const void* in = MODE == MODE_UPDATE_X ? c.Pq : c.C;
  void* out = MODE == MODE_DRIFTMAX ? c.Pq : c.Un;
  const uint32_t step = step_begin<MODE>(geo_of(c), a);
  if constexpr (is_fx<T>())
    fx_update_body<T, MODE>(geo_of(c), (const V2*)c.U, (const int4*)in, out, a, step, it.vb);
  else
    k_update_gather_body<T, MODE>(geo_of(c), (const V2*)c.U, (const V2*)in, (V2*)out, a, step, it.vb);
  step_size<MODE>(geo_of(c), a);
}

template <typename T>
cudaError_t prepare_ens_step() {
  return cudaFuncSetAttribute(k_ens_force_a<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, FX_PARK_BYTES);
}

// Launch family fam of the CL step for link type T (FP64 runs the clover
// field and the theta force as two and three kernels).
template <typename T>
cudaError_t launch_ens_step_family(int fam, const ChainDesc* cd, const WorkItem* w, int nw, cudaStream_t st) {
  if (nw <= 0) return cudaSuccess;
  const unsigned n = (unsigned)nw;
  switch (fam) {
    case ENS_INVERSE:
      if constexpr (is_fx<T>()) k_ens_inverse<T><<<n, ENS_BLOCK, 0, st>>>(cd, w);
      break;
    case ENS_PLAQ: k_ens_plaq<T><<<n, ENS_BLOCK, 0, st>>>(cd, w); break;
    case ENS_CLOVER:
      if constexpr (is_fx<T>()) k_ens_clover_half<T><<<n, ENS_BLOCK, 0, st>>>(cd, w);
      k_ens_clover<T><<<n, ENS_BLOCK, 0, st>>>(cd, w); break;
    case ENS_FORCE_WILSON: k_ens_force_wilson<T><<<n, ENS_BLOCK, 0, st>>>(cd, w); break;
    case ENS_FORCE_THETA:
      if constexpr (is_fx<T>()) {
        k_ens_force_t<T><<<n, ENS_BLOCK, 0, st>>>(cd, w);
        k_ens_force_a<T><<<n, ENS_BLOCK, FX_PARK_BYTES, st>>>(cd, w);
        k_ens_force_b<T><<<n, ENS_BLOCK, 0, st>>>(cd, w);
      } else {
        k_ens_force_ab<T><<<n, ENS_BLOCK, 0, st>>>(cd, w);
      }
      break;
    case ENS_UPDATE: k_ens_update<T, MODE_UPDATE><<<n, ENS_BLOCK, 0, st>>>(cd, w); break;
    case ENS_DRIFTMAX: k_ens_update<T, MODE_DRIFTMAX><<<n, ENS_BLOCK, 0, st>>>(cd, w); break;
    case ENS_UPDATE_X: k_ens_update<T, MODE_UPDATE_X><<<n, ENS_BLOCK, 0, st>>>(cd, w); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace clgc
