// link_fx.cuh -- links of the FP64 form (double) and of the DF64 form (df64,
// double-float) to and from fixed point (fixed.cuh).  The two forms differ in
// what a link is stored as and in nothing else.
#pragma once
#include "fixed.cuh"

namespace clgc {

// Link types whose kernels work in fixed point.
template <typename L>
__host__ __device__ constexpr bool is_fx() { return sizeof(typename vec2_of<L>::type) == 16; }

__device__ __forceinline__ double real_d(double x) { return x; }
__device__ __forceinline__ double real_d(float x) { return (double)x; }
__device__ __forceinline__ double real_d(df64 x) { return (double)x.hi + (double)x.lo; }
// Link (mu, s) as doubles (exact).
template <typename L>
__device__ __forceinline__ void load_link_d(mat<double>& d, const typename vec2_of<L>::type* U, int mu, int s, int V) {
  mat<L> u;
  load(u, U, mu, s, V);
#pragma unroll
  for (int k = 0; k < 9; ++k) d.e[k] = cx<double>{real_d(u.e[k].re), real_d(u.e[k].im)};
}
__device__ __forceinline__ void store_link(double2* U, int mu, int s, int V, const mat<double>& d) { store(U, mu, s, V, d); }
__device__ __forceinline__ void store_link(float4* U, int mu, int s, int V, const mat<double>& d) {
  mat<df64> u;
#pragma unroll
  for (int k = 0; k < 9; ++k) u.e[k] = cx<df64>{df64(d.e[k].re), df64(d.e[k].im)};
  store(U, mu, s, V, u);
}
// In fixed point; false out of range.
__device__ __forceinline__ bool fx_of_link(fx& r, double x) {
  unsigned mag = 0;
  r = fx_of_double(x, mag);
  return fx_mag_ok(mag);
}
__device__ __forceinline__ bool fx_of_link(fx& r, df64 x) {
  // hi and lo each to the nearest 2^-30, the rest (exact) to the low limb
  const float a = x.hi * 0x1p30f, b = x.lo * 0x1p30f;
  const int h = __float2int_rn(a), m = __float2int_rn(b);
  r = fx_of_bits(mad_wide(h + m, 1 << 30, (long long)__float2int_rn(((a - (float)h) + (b - (float)m)) * 0x1p30f)));
  return fabsf(x.hi) < 1.4375f;
}
template <typename L>
__device__ __forceinline__ bool fx_load_link(mat<fx>& u, const typename vec2_of<L>::type* U, int mu, int s, int V) {
  mat<L> w;
  load(w, U, mu, s, V);
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const bool a = fx_of_link(u.e[k].re, w.e[k].re), b = fx_of_link(u.e[k].im, w.e[k].im);
    ok = ok && a && b;
  }
  return ok;
}
__device__ __forceinline__ double2 fx_link_word(double2*, cx<fx> a) { return make_double2(fx_to_double(a.re), fx_to_double(a.im)); }
__device__ __forceinline__ df64 fx_to_df64(fx a) {
  const float hi = (float)a.h;
  const float rem = (float)(a.h - __float2int_rn(hi));
  return df_two_sum(hi * 0x1p-30f, fmaf(a.l, 0x1p-30f, rem) * 0x1p-30f);
}
__device__ __forceinline__ float4 fx_link_word(float4*, cx<fx> a) { return df_pack(fx_to_df64(a.re), fx_to_df64(a.im)); }
template <class V2>
__device__ __forceinline__ void fx_store_link(V2* U, int mu, int s, int V, const mat<fx>& u) {
  V2* p = U + (size_t)mu * 9 * V + s;
#pragma unroll
  for (int k = 0; k < 9; ++k) p[(size_t)k * V] = fx_link_word(U, u.e[k]);
}
template <typename L>
struct link_field {  // the general paths' view of the links
  const typename vec2_of<L>::type* p;
};
template <typename L>
__device__ __forceinline__ void load(mat<double>& d, link_field<L> f, int mu, int s, int V) {
  load_link_d<L>(d, f.p, mu, s, V);
}

}  // namespace clgc
