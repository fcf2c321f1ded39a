// noise_fx.cuh -- the CL noise of the FP64 form in fixed point (fixed.cuh): the
// Philox words and Box-Muller pairs of philox.cuh, no FP64 instruction.
//
// GB300 issues FP64 at 1/64 of its FP32 rate; the FP64 pair (table-driven ln
// and sincospi, sqrt) took ~45 issue slots of 64 cycles.  The uniforms are
// 53-bit integers, so everything starts exact: the significand of u times a
// 10-bit reciprocal is exact in 64 bits, and so is the angle's distance from
// the nearest multiple of pi / 64.  The normal numbers come out divided by 8
// (|g| <= 8.6) to 2^-57, below the rounding of an FP64 evaluation.
#pragma once
#include "fixed.cuh"
#include "noise_fx_tables.cuh"
#include "philox.cuh"

namespace clgc {

__device__ __forceinline__ fx fx_constant(int h, int l) { return fx{(float)l, h}; }

// One Horner step, a q + c, of numbers within bounds by construction.
__device__ __forceinline__ fx fx_horner(const fx_left& a, fx q, fx c) {
  fx_acc s = fx_from(c);
  fx_mac(s, a, fx_rhs(q));
  return fx_split(fx_sum(s));
}
__device__ __forceinline__ fx fx_times(const fx_left& a, const fx_right& b) {
  fx_acc s = fx_zero();
  fx_mac(s, a, b);
  return fx_split(fx_sum(s));
}
// 1 / n as a constant
__device__ __forceinline__ fx fx_one_over(int n, int sign) {
  const long long v = ((1ll << 60) + n / 2) / n, h = (v + (1ll << 29)) >> 30;
  return fx_constant((int)(sign * h), (int)(sign * (v - (h << 30))));
}

// sqrt(-2 ln u) / 8 for u = (k + 1/2) 2^-52.
__device__ __forceinline__ fx fx_radius(uint64_t k) {
  const uint64_t n = 2 * k + 1;  // u = n 2^-53
  const int lz = __clzll((long long)n);
  const uint64_t m = n << (lz - 11);  // leading one at bit 52
  const int i = (int)(m >> 45) & 127;
  const bool fold = i >= NFX_LN_FOLD;      // take m / 2
  const int ne = lz - 10 - (fold ? 1 : 0);  // u = 2^-ne m', m' in [0.7, 1.42)
  const longlong2 tab = __ldg(&NFX_LN_TAB[i]);
  // t = m' R / 512 - 1, exact in units of 2^-62, |t| < 2^-7.3
  const long long t62 = (long long)(m * (uint64_t)tab.x << (fold ? 0 : 1)) - (1ll << 62);
  const fx t = fx_of_bits(t62 >> 2);
  // q = ln(1 + t) / t = 1 - t/2 + t^2/3 - ... - t^7/8 (the next term is below 2^-61)
  const fx_left tl = fx_lhs(t);
  fx q = fx_one_over(8, -1);
  q = fx_horner(tl, q, fx_one_over(7, 1));
  q = fx_horner(tl, q, fx_one_over(6, -1));
  q = fx_horner(tl, q, fx_one_over(5, 1));
  q = fx_horner(tl, q, fx_one_over(4, -1));
  q = fx_horner(tl, q, fx_one_over(3, 1));
  q = fx_horner(tl, q, fx_one_over(2, -1));
  q = fx_horner(tl, q, fx_constant(1 << 30, 0));
  // y = -2 ln u = w 2^E with w in [1/2, 1.01).  Next to u = 1 (ne = 0, R = 512)
  // y = -2 t q keeps its relative precision: |t| normalised, times q.
  const bool near = ne == 0 && tab.x == 512;
  fx_acc p = fx_zero();
  fx_mac(p, tl, fx_rhs(q));
  const long long lnu = (long long)ne * NFX_LN2 + tab.y - ((fx_sum(p) - (1 << 29)) >> 3);  // -ln u, 2^-57
  const uint64_t v = near ? (uint64_t)(-t62) : (uint64_t)lnu;
  const int z = __clzll((long long)v);
  fx w = fx_of_bits((long long)((v << z) >> 4));
  if (near) w = fx_times(fx_lhs(w), fx_rhs(q));
  int E = near ? 3 - z : 8 - z;
  long long wb = fx_bits(w);
  if (E & 1) {
    wb >>= 1;
    E += 1;
  }
  // s = sqrt(w): a float root, its exact remainder, and a second correction
  const float wf = (float)(int)(wb >> 30) * 0x1p-30f, ri = 0.5f * rsqrtf(wf);
  const int h0 = __float2int_rn(2.0f * wf * ri * 0x1p30f);
  const long long rho = wb - (long long)h0 * h0;            // 2^-60
  const float d1 = (float)rho * 0x1p-30f * ri;               // 2^-30
  const float dh = rintf(d1);
  const fx s1 = {(d1 - dh) * 0x1p30f, h0 + (int)dh};
  fx_acc r = fx_acc{wb, 0ull};
  fx_mac(r, fx_lhs_neg(s1), fx_rhs(s1));
  const float d2 = (float)(fx_sum(r) - (1 << 29)) * ri;      // 2^-60
  const long long s = fx_bits(fx{s1.l + d2, s1.h});
  // times 2^(E / 2) / 8 (E <= 8)
  const int sh = 4 - (E >> 1);
  return fx_of_bits(sh > 63 ? 0 : (2 * s) >> sh);
}

// sin and cos of 2 pi (k + 1/2) 2^-52.
__device__ __forceinline__ void fx_sincos(uint64_t k, fx& sn, fx& cs) {
  const uint64_t n = 2 * k + 1;  // the angle is pi n 2^-52
  const int j = (int)((n + (1ull << 45)) >> 46);
  const long long y = (long long)n - ((long long)j << 46);  // |y| <= 2^45, units of 2^-52 pi
  // th = pi y 2^-52 = (pi / 4) (4 y 2^-52), |th| < 0.025
  const fx th = fx_times(fx_lhs(fx_constant(NFX_PI_4_H, NFX_PI_4_L)), fx_rhs(fx_of_bits(y << 10)));
  const fx_left tl = fx_lhs(th);
  const fx_left t2 = fx_lhs(fx_times(tl, fx_rhs(th)));
  // sin th = th (1 - t2/6 + t2^2/120 - t2^3/5040), cos th = 1 - t2/2 + t2^2/24 - t2^3/720 + t2^4/40320
  fx s = fx_one_over(5040, -1), c = fx_one_over(40320, 1);
  c = fx_horner(t2, c, fx_one_over(720, -1));
  s = fx_horner(t2, s, fx_one_over(120, 1));
  c = fx_horner(t2, c, fx_one_over(24, 1));
  s = fx_horner(t2, s, fx_one_over(6, -1));
  c = fx_horner(t2, c, fx_one_over(2, -1));
  s = fx_horner(t2, s, fx_constant(1 << 30, 0));
  c = fx_horner(t2, c, fx_constant(1 << 30, 0));
  const fx_right sr = fx_rhs(fx_times(tl, fx_rhs(s))), cr = fx_rhs(c);
  const int4 tab = __ldg(&NFX_SC_TAB[j]);
  const fx S = {(float)tab.x, tab.y}, C = {(float)tab.z, tab.w};
  fx_acc a = fx_zero(), b = fx_zero();
  fx_mac(a, fx_lhs(S), cr);
  fx_mac(a, fx_lhs(C), sr);
  fx_mac(b, fx_lhs(C), cr);
  fx_mac(b, fx_lhs_neg(S), sr);
  sn = fx_split(fx_sum(a));
  cs = fx_split(fx_sum(b));
}

// Pair j of the normal numbers of normals_f64, divided by 8.
__device__ __forceinline__ void normal_pair_fx(fx& g0, fx& g1, uint64_t seed, uint32_t step, uint32_t site, uint32_t slot,
                                               uint32_t stream, uint32_t j) {
  const uint4 w = philox_words(seed, step, site, slot, stream, j);
  const uint64_t k1 = ((uint64_t)(w.x >> 6) << 26) | (w.y >> 6), k2 = ((uint64_t)(w.z >> 6) << 26) | (w.w >> 6);
  const fx_left r = fx_lhs(fx_radius(k1));
  fx s, c;
  fx_sincos(k2, s, c);
  g0 = fx_times(r, fx_rhs(c));
  g1 = fx_times(r, fx_rhs(s));
}
template <int NP>
__device__ __forceinline__ void normals_fx(fx* g, uint64_t seed, uint32_t step, uint32_t site, uint32_t slot,
                                           uint32_t stream) {
#pragma unroll
  for (int j = 0; j < NP; ++j) normal_pair_fx(g[2 * j], g[2 * j + 1], seed, step, site, slot, stream, (uint32_t)j);
}

}  // namespace clgc
