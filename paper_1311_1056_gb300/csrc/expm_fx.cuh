// expm_fx.cuh -- the CL update's exponential and re-projection in fixed point
// (fixed.cuh): exp(A) of a traceless A by the Cayley-Hamilton reduction of
// expm.cuh, for the FP64 form (through the whole update) and the FP32-storage
// form (whose exponential is rounded to float).
#pragma once
#include "expm.cuh"
#include "fixed.cuh"

namespace clgc {

// 1 / n! in units of 2^-60, rounded, as high and (balanced) low limb.
struct fx_const {
  int h, l;
};
__host__ __device__ constexpr long long fx_inv_factorial(int n) {
  long long f = 1;
  for (int k = 2; k <= n && k < 20; ++k) f *= k;
  return n > 19 ? 0 : ((1ll << 60) + f / 2) / f;
}
__host__ __device__ constexpr fx_const fx_split_const(long long v) {
  const long long h = (v + (1ll << 29)) >> 30;
  return fx_const{(int)h, (int)(v - (h << 30))};
}
#define FX_F(n) fx_split_const(fx_inv_factorial(n))
__constant__ fx_const c_fx_invfact[28] = {FX_F(0),  FX_F(1),  FX_F(2),  FX_F(3),  FX_F(4),  FX_F(5),  FX_F(6),
                                          FX_F(7),  FX_F(8),  FX_F(9),  FX_F(10), FX_F(11), FX_F(12), FX_F(13),
                                          FX_F(14), FX_F(15), FX_F(16), FX_F(17), FX_F(18), FX_F(19), FX_F(20),
                                          FX_F(20), FX_F(20), FX_F(20), FX_F(20), FX_F(20), FX_F(20), FX_F(20)};
#undef FX_F
__device__ __forceinline__ fx_acc fx_from_invfact(int n) {
  const fx_const c = c_fx_invfact[n];
  return fx_acc{mad_wide(c.h, 1 << 30, (long long)c.l), 0ull};
}
__device__ __forceinline__ fx fx_third() {
  const fx_const c = fx_split_const(((1ll << 60) + 1) / 3);
  return fx{(float)c.l, c.h};
}
template <int B>
__device__ __forceinline__ cx<fx> fx_get(const fx_acc& re, const fx_acc& im, fx_chk& ck) {
  return cx<fx>{fx_get<B>(re, ck), fx_get<B>(im, ck)};
}

// Frobenius norm, to float precision.
__device__ __forceinline__ float fx_norm(const mat<fx>& a) {
  float s = 0.0f;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const float x = fmaf(a.e[k].re.l, 0x1p-30f, (float)a.e[k].re.h), y = fmaf(a.e[k].im.l, 0x1p-30f, (float)a.e[k].im.h);
    s = fmaf(x, x, fmaf(y, y, s));
  }
  return sqrtf(s) * 0x1p-30f;
}

// A <- exp(A), r = ||A||_F.  Arguments above 0.8 are halved until below and the
// result squared; false beyond 6.4 or when a number leaves the range.
__device__ __forceinline__ bool fx_expm_traceless(mat<fx>& A, float r, float tol) {
  fx_chk ck;
  int s = 0;
  while (r > 0.8f && s < 3) {
    r *= 0.5f;
    ++s;
  }
  if (!(r <= 0.8f)) return false;
  if (s > 0) {
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      A.e[k].re = fx_of_bits(fx_bits(A.e[k].re) >> s);
      A.e[k].im = fx_of_bits(fx_bits(A.e[k].im) >> s);
    }
  }
  mat<fx> Q = A;
  fx_mul_left<FX_WIDE>(Q, A, ck);  // A^2
  // c1 = Tr A^2 / 2, c0 = Tr A^3 / 3
  const cx<fx> c1 = {fx_of_bits((fx_bits(Q.e[0].re) + fx_bits(Q.e[4].re) + fx_bits(Q.e[8].re)) >> 1),
                     fx_of_bits((fx_bits(Q.e[0].im) + fx_bits(Q.e[4].im) + fx_bits(Q.e[8].im)) >> 1)};
  cx<fx> c0;
  {
    fx_acc re = fx_zero(), im = fx_zero();
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int k = 0; k < 3; ++k) fx_cmac(re, im, fx_lhs(Q.e[3 * i + k]), fx_rhs(A.e[3 * k + i]));
    const cx<fx> t = fx_get<FX_WIDE>(re, im, ck);
    const fx_left third = fx_lhs(fx_third());
    re = im = fx_zero();
    fx_mac(re, third, fx_rhs(t.re));
    fx_mac(im, third, fx_rhs(t.im));
    c0 = fx_get<FX_WIDE>(re, im, ck);
  }
  const fx_cright b0 = fx_rhs(c0), b1 = fx_rhs(c1);
  const int N = taylor_terms(r, tol);
  const fx_const f = c_fx_invfact[N];
  cx<fx> a = {fx{(float)f.l, f.h}, fx{0.0f, 0}}, b = {fx{0.0f, 0}, fx{0.0f, 0}}, c = b;
#pragma unroll 1
  for (int k = N - 1; k >= 0; --k) {
    const fx_cleft x = fx_lhs(c);
    fx_acc ar = fx_from_invfact(k), ai = fx_zero(), br = fx_from(a.re), bi = fx_from(a.im);
    fx_cmac(ar, ai, x, b0);
    fx_cmac(br, bi, x, b1);
    c = b;
    b = fx_get<FX_WIDE>(br, bi, ck);
    a = fx_get<FX_WIDE>(ar, ai, ck);
  }
  const fx_cleft lb = fx_lhs(b), lc = fx_lhs(c);
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    fx_acc re = k % 4 == 0 ? fx_from(a.re) : fx_zero(), im = k % 4 == 0 ? fx_from(a.im) : fx_zero();
    fx_cmac(re, im, lb, fx_rhs(A.e[k]));
    fx_cmac(re, im, lc, fx_rhs(Q.e[k]));
    A.e[k] = fx_get<FX_WIDE>(re, im, ck);
  }
#pragma unroll 1
  for (int i = 0; i < s; ++i) {
    Q = A;
    fx_mul_left<FX_WIDE>(A, Q, ck);
  }
  return !ck.bad();
}

// det a - 1.
__device__ __forceinline__ cx<fx> fx_det_minus_one(const mat<fx>& a, fx_chk& ck) {
  fx_acc re = fx_acc{-(1ll << 60), 0ull}, im = fx_zero();
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const int j1 = (j + 1) % 3, j2 = (j + 2) % 3;
    fx_acc cr = fx_zero(), ci = fx_zero();
    fx_cmac(cr, ci, fx_lhs(a.e[3 + j1]), fx_rhs(a.e[6 + j2]));
    fx_cmac(cr, ci, fx_lhs_neg(a.e[3 + j2]), fx_rhs(a.e[6 + j1]));
    fx_cmac(re, im, fx_lhs(a.e[j]), fx_rhs(fx_get<FX_WIDE>(cr, ci, ck)));
  }
  return fx_get<FX_WIDE>(re, im, ck);
}

// Floats to and from fixed point.  |x| < 2; exact but for what lies below 2^-60.
__device__ __forceinline__ fx fx_of_float(float x) {
  const float y = x * 0x1p30f;
  const int h = __float2int_rn(y);
  return fx{(y - (float)h) * 0x1p30f, h};
}
// Rounded once (the high limb's own rounding is made good by its remainder).
__device__ __forceinline__ float fx_to_float(fx a) {
  const float hi = (float)a.h;
  const float rem = (float)(a.h - __float2int_rn(hi));
  return fmaf(fmaf(a.l, 0x1p-30f, rem), 0x1p-30f, hi * 0x1p-30f);
}

}  // namespace clgc
