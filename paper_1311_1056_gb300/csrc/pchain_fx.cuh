// pchain_fx.cuh -- the 2x2 complex algebra of the SU(2) chain (pchain.cu) in
// fixed point (fixed.cuh): the Langevin update and the cooling sweep of one
// link per thread.
//
// Why: a chain's block is a warp or a few, so its time is that of one warp's
// FP64 instructions, 64 cycles each (~2,600 of them in a step with five
// sweeps).  A 2x2 product is ~350 cycles here against 2,048, a term of a power
// series 100 against 640.  512 chains of 30 links, 8 steps of up to 5 sweeps:
// 0.74 ms in FP64, 0.35 ms here (with the cyclic products by doubling), now a
// lone warp's latency: 15,000 instructions a step at 4 cycles each.  The functions return false when a number leaves the
// range; nothing has been written by then and the caller redoes that part of
// the step in FP64.
#pragma once
#include "expm_fx.cuh"
#include "noise_fx.cuh"

namespace clgc {

struct F2 {
  cx<fx> e[4];  // row-major
};

// n 2x2 matrices in shared memory, component-major (one 8-byte word a number).
struct SF2 {
  int2* p;
  int n;
  __device__ __forceinline__ fx word(int q, int k) const {
    const int2 v = p[q * n + k];
    return fx{__int_as_float(v.x), v.y};
  }
  __device__ __forceinline__ void word(int q, int k, fx a) const { p[q * n + k] = make_int2(__float_as_int(a.l), a.h); }
  __device__ __forceinline__ F2 get(int k) const {
    F2 r;
#pragma unroll
    for (int q = 0; q < 4; ++q) r.e[q] = cx<fx>{word(2 * q, k), word(2 * q + 1, k)};
    return r;
  }
  __device__ __forceinline__ void set(int k, const F2& m) const {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      word(2 * q, k, m.e[q].re);
      word(2 * q + 1, k, m.e[q].im);
    }
  }
};

// 2^S a b, entries within bounds or ck set (S <= 2: windows of links held as
// 2^-S times their value).
template <bool SCALED>
__device__ __forceinline__ F2 f2_mul(const F2& a, const F2& b, int S, fx_chk& ck) {
  F2 r;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const fx_cleft x0 = fx_lhs(a.e[2 * i]), x1 = fx_lhs(a.e[2 * i + 1]);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      fx_acc s[2] = {fx_zero(), fx_zero()};
      fx_cmac(s[0], s[1], x0, fx_rhs(b.e[j]));
      fx_cmac(s[0], s[1], x1, fx_rhs(b.e[2 + j]));
      if (SCALED) {
        fx v[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const long long t = fx_sum(s[h]) - (1 << 29);
          if ((unsigned)((int)(t >> 32) + (0x17000000 >> S)) >= (0x2E000000u >> S)) ck.fail();
          v[h] = fx_of_bits(t << S);
        }
        r.e[2 * i + j] = cx<fx>{v[0], v[1]};
      } else {
        r.e[2 * i + j] = fx_get<FX_WIDE>(s[0], s[1], ck);
      }
    }
  }
  return r;
}

// 1 / ((2j - 1) 2j) and 1 / (2j (2j + 1)): the ratios of the terms of cosh and
// of sinh(s) / s.
#define PC_R(d) fx_split_const(((1ll << 60) + (d) / 2) / (d))
__constant__ fx_const c_pc_cosh[12] = {PC_R(2),   PC_R(2),   PC_R(12),  PC_R(30),  PC_R(56),  PC_R(90),
                                       PC_R(132), PC_R(182), PC_R(240), PC_R(306), PC_R(380), PC_R(462)};
__constant__ fx_const c_pc_sinh[12] = {PC_R(6),   PC_R(6),   PC_R(20),  PC_R(42),  PC_R(72),  PC_R(110),
                                       PC_R(156), PC_R(210), PC_R(272), PC_R(342), PC_R(420), PC_R(506)};
#undef PC_R
// Terms (of s^2j / (2j)!, j = 1 ..) that leave a remainder below 2^-61.
__device__ __forceinline__ int pc_terms(float s2) {
  return s2 < 0x1p-18f ? 2 : s2 < 0x1p-10f ? 4 : s2 < 0x1p-4f ? 6 : s2 < 0.25f ? 8 : 11;
}
__device__ __forceinline__ float fx_approx(fx a) { return (float)a.h * 0x1p-30f; }
__device__ __forceinline__ float pc_warp_max(float x) {  // x >= 0
  return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(x)));
}
// x <- s2 r (1 + x), r real
__device__ __forceinline__ void pc_term(cx<fx>& x, const fx_cleft& s2, fx_const r, fx_chk& ck) {
  const fx_left rl = fx_lhs(fx{(float)r.l, r.h});
  fx_acc re = fx_acc{mad_wide(r.h, 1 << 30, (long long)r.l), 0ull}, im = fx_zero();
  fx_mac(re, rl, fx_rhs(x.re));
  fx_mac(im, rl, fx_rhs(x.im));
  const fx_cright u = {fx_rhs(fx_split(fx_sum(re))), fx_rhs(fx_split(fx_sum(im)))};
  re = im = fx_zero();
  fx_cmac(re, im, s2, u);
  x = fx_get<FX_WIDE>(re, im, ck);
}
__device__ __forceinline__ void pc_term(fx& x, const fx_left& s2, fx_const r, fx_chk& ck) {
  fx_acc u = fx_acc{mad_wide(r.h, 1 << 30, (long long)r.l), 0ull};
  fx_mac(u, fx_lhs(fx{(float)r.l, r.h}), fx_rhs(x));
  fx_acc v = fx_zero();
  fx_mac(v, s2, fx_rhs(fx_split(fx_sum(u))));
  x = fx_get<FX_WIDE>(v, ck);
}

// The Langevin step's constants: -eps beta, and sqrt(2 eps) 8 2^-E.
struct PcStepFx {
  long long mb[2];
  fx sq;
  int E;
  bool ok;
};
__device__ __forceinline__ PcStepFx pc_step_fx(double mbr, double mbi, double sq) {
  PcStepFx c;
  unsigned mag = 0;
  c.mb[0] = fx_bits_of_double(mbr, mag);
  c.mb[1] = fx_bits_of_double(mbi, mag);
  const bool mb_ok = mag < 0x3FD70000u;  // 0.359375: four times it stays in bounds
  c.E = 0;
  double s = 8.0 * sq;
  while (s >= 1.4 && c.E < 2) {
    s *= 0.5;
    ++c.E;
  }
  mag = 0;
  c.sq = fx_of_double(s, mag);
  c.ok = mb_ok && fx_mag_ok(mag);
  return c;
}

// W = exp(A) U / sqrt(det), A = 2^S mb (P - Tr P / 2) + i sq g_a sigma_a, g
// the normal numbers over 8; P is 2^-S times the cyclic product.
__device__ __forceinline__ F2 pc_update_fx(const F2& P, int S, const F2& U, const fx* g, const PcStepFx& c, fx_chk& ck) {
  const fx_cleft mb = fx_lhs(cx<fx>{fx_of_bits(c.mb[0] << S), fx_of_bits(c.mb[1] << S)});
  long long nz[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) nz[q] = fx_bits(fx_times(fx_lhs(c.sq), fx_rhs(g[q]))) << c.E;
  const cx<fx> d = {fx_of_bits((fx_bits(P.e[0].re) - fx_bits(P.e[3].re)) >> 1),
                    fx_of_bits((fx_bits(P.e[0].im) - fx_bits(P.e[3].im)) >> 1)};
  // A = [[a0, a1], [a2, -a0]]; i sigma_a g_a = [[i g3, g2 + i g1], [-g2 + i g1, -i g3]]
  fx_acc re = fx_zero(), im = fx_acc{nz[2], 0ull};
  fx_cmac(re, im, mb, fx_rhs(d));
  const cx<fx> a0 = fx_get<FX_WIDE>(re, im, ck);
  re = fx_acc{nz[1], 0ull}, im = fx_acc{nz[0], 0ull};
  fx_cmac(re, im, mb, fx_rhs(P.e[1]));
  const cx<fx> a1 = fx_get<FX_WIDE>(re, im, ck);
  re = fx_acc{-nz[1], 0ull}, im = fx_acc{nz[0], 0ull};
  fx_cmac(re, im, mb, fx_rhs(P.e[2]));
  const cx<fx> a2 = fx_get<FX_WIDE>(re, im, ck);
  // s^2 = -det A; C = cosh(s) - 1, H = sinh(s) / s - 1
  re = im = fx_zero();
  fx_cmac(re, im, fx_lhs(a0), fx_rhs(a0));
  fx_cmac(re, im, fx_lhs(a1), fx_rhs(a2));
  const cx<fx> s2 = fx_get<FX_WIDE>(re, im, ck);
  const fx_cleft sl = fx_lhs(s2);
  cx<fx> C = {fx{0.0f, 0}, fx{0.0f, 0}}, H = C;
#pragma unroll 1
  for (int j = pc_terms(pc_warp_max(fabsf(fx_approx(s2.re)) + fabsf(fx_approx(s2.im)))); j >= 1; --j) {
    pc_term(C, sl, c_pc_cosh[j], ck);
    pc_term(H, sl, c_pc_sinh[j], ck);
  }
  // X = exp(A) - 1, W = U + X U
  F2 X;
  const fx_cleft hl = fx_lhs(H);
  re = fx_from(C.re + a0.re), im = fx_from(C.im + a0.im);
  fx_cmac(re, im, hl, fx_rhs(a0));
  X.e[0] = fx_get<FX_WIDE>(re, im, ck);
  re = fx_from(C.re - a0.re), im = fx_from(C.im - a0.im);
  fx_cmac(re, im, fx_lhs_neg(H), fx_rhs(a0));
  X.e[3] = fx_get<FX_WIDE>(re, im, ck);
  re = fx_from(a1.re), im = fx_from(a1.im);
  fx_cmac(re, im, hl, fx_rhs(a1));
  X.e[1] = fx_get<FX_WIDE>(re, im, ck);
  re = fx_from(a2.re), im = fx_from(a2.im);
  fx_cmac(re, im, hl, fx_rhs(a2));
  X.e[2] = fx_get<FX_WIDE>(re, im, ck);
  F2 W;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const fx_cleft x0 = fx_lhs(X.e[2 * i]), x1 = fx_lhs(X.e[2 * i + 1]);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      re = fx_from(U.e[2 * i + j].re), im = fx_from(U.e[2 * i + j].im);
      fx_cmac(re, im, x0, fx_rhs(U.e[j]));
      fx_cmac(re, im, x1, fx_rhs(U.e[2 + j]));
      W.e[2 * i + j] = fx_get<FX_WIDE>(re, im, ck);
    }
  }
  // W <- W (1 + y), y = (1 + dl)^(-1/2) - 1 = -dl / 2 + 3 dl^2 / 8 for dl = det W - 1 below 2^-20
  re = fx_acc{-(1ll << 60), 0ull}, im = fx_zero();
  fx_cmac(re, im, fx_lhs(W.e[0]), fx_rhs(W.e[3]));
  fx_cmac(re, im, fx_lhs_neg(W.e[1]), fx_rhs(W.e[2]));
  const cx<fx> dl = fx_get<FX_WIDE>(re, im, ck);
  if (max(abs(dl.re.h), abs(dl.im.h)) >= 1 << 10) ck.fail();
  const float dr = fmaf(dl.re.l, 0x1p-30f, (float)dl.re.h), di = fmaf(dl.im.l, 0x1p-30f, (float)dl.im.h);  // 2^-30
  const cx<fx> y = {fx_of_bits((long long)rintf(0.375f * (dr * dr - di * di)) - (fx_bits(dl.re) >> 1)),
                    fx_of_bits((long long)rintf(0.75f * dr * di) - (fx_bits(dl.im) >> 1))};
  const fx_cleft yl = fx_lhs(y);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    re = fx_from(W.e[q].re), im = fx_from(W.e[q].im);
    fx_cmac(re, im, yl, fx_rhs(W.e[q]));
    W.e[q] = fx_get<FX_WIDE>(re, im, ck);
  }
  return W;
}

// The cooling gradient of link k (u) with its predecessor w: G = u u^+ - w^+ w,
// g = { Re G01, -Im G01, (G00 - G11) / 2 } (f_a / 4), t = (Tr u u^+ / 2 - 1) 2^61.
__device__ __forceinline__ float f2_norm2(const F2& u) {
  float s = 0.0f;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float x = fx_approx(u.e[q].re), y = fx_approx(u.e[q].im);
    s = fmaf(x, x, fmaf(y, y, s));
  }
  return s;
}
__device__ __forceinline__ void fx_abs2(fx_acc& s, cx<fx> a) {
  fx_mac(s, fx_lhs(a.re), fx_rhs(a.re));
  fx_mac(s, fx_lhs(a.im), fx_rhs(a.im));
}
// s += conj(a) b or s += a conj(b) (re and im)
__device__ __forceinline__ void fx_conj_mac(fx_acc& re, fx_acc& im, cx<fx> a, cx<fx> b) {
  const fx_left ar = fx_lhs(a.re), ai = fx_lhs(a.im), nai = fx_lhs_neg(a.im);
  const fx_right br = fx_rhs(b.re), bi = fx_rhs(b.im);
  fx_mac(re, ar, br);
  fx_mac(re, ai, bi);
  fx_mac(im, ar, bi);
  fx_mac(im, nai, br);
}
__device__ __forceinline__ void pc_grad_fx(const F2& u, const F2& w, fx g[3], long long& t, fx_chk& ck) {
  // sums of squares stay below 4 (and the sixteen products of G01 with them): no wrap
  if (!(f2_norm2(u) < 3.9f)) ck.fail();
  fx_acc r0 = fx_zero(), r1 = fx_zero(), c0 = fx_zero(), c1 = fx_zero();
  fx_abs2(r0, u.e[0]);
  fx_abs2(r0, u.e[1]);
  fx_abs2(r1, u.e[2]);
  fx_abs2(r1, u.e[3]);
  fx_abs2(c0, w.e[0]);
  fx_abs2(c0, w.e[2]);
  fx_abs2(c1, w.e[1]);
  fx_abs2(c1, w.e[3]);
  const long long a = fx_sum(r0) - (1 << 29), b = fx_sum(r1) - (1 << 29);
  t = a + b - (1ll << 61);
  const long long df = (a - b - (fx_sum(c0) - fx_sum(c1))) >> 1;
  ck.see<FX_WIDE>((int)(df >> 32));
  g[2] = fx_of_bits(df);
  // G01 = u00 conj(u10) + u01 conj(u11) - conj(w00) w01 - conj(w10) w11
  fx_acc re = fx_zero(), im = fx_zero(), wr = fx_zero(), wi = fx_zero();
  fx_conj_mac(re, im, u.e[2], u.e[0]);
  fx_conj_mac(re, im, u.e[3], u.e[1]);
  fx_conj_mac(wr, wi, w.e[0], w.e[1]);
  fx_conj_mac(wr, wi, w.e[2], w.e[3]);
  const long long x = fx_sum(re) - fx_sum(wr), y = fx_sum(wi) - fx_sum(im);
  ck.see<FX_WIDE>((int)(x >> 32));
  ck.see<FX_WIDE>((int)(y >> 32));
  g[0] = fx_of_bits(x);
  g[1] = fx_of_bits(y);
}

// exp(h_a sigma_a), h = s g: the entries {00, 11, Re 01, Im 10}.
__device__ __forceinline__ void pc_omega_fx(fx om[4], const fx g[3], fx s, fx_chk& ck) {
  fx h[3];
  fx_acc r = fx_zero();
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    fx_acc v = fx_zero();
    fx_mac(v, fx_lhs(s), fx_rhs(g[q]));
    h[q] = fx_get<FX_WIDE>(v, ck);
    fx_mac(r, fx_lhs(h[q]), fx_rhs(h[q]));
  }
  const fx r2 = fx_get<FX_WIDE>(r, ck);
  const fx_left rl = fx_lhs(r2);
  fx C = {0.0f, 0}, H = C;
#pragma unroll 1
  for (int j = pc_terms(pc_warp_max(fabsf(fx_approx(r2)))); j >= 1; --j) {
    pc_term(C, rl, c_pc_cosh[j], ck);
    pc_term(H, rl, c_pc_sinh[j], ck);
  }
  const fx_left hl = fx_lhs(H);
  fx x[3];  // sinh(r) / r h
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    fx_acc v = fx_from(h[q]);
    fx_mac(v, hl, fx_rhs(h[q]));
    x[q] = fx_get<FX_WIDE>(v, ck);
  }
  fx_acc v = fx_acc{1ll << 60, 0ull};
  v.a += fx_bits(C) + fx_bits(x[2]);
  om[0] = fx_get<FX_WIDE>(v, ck);
  v.a -= 2 * fx_bits(x[2]);
  om[1] = fx_get<FX_WIDE>(v, ck);
  om[2] = x[0];
  om[3] = x[1];
}

// om u and u om^-1 for Hermitian om of determinant one (entries as above).
struct PcOmega {
  fx_left d0, d1, b, nb, c, nc;
};
__device__ __forceinline__ PcOmega pc_omega_lhs(fx d0, fx d1, fx b, fx c) {
  return PcOmega{fx_lhs(d0), fx_lhs(d1), fx_lhs(b), fx_lhs_neg(b), fx_lhs(c), fx_lhs_neg(c)};
}
__device__ __forceinline__ cx<fx> pc_row(const fx_left& d, cx<fx> u, const fx_left& br, const fx_left& bi, const fx_left& nbi,
                                         cx<fx> v, fx_chk& ck) {  // d u + (br + i bi) v
  const fx_cright y = fx_rhs(v), x = fx_rhs(u);
  fx_acc re = fx_zero(), im = fx_zero();
  fx_mac(re, d, x.re);
  fx_mac(im, d, x.im);
  fx_mac(re, br, y.re);
  fx_mac(im, br, y.im);
  fx_mac(re, nbi, y.im);
  fx_mac(im, bi, y.re);
  return fx_get<FX_WIDE>(re, im, ck);
}
__device__ __forceinline__ F2 pc_apply_fx(const fx om[4], const F2& u, const fx on[4], fx_chk& ck) {
  F2 t, r;
  {  // [[d0, b - i c], [b + i c, d1]] u
    const PcOmega o = pc_omega_lhs(om[0], om[1], om[2], om[3]);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      t.e[j] = pc_row(o.d0, u.e[j], o.b, o.nc, o.c, u.e[2 + j], ck);
      t.e[2 + j] = pc_row(o.d1, u.e[2 + j], o.b, o.c, o.nc, u.e[j], ck);
    }
  }
  {  // t [[d1, -b + i c], [-b - i c, d0]]
    const PcOmega o = pc_omega_lhs(on[0], on[1], on[2], on[3]);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      r.e[2 * i] = pc_row(o.d1, t.e[2 * i], o.nb, o.nc, o.c, t.e[2 * i + 1], ck);
      r.e[2 * i + 1] = pc_row(o.d0, t.e[2 * i + 1], o.nb, o.c, o.nc, t.e[2 * i], ck);
    }
  }
  return r;
}

}  // namespace clgc
