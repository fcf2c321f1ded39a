// cool_fx.cuh -- the cooling sweeps of the FP64 form in fixed point
// (fixed.cuh): gradient, Omega and apply, the formulas of kernels.cu.
//
// A cooling call keeps the links as fixed-point words Ux in the lattice's
// second link buffer: its first gradient reads the links and writes them, every
// sweep reads and writes Ux, and the last apply writes the links back.
// (Converting 64-bit words both ways in every sweep would cost two fifths of
// it.)  Omega and Omega^{-1} are packed Hermitian fields of 9 words per site.  A
// link, Omega or f that leaves the fixed-point range is stored as doubles
// (fixed.cuh) and the threads that meet it work in FP64.
#pragma once
#include "expm_fx.cuh"
#include "fixed.cuh"
#include "lattice.cuh"
#include "launch.h"

namespace clgc {

// ---------------------------------------------------------- packed fields
struct fx_herm {
  fx d[3];
  cx<fx> o[3];  // 01, 02, 12
};
__device__ __forceinline__ fx fx_word(int2 w) { return fx{__int_as_float(w.x), w.y}; }
__device__ __forceinline__ void fx_unpack_herm(fx_herm& h, const int2* v, fx_chk& ck) {
  fx w[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) w[k] = fx_word(v[k]);
  if (fx_is_raw(w[0].l)) ck.fail();
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    h.d[k] = w[k];
    h.o[k] = cx<fx>{w[3 + 2 * k], w[4 + 2 * k]};
  }
}
__device__ __forceinline__ void fx_load_herm(fx_herm& h, const int2* __restrict__ P, int s, int V, fx_chk& ck) {
  int2 v[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) v[k] = __ldg(P + (size_t)k * V + s);
  fx_unpack_herm(h, v, ck);
}
__device__ __forceinline__ void fx_store_herm(int2* P, int s, int V, const fx_herm& h) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    P[(size_t)k * V + s] = make_int2(__float_as_int(h.d[k].l), h.d[k].h);
    P[(size_t)(3 + 2 * k) * V + s] = make_int2(__float_as_int(h.o[k].re.l), h.o[k].re.h);
    P[(size_t)(4 + 2 * k) * V + s] = make_int2(__float_as_int(h.o[k].im.l), h.o[k].im.h);
  }
}
// FP32-storage form: the packed field of floats.
__device__ __forceinline__ void fx_store_herm(float* P, int s, int V, const fx_herm& h) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    P[(size_t)k * V + s] = fx_to_float(h.d[k]);
    P[(size_t)(3 + 2 * k) * V + s] = fx_to_float(h.o[k].re);
    P[(size_t)(4 + 2 * k) * V + s] = fx_to_float(h.o[k].im);
  }
}
// The general path's packed fields: doubles in, doubles out.
struct tagged_herm {
  int2* p;
};
__device__ __forceinline__ void store_herm(tagged_herm f, int s, int V, const herm& h) {
  const double w[9] = {h.d0, h.d1, h.d2, h.o01.re, h.o01.im, h.o02.re, h.o02.im, h.o12.re, h.o12.im};
#pragma unroll
  for (int k = 0; k < 9; ++k) f.p[(size_t)k * V + s] = k == 0 ? fx_raw_first(w[0]) : make_int2(__double2loint(w[k]), __double2hiint(w[k]));
}
__device__ __forceinline__ void load_herm_mat(mat<double>& m, tagged_herm f, int s, int V) {
  double w[9];
  const bool raw = fx_is_raw(__int_as_float(f.p[s].x));
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const int2 v = f.p[(size_t)k * V + s];
    w[k] = !raw ? fx_to_double(fx_word(v)) : k == 0 ? fx_raw_first(v) : __hiloint2double(v.y, v.x);
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) m.e[4 * k] = cx<double>{w[k], 0.0};
  m.e[1] = cx<double>{w[3], w[4]};
  m.e[3] = cx<double>{w[3], -w[4]};
  m.e[2] = cx<double>{w[5], w[6]};
  m.e[6] = cx<double>{w[5], -w[6]};
  m.e[5] = cx<double>{w[7], w[8]};
  m.e[7] = cx<double>{w[7], -w[8]};
}

// -------------------------------------------------------------- gradient
// G_x = sum_mu (U U^+ - U^+_{x-mu} U_{x-mu}) as 60-bit integers: diagonal, and
// re / im of 01, 02, 12.
struct fx_gradient {
  long long d[3], o[6];  // times 2^-e, below one
  int e, wild;           // wild: e, where it comes from links beyond the bound
};
// rows (or conjugated columns) r0, r1, r2 of one link: += sign r_i conj(r_j); n: their squares in float
__device__ __forceinline__ void fx_outer(fx_acc* D, fx_acc* O, float* n, cx<fx> r0, cx<fx> r1, cx<fx> r2, bool neg) {
  const cx<fx> r[3] = {r0, r1, r2};
  fx_cright R[3];
  fx_cleft X[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    R[i] = fx_rhs(r[i]);
    X[i] = neg ? fx_lhs_neg(r[i]) : fx_lhs(r[i]);
    fx_mac(D[i], X[i].re, R[i].re);
    fx_mac(D[i], X[i].im, R[i].im);
    const float a = (float)r[i].re.h, b = (float)r[i].im.h;
    n[i] = fmaf(a, a, fmaf(b, b, n[i]));
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) {  // (0,1), (0,2), (1,2)
    const int i = q < 2 ? 0 : 1, j = q == 0 ? 1 : 2;
    // x conj(y): re x.re y.re + x.im y.im, im x.im y.re - x.re y.im
    fx_mac(O[2 * q], X[i].re, R[j].re);
    fx_mac(O[2 * q], X[i].im, R[j].im);
    fx_mac(O[2 * q + 1], X[i].im, R[j].re);
    const fx_left nre = {-X[i].re.h, fx_neg(X[i].re.p)};
    fx_mac(O[2 * q + 1], nre, R[j].im);
  }
}
// ----------------------------------------------------------- exponential
// exp(H), or exp(-H), of a traceless Hermitian H, as expm_hermitian_pair: H^2,
// the two invariants, Horner's rule on the Cayley-Hamilton coefficients, in
// fixed point.  (One sign: two threads share a site's pair.)  False when a
// number leaves the range: |H|_F above 0.34.  Both signs agree on that: they see
// the same numbers up to the test of |H|, and below it no coefficient and no
// entry of the result can exceed exp(0.34) < 1.4375.
struct fx_exp_series {  // what both signs share
  fx_herm Q;            // H^2
  fx c0, c1;            // det H, Tr H^2 / 2
  int N;                // terms
};
__device__ __forceinline__ bool fx_exp_setup(fx_exp_series& S, const fx_herm& H, float tol) {
  fx_chk ck;
  fx_herm& Q = S.Q;
  {
    fx_cleft L[3];
    fx_cright R[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      L[q] = fx_lhs(H.o[q]);
      R[q] = fx_rhs(H.o[q]);
    }
    // |o01|^2, |o02|^2, |o12|^2 into the two diagonals each belongs to
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      fx_acc a = fx_zero();
      fx_mac(a, fx_lhs(H.d[i]), fx_rhs(H.d[i]));
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const int qi = q < 2 ? 0 : 1, qj = q == 0 ? 1 : 2;
        if (qi != i && qj != i) continue;
        fx_mac(a, L[q].re, R[q].re);
        fx_mac(a, L[q].im, R[q].im);
      }
      Q.d[i] = fx_get<FX_WIDE>(a, ck);
    }
    // (H^2)_01 = (d0 + d1) o01 + o02 conj(o12), _02 = (d0 + d2) o02 + o01 o12,
    // _12 = (d1 + d2) o12 + conj(o01) o02; d_i + d_j = -d_k
    fx_acc re, im;
    fx_left nd = fx_lhs(-H.d[2]);
    re = im = fx_zero();
    fx_mac(re, nd, R[0].re);
    fx_mac(im, nd, R[0].im);
    fx_mac(re, L[1].re, R[2].re);
    fx_mac(re, L[1].im, R[2].im);
    fx_mac(im, L[1].im, R[2].re);
    fx_mac(im, fx_lhs_neg(H.o[1].re), R[2].im);
    Q.o[0] = cx<fx>{fx_get<FX_WIDE>(re, ck), fx_get<FX_WIDE>(im, ck)};
    nd = fx_lhs(-H.d[1]);
    re = im = fx_zero();
    fx_mac(re, nd, R[1].re);
    fx_mac(im, nd, R[1].im);
    fx_cmac(re, im, L[0], R[2]);
    Q.o[1] = cx<fx>{fx_get<FX_WIDE>(re, ck), fx_get<FX_WIDE>(im, ck)};
    nd = fx_lhs(-H.d[0]);
    re = im = fx_zero();
    fx_mac(re, nd, R[2].re);
    fx_mac(im, nd, R[2].im);
    fx_mac(re, L[0].re, R[1].re);
    fx_mac(re, L[0].im, R[1].im);
    fx_mac(im, L[0].re, R[1].im);
    fx_mac(im, L[0].nim, R[1].re);
    Q.o[2] = cx<fx>{fx_get<FX_WIDE>(re, ck), fx_get<FX_WIDE>(im, ck)};
  }
  // c1 = Tr H^2 / 2, c0 = det H = Tr H^3 / 3 = (sum_i Q_ii d_i + 2 Re sum Q_ij conj(o_ij)) / 3
  // Tr H^2 / 2 in 64 bits: as a number it would wrap at 2 and pass for a small one
  const long long h2 = (fx_bits(Q.d[0]) + fx_bits(Q.d[1]) + fx_bits(Q.d[2])) >> 1;
  if (ck.bad() || h2 > (1ll << 56)) return false;  // |H|_F above 0.354
  const fx c1 = fx_of_bits(h2);
  fx_acc t = fx_zero(), t2 = fx_zero();
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    fx_mac(t, fx_lhs(Q.d[i]), fx_rhs(H.d[i]));
    fx_mac(t2, fx_lhs(Q.o[i].re), fx_rhs(H.o[i].re));
    fx_mac(t2, fx_lhs(Q.o[i].im), fx_rhs(H.o[i].im));
  }
  const fx t3 = fx_of_bits(fx_sum(t) + 2 * (fx_sum(t2) - (1 << 29)) - (1 << 29));
  fx_acc z = fx_zero();
  fx_mac(z, fx_lhs(fx_third()), fx_rhs(t3));
  const fx c0 = fx_get<FX_WIDE>(z, ck);
  const float r = sqrtf(2.0f * fmaxf(fmaf(c1.l, 0x1p-60f, (float)c1.h * 0x1p-30f), 0.0f));
  if (ck.bad() || !(r < 0.34f)) return false;
  S.c0 = c0;
  S.c1 = c1;
  S.N = taylor_terms(r, tol);
  return true;
}
// exp(H), inverse: exp(-H).  det(-H) = -det H: exp(-H) = a - b H + c H^2 with c0 negated.
__device__ __forceinline__ void fx_exp_sum(fx_herm& om, const fx_exp_series& S, const fx_herm& H, bool inverse) {
  fx_chk ck;  // nothing to check: see above
  const fx_herm& Q = S.Q;
  const int N = S.N;
  const fx_right b1 = fx_rhs(S.c1), b0 = fx_rhs(inverse ? -S.c0 : S.c0);
  const fx_const f = c_fx_invfact[N];
  fx a = {(float)f.l, f.h}, b = {0.0f, 0}, c = {0.0f, 0};
#pragma unroll 1
  for (int k = N - 1; k >= 0; --k) {
    fx_acc s = fx_from_invfact(k), u = fx_from(a);
    const fx_left x = fx_lhs(c);
    fx_mac(s, x, b0);
    fx_mac(u, x, b1);
    c = b;
    b = fx_get<FX_WIDE>(u, ck);
    a = fx_get<FX_WIDE>(s, ck);
  }
  const fx_left lb = fx_lhs(inverse ? -b : b), lc = fx_lhs(c);
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const int q = (k - 3) >> 1;
    const fx hk = k < 3 ? H.d[k] : (k & 1) ? H.o[q].re : H.o[q].im, qk = k < 3 ? Q.d[k] : (k & 1) ? Q.o[q].re : Q.o[q].im;
    fx_acc s = k < 3 ? fx_from(a) : fx_zero();
    fx_mac(s, lb, fx_rhs(hk));
    fx_mac(s, lc, fx_rhs(qk));
    const fx w = fx_get<FX_WIDE>(s, ck);
    if (k < 3)
      om.d[k] = w;
    else if (k & 1)
      om.o[q].re = w;
    else
      om.o[q].im = w;
  }
}

// H = 4 c (G - Tr G / 3), c = -eps alpha_ad (f_a lambda_a = 4 (G - Tr G / 3)).
// Only the product c G has to fit: c goes in as c 2^t, in [1/2, 1), and G as
// G 2^-t.  (With c itself as the factor, f >= 1.44 or c >= 0.36 sent a site and
// with it the links around it through FP64; fields of norm 1.01, where cooled
// chains live, have some such f at every other site.)
__device__ __forceinline__ int fx_strength_exponent(double c) {
  const int e = (__double2hiint(c) >> 20) & 0x7ff;
  return max(-24, min(24, 1022 - e));
}
// v 2^-n
__device__ __forceinline__ fx fx_shifted(long long v, int n, fx_chk& ck) {
  const long long w = n >= 0 ? v >> n : v << -n;
  if (n < 0 && (w >> -n) != v) ck.fail();
  ck.see<FX_WIDE>((int)(w >> 32));
  return fx_of_bits(w);
}
__device__ __forceinline__ bool fx_herm_of_gradient(fx_herm& H, const fx_gradient& G, double c) {
  fx_chk ck;
  unsigned mag = 0;
  const int t = fx_strength_exponent(4.0 * c);
  const fx_left c4 = fx_lhs(fx_of_double(fx_pow2(4.0 * c, t), mag));
  const long long third = (G.d[0] + G.d[1] + G.d[2]) / 3;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const long long v = k < 3 ? G.d[k] - third : G.o[k - 3];
    fx_acc a = fx_zero();
    fx_mac(a, c4, fx_rhs(fx_shifted(v, t - G.e, ck)));
    const fx w = fx_get<FX_WIDE>(a, ck);
    const int q = (k - 3) >> 1;
    if (k < 3)
      H.d[k] = w;
    else if (k & 1)
      H.o[q].re = w;
    else
      H.o[q].im = w;
  }
  return !ck.bad() && fx_mag_ok(mag);
}
// The same from f: H = c f_a lambda_a.
__device__ __forceinline__ fx fx_of_real(double x, int t, unsigned& mag) { return fx_of_double(fx_pow2(x, -t), mag); }
__device__ __forceinline__ fx fx_of_real(float x, int t, unsigned& mag) {
  x *= __int_as_float((127 - t) << 23);
  if (!(fabsf(x) < 1.4375f)) mag = 0xffffffffu;
  return fx_of_float(x);
}
template <typename T>
__device__ __forceinline__ bool fx_herm_of_f(fx_herm& H, const T* f, double c0) {
  fx_chk ck;
  unsigned mag = 0;
  const int t = fx_strength_exponent(c0);
  const double c = fx_pow2(c0, t);
  const fx_left cl = fx_lhs(fx_of_double(c, mag)), cn = fx_lhs(fx_of_double(-c, mag)),
                c3 = fx_lhs(fx_of_double(c * 0.57735026918962576451, mag)),
                m3 = fx_lhs(fx_of_double(-2.0 * (c * 0.57735026918962576451), mag));
  fx_right F[8];
#pragma unroll
  for (int a = 0; a < 8; ++a) F[a] = fx_rhs(fx_of_real(f[a], t, mag));
  auto one = [&](const fx_left& x, const fx_right& y) {
    fx_acc s = fx_zero();
    fx_mac(s, x, y);
    return fx_get<FX_WIDE>(s, ck);
  };
  auto two = [&](const fx_left& x, const fx_right& y, const fx_left& x2, const fx_right& y2) {
    fx_acc s = fx_zero();
    fx_mac(s, x, y);
    fx_mac(s, x2, y2);
    return fx_get<FX_WIDE>(s, ck);
  };
  H.d[0] = two(cl, F[2], c3, F[7]);
  H.d[1] = two(cn, F[2], c3, F[7]);
  H.d[2] = one(m3, F[7]);
  H.o[0] = cx<fx>{one(cl, F[0]), one(cn, F[1])};
  H.o[1] = cx<fx>{one(cl, F[3]), one(cn, F[4])};
  H.o[2] = cx<fx>{one(cl, F[5]), one(cn, F[6])};
  return !ck.bad() && fx_mag_ok(mag);
}

// ----------------------------------------------------------------- apply
// u <- Omega u Omega'^{-1}, row by row (each row of Omega u goes straight into
// the second product); with WITH_NORM also Tr u u^+ - 3 as a 60-bit integer.
struct fx_apply_ops {  // Omega as left factors
  fx_left d[3];
  fx_cleft o[3];
};
__device__ __forceinline__ void fx_lhs(fx_apply_ops& L, const fx_herm& h) {
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    L.d[q] = fx_lhs(h.d[q]);
    L.o[q] = fx_lhs(h.o[q]);
  }
}
__device__ __forceinline__ fx_cleft fx_conj(const fx_cleft& a) { return fx_cleft{a.re, a.nim, a.im}; }
template <bool WITH_NORM>
__device__ __forceinline__ void fx_apply_link(mat<fx>& u, const fx_apply_ops& L, const fx_herm& oi, fx_chk& ck, long long& dev) {
  fx_rmat y;
  fx_rhs(y, u);
  fx_right rd[3], ro[3][3];  // Omega'^{-1} as right factors: re, im, -im
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    rd[q] = fx_rhs(oi.d[q]);
    ro[q][0] = fx_rhs(oi.o[q].re);
    ro[q][1] = fx_rhs(oi.o[q].im);
    ro[q][2] = fx_rhs(-oi.o[q].im);
  }
  fx_acc n = fx_zero();
  float nf = 0.0f;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    fx_cleft t[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      fx_acc re = fx_zero(), im = fx_zero();
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        if (k == i) {
          fx_mac(re, L.d[i], y.e[3 * k + j].re);
          fx_mac(im, L.d[i], y.e[3 * k + j].im);
        } else {
          const int q = i + k - 1;  // 01 -> 0, 02 -> 1, 12 -> 2
          fx_cmac(re, im, k > i ? L.o[q] : fx_conj(L.o[q]), y.e[3 * k + j]);
        }
      }
      t[j] = fx_lhs(cx<fx>{fx_get<FX_WIDE>(re, ck), fx_get<FX_WIDE>(im, ck)});
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      fx_acc re = fx_zero(), im = fx_zero();
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        if (k == j) {
          fx_mac(re, t[k].re, rd[j]);
          fx_mac(im, t[k].im, rd[j]);
        } else {  // element (k, j): o_kj for k < j, conj(o_jk) for k > j
          const int q = j + k - 1, c = k < j ? 1 : 2;
          fx_mac(re, t[k].re, ro[q][0]);
          fx_mac(re, t[k].nim, ro[q][c]);
          fx_mac(im, t[k].re, ro[q][c]);
          fx_mac(im, t[k].im, ro[q][0]);
        }
      }
      const cx<fx> r = {fx_get<FX_WIDE>(re, ck), fx_get<FX_WIDE>(im, ck)};
      u.e[3 * i + j] = r;
      if (WITH_NORM) {
        fx_mac(n, fx_lhs(r.re), fx_rhs(r.re));
        fx_mac(n, fx_lhs(r.im), fx_rhs(r.im));
        const float a = (float)r.re.h, b = (float)r.im.h;
        nf = fmaf(a, a, fmaf(b, b, nf));
      }
    }
  }
  if (WITH_NORM) {
    dev += fx_sum(n) - ((3ll << 60) + (1 << 29));
    if (!(nf < 4.9f * 0x1p60f)) ck.fail();  // the sum of four deviations must fit
  }
}

}  // namespace clgc
