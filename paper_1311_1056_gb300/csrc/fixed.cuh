// fixed.cuh -- 60-bit fixed-point 3x3 complex algebra on the integer and FP32
// pipes, the arithmetic of the FP64 form's matrix products.
//
// Why: GB300 issues 2 FP64 multiply-adds per SM and clock.  Links, plaquettes
// and everything the CL step derives from them are numbers of order one, which
// is what fixed point is for.  A number is
//   x = (h 2^30 + l) 2^-60,   h an int, l a float (an integer, |l| <= 2^29),
// and a product splits by size:
//   x y = h h' 2^-60 + (h l' + l h') 2^-90 + l l' 2^-120.
// The first term is exact in 64 bits (IMAD.WIDE) and sums without rounding;
// the second is below 2^-30 of the first, so float (one packed FFMA2 for its
// two products) carries it to ~2^-56; the third is below 2^-62 and dropped.
// A 3x3 product takes ~1,390 cycles of a scheduler and warp against ~7,500 in
// FP64 (and 1,870 with both limbs integers), and its error is smaller: rms
// 2.4e-17 against 3.6e-17 for random SU(3) factors, 4.8e-17 against 7.2e-17
// after four products (FP64 rounds each of its six partial sums).
//
// Ranges.  |x| < FX_BOUND = 1.4375 holds for every operand and stored number:
// a sum of six products and one summand then stays below 16 - FX_BOUND, and
// as sums wrap at 16 a result that is out of bounds cannot look as if it were
// in.  Every result is checked (fx_chk).  A matrix that does not fit (a
// runaway field, NaN) is stored as plain doubles instead, marked in its first
// word (fx_is_raw); a thread that meets one, or whose own results do not fit,
// redoes its work in FP64 (the general path).
#pragma once
#include "su3.cuh"

namespace clgc {

// a b + c and a b.  Written in C++ the sums of products are reassociated and
// cost twice the instructions.
__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}
typedef unsigned long long fx_pair;  // two packed floats
__device__ __forceinline__ fx_pair fx_pack(float a, float b) {
  fx_pair r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ fx_pair fx_fma2(fx_pair a, fx_pair b, fx_pair c) {
  fx_pair r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

__device__ __forceinline__ fx_pair fx_neg(fx_pair a) { return a ^ 0x8000000080000000ull; }

// Range check: the largest of the results' high words, offset to be unsigned.
// WIDE: |x| < 1.4375; NARROW: |x| < 0.359375, for results that are multiplied by
// four; MID: |x| < 1, for results that are added to others (a sum below 2.5625
// cannot wrap into the bound of WIDE).
enum { FX_WIDE = 0, FX_NARROW = 1, FX_MID = 2 };
struct fx_chk {
  unsigned m0, m1, m2;
  __device__ __forceinline__ fx_chk() : m0(0), m1(0), m2(0) {}
  template <int B>
  __device__ __forceinline__ void see(int hi) {  // hi: units of 2^-28
    if (B == FX_WIDE)
      m0 = max(m0, (unsigned)hi + 0x17000000u);
    else if (B == FX_NARROW)
      m1 = max(m1, (unsigned)hi + 0x05C00000u);
    else
      m2 = max(m2, (unsigned)hi + 0x10000000u);
  }
  __device__ __forceinline__ void fail() { m0 = 0xffffffffu; }
  __device__ __forceinline__ bool bad() const { return m0 >= 0x2E000000u || m1 >= 0x0B800000u || m2 >= 0x20000000u; }
};

__device__ __forceinline__ fx operator-(fx a) { return fx{-a.l, -a.h}; }
__device__ __forceinline__ fx operator+(fx a, fx b) { return fx{a.l + b.l, a.h + b.h}; }
__device__ __forceinline__ fx operator-(fx a, fx b) { return fx{a.l - b.l, a.h - b.h}; }
__device__ __forceinline__ fx fx_twice(fx a) { return fx{2.0f * a.l, 2 * a.h}; }
// a + SIGN b with the low limb brought back below 2^29 (the carry by rounding the
// limbs' sum to a multiple of 2^30), so that nothing is lost in it.
template <int SIGN>
__device__ __forceinline__ fx fx_sum_of(fx a, fx b) {
  const float bl = SIGN > 0 ? b.l : -b.l;
  const float r = (a.l + bl) + 0x1.8p53f, c = r - 0x1.8p53f;
  return fx{fmaf(-0.5f, c, a.l) + fmaf(-0.5f, c, bl), a.h + SIGN * b.h + (__float_as_int(r) - __float_as_int(0x1.8p53f))};
}

// The 60-bit integer of a number, and back.
__device__ __forceinline__ long long fx_bits(fx a) { return mad_wide(a.h, 1 << 30, (long long)__float2int_rn(a.l)); }
// r carries an offset of 2^29, which makes the truncating split a balanced one.
__device__ __forceinline__ fx fx_split(long long r) {
  return fx{(float)(((int)r & ((1 << 30) - 1)) - (1 << 29)), (int)(r >> 30)};
}
__device__ __forceinline__ fx fx_of_bits(long long v) { return fx_split(v + (1 << 29)); }

// Operands: left factors carry (h, l) as floats, right factors (l, h).
struct fx_left {
  int h;
  fx_pair p;
};
struct fx_right {
  int h;
  fx_pair p;
};
__device__ __forceinline__ fx_left fx_lhs(fx a) { return fx_left{a.h, fx_pack((float)a.h, a.l)}; }
__device__ __forceinline__ fx_left fx_lhs_neg(fx a) { return fx_left{-a.h, fx_pack(-(float)a.h, -a.l)}; }
__device__ __forceinline__ fx_right fx_rhs(fx a) { return fx_right{a.h, fx_pack(a.l, (float)a.h)}; }
struct fx_cleft {
  fx_left re, im, nim;  // nim = -im
};
struct fx_cright {
  fx_right re, im;
};
__device__ __forceinline__ fx_cleft fx_lhs(cx<fx> a) { return fx_cleft{fx_lhs(a.re), fx_lhs(a.im), fx_lhs_neg(a.im)}; }
__device__ __forceinline__ fx_cleft fx_lhs_neg(cx<fx> a) { return fx_cleft{fx_lhs_neg(a.re), fx_lhs_neg(a.im), fx_lhs(a.im)}; }
__device__ __forceinline__ fx_cright fx_rhs(cx<fx> a) { return fx_cright{fx_rhs(a.re), fx_rhs(a.im)}; }

// Accumulator of a sum of products: a in units of 2^-60, c (two partial sums) of 2^-90.
struct fx_acc {
  long long a;
  fx_pair c;
};
// The same with less rounding, for the link inverses, plaquettes and clover field, whose
// errors all later results inherit: twice as many partial sums, added as integers.
// An element of a 3x3 product is off by 1.5e-17 (rms) in place of 2.0e-17, of a
// product-accumulate by 1.5e-17 in place of 2.7e-17; charge density on thermalised links
// 5.1e-16 -> 4.4e-16 of its size (FP64 arithmetic 4.5e-16), for plaquettes and clover
// field of a 32^4 step 2.45 -> 2.59 ms, observables 2.89 -> 3.03.
struct fx_acc_fine {
  long long a;
  fx_pair c, d;
};
template <typename A = fx_acc>
__device__ __forceinline__ A fx_zero() { return A{}; }
// S: the summand times 2^-S
template <int S = 0>
__device__ __forceinline__ fx_acc fx_from(fx c) {
  return fx_acc{mad_wide(c.h, 1 << (30 - S), 0), fx_pack(c.l * (float)(1 << (30 - S)), 0.0f)};
}
__device__ __forceinline__ void fx_mac(fx_acc& s, const fx_left& x, const fx_right& y) {
  s.a = mad_wide(x.h, y.h, s.a);
  s.c = fx_fma2(x.p, y.p, s.c);
}
__device__ __forceinline__ void fx_cmac(fx_acc& re, fx_acc& im, const fx_cleft& a, const fx_cright& b) {
  fx_mac(re, a.re, b.re);
  fx_mac(im, a.re, b.im);
  fx_mac(re, a.nim, b.im);
  fx_mac(im, a.im, b.re);
}
__device__ __forceinline__ void fx_cmac(fx_acc_fine& re, fx_acc_fine& im, const fx_cleft& a, const fx_cright& b) {
  re.a = mad_wide(a.nim.h, b.im.h, mad_wide(a.re.h, b.re.h, re.a));
  im.a = mad_wide(a.im.h, b.re.h, mad_wide(a.re.h, b.im.h, im.a));
  re.c = fx_fma2(a.re.p, b.re.p, re.c);
  im.c = fx_fma2(a.re.p, b.im.p, im.c);
  re.d = fx_fma2(a.nim.p, b.im.p, re.d);
  im.d = fx_fma2(a.im.p, b.re.p, im.d);
}
template <typename A, int S>
__device__ __forceinline__ A fx_start(fx c) {
  if constexpr (sizeof(A) == sizeof(fx_acc))
    return fx_from<S>(c);
  else
    return A{mad_wide(c.h, 1 << (30 - S), (long long)__float2int_rn(c.l * (1.0f / (1 << S)))), 0ull, 0ull};
}
__device__ __forceinline__ int fx_small(fx_pair c) {
  float c0, c1;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(c0), "=f"(c1) : "l"(c));
  return __float2int_rn(c0 * 0x1p-33f) + __float2int_rn(c1 * 0x1p-33f);
}
__device__ __forceinline__ long long fx_sum(const fx_acc_fine& s) {
  return mad_wide(fx_small(s.c) + fx_small(s.d) + (1 << 26), 8, s.a);
}
// The sum as a 60-bit integer with an offset of 2^29: the small terms are
// rounded to 2^-57 (in range for any operands within bounds) and folded in.
// LONG: sums of up to 48 products (rounded to 2^-56).
template <bool LONG = false>
__device__ __forceinline__ long long fx_sum(const fx_acc& s) {
  float c0, c1;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(c0), "=f"(c1) : "l"(s.c));
  return LONG ? mad_wide(__float2int_rn((c0 + c1) * 0x1p-34f) + (1 << 25), 16, s.a)
              : mad_wide(__float2int_rn((c0 + c1) * 0x1p-33f) + (1 << 26), 8, s.a);
}
// The result times 2^-S, within bound B.
template <int B, int S = 0, typename A>
__device__ __forceinline__ fx fx_get(const A& s, fx_chk& ck) {
  long long r = fx_sum(s);
  if (S) r = (r >> S) + ((1 << 29) - (1 << (29 - S)));
  ck.see<B>((int)(r >> 32));
  return fx_split(r);
}

// The products run row by row in a rolled loop, the rows of the operands
// passing through the same registers (rotated by one row each time, so that no
// register is indexed): unrolled, the theta force is 120 KB of code and its
// warps wait on instruction fetch (12.5 against 8.6 ms per 32^4 step with
// integer limbs).
__device__ __forceinline__ void fx_rotate(mat<fx>& a, const cx<fx>* last) {
#pragma unroll
  for (int k = 0; k < 6; ++k) a.e[k] = a.e[k + 3];
#pragma unroll
  for (int k = 0; k < 3; ++k) a.e[6 + k] = last[k];
}
struct fx_rmat {
  fx_cright e[9];
};
__device__ __forceinline__ void fx_rhs(fx_rmat& r, const mat<fx>& b) {
#pragma unroll
  for (int k = 0; k < 9; ++k) r.e[k] = fx_rhs(b.e[k]);
}
// a <- 2^-S a b
template <int B, int S = 0, typename A = fx_acc>
__device__ __forceinline__ void fx_mul_left(mat<fx>& a, const mat<fx>& b, fx_chk& ck) {
  fx_rmat y;
  fx_rhs(y, b);
#pragma unroll 1
  for (int i = 0; i < 3; ++i) {
    fx_cleft x[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) x[k] = fx_lhs(a.e[k]);
    cx<fx> r[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      A re = fx_zero<A>(), im = fx_zero<A>();
#pragma unroll
      for (int k = 0; k < 3; ++k) fx_cmac(re, im, x[k], y.e[3 * k + j]);
      r[j] = cx<fx>{fx_get<B, S>(re, ck), fx_get<B, S>(im, ck)};
    }
    fx_rotate(a, r);
  }
}
// c <- 2^-S c + a b (SIGN > 0) or 2^-S c - a b.  Here and in fx_adj the rows
// (columns) of a have gone round once at the end: a is what it was, without a
// second copy.
template <int B, int SIGN, int S = 0, typename A = fx_acc>
__device__ __forceinline__ void fx_mul_acc(mat<fx>& c, mat<fx>& a, const mat<fx>& b, fx_chk& ck) {
  fx_rmat y;
  fx_rhs(y, b);
#pragma unroll 1
  for (int i = 0; i < 3; ++i) {
    cx<fx> r[3];
    fx_cleft x[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) x[k] = SIGN < 0 ? fx_lhs_neg(a.e[k]) : fx_lhs(a.e[k]);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      A re = fx_start<A, S>(c.e[j].re), im = fx_start<A, S>(c.e[j].im);
#pragma unroll
      for (int k = 0; k < 3; ++k) fx_cmac(re, im, x[k], y.e[3 * k + j]);
      r[j] = cx<fx>{fx_get<B>(re, ck), fx_get<B>(im, ck)};
    }
    fx_rotate(c, r);
    const cx<fx> z[3] = {a.e[0], a.e[1], a.e[2]};
    fx_rotate(a, z);
  }
}
// r = s a, s real
template <int B>
__device__ __forceinline__ void fx_scaled(mat<fx>& r, const mat<fx>& a, fx s, fx_chk& ck) {
  const fx_left x = fx_lhs(s);
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    fx_acc re = fx_zero(), im = fx_zero();
    fx_mac(re, x, fx_rhs(a.e[k].re));
    fx_mac(im, x, fx_rhs(a.e[k].im));
    r.e[k] = cx<fx>{fx_get<B>(re, ck), fx_get<B>(im, ck)};
  }
}
// c += [a, b]
template <int B>
__device__ __forceinline__ void fx_commutator_acc(mat<fx>& c, mat<fx>& a, mat<fx>& b, fx_chk& ck) {
  fx_mul_acc<B, +1>(c, a, b, ck);
  fx_mul_acc<B, -1>(c, b, a, ck);
}
// c = [a, b] + s a, s real
template <int B>
__device__ __forceinline__ void fx_commutator(mat<fx>& c, mat<fx>& a, mat<fx>& b, fx s, fx_chk& ck) {
  fx_scaled<B>(c, a, s, ck);
  fx_commutator_acc<B>(c, a, b, ck);
}

// Adjugate (the inverse of a matrix of determinant one): row i of r from
// columns i + 1 and i + 2 of a, which rotate through the same registers.
template <typename A = fx_acc>
__device__ __forceinline__ void fx_adj(mat<fx>& r, mat<fx>& a, fx_chk& ck) {
#pragma unroll 1
  for (int i = 0; i < 3; ++i) {
    cx<fx> row[3];
    fx_cright u[3], v[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      u[j] = fx_rhs(a.e[3 * j + 1]);
      v[j] = fx_rhs(a.e[3 * j + 2]);
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int j1 = (j + 1) % 3, j2 = (j + 2) % 3;
      A re = fx_zero<A>(), im = fx_zero<A>();
      fx_cmac(re, im, fx_lhs(a.e[3 * j1 + 1]), v[j2]);
      fx_cmac(re, im, fx_lhs_neg(a.e[3 * j1 + 2]), u[j2]);
      row[j] = cx<fx>{fx_get<FX_WIDE>(re, ck), fx_get<FX_WIDE>(im, ck)};
    }
    fx_rotate(r, row);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const cx<fx> z = a.e[3 * j];
      a.e[3 * j] = a.e[3 * j + 1];
      a.e[3 * j + 1] = a.e[3 * j + 2];
      a.e[3 * j + 2] = z;
    }
  }
}

// c <- c + SIGN a, |a| < 1
template <int SIGN>
__device__ __forceinline__ void fx_add_to(mat<fx>& c, const mat<fx>& a, fx_chk& ck) {
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    c.e[k] = cx<fx>{fx_sum_of<SIGN>(c.e[k].re, a.e[k].re), fx_sum_of<SIGN>(c.e[k].im, a.e[k].im)};
    ck.see<FX_WIDE>(c.e[k].re.h >> 2);
    ck.see<FX_WIDE>(c.e[k].im.h >> 2);
  }
}
// a <- 2^k a
__device__ __forceinline__ void fx_shift_up(mat<fx>& a, int k) {
#pragma unroll
  for (int q = 0; q < 9; ++q) a.e[q] = cx<fx>{fx_of_bits(fx_bits(a.e[q].re) << k), fx_of_bits(fx_bits(a.e[q].im) << k)};
}
// c <- (c + a) / 4
__device__ __forceinline__ void fx_quarter_sum(mat<fx>& c, const mat<fx>& a) {
#pragma unroll
  for (int k = 0; k < 9; ++k)
    c.e[k] = cx<fx>{fx_of_bits((fx_bits(c.e[k].re) + fx_bits(a.e[k].re)) >> 2), fx_of_bits((fx_bits(c.e[k].im) + fx_bits(a.e[k].im)) >> 2)};
}
// ---------------------------------------------------------- conversions
// Double to fixed point, rounded to nearest (ties away).  Only |x| < 2 has an
// image; `mag` collects the magnitudes' high words for the caller's check.
__device__ __forceinline__ long long fx_bits_of_double(double x, unsigned& mag) {
  const int hi = __double2hiint(x);
  const unsigned lo = (unsigned)__double2loint(x);
  mag = max(mag, (unsigned)hi & 0x7fffffffu);
  const int e = (hi >> 20) & 0x7ff;
  // significand with its leading one at bit 62; x 2^60 = m 2^(e - 1025)
  const unsigned mh = (__funnelshift_l(lo, (unsigned)hi, 10) & 0x3fffffffu) | 0x40000000u;
  const unsigned long long m = ((unsigned long long)mh << 32) | (lo << 10);
  const int r = max(min(1024 - e, 63), 0);
  const long long v = (long long)(((m >> r) + 1) >> 1);
  const long long s = (long long)(hi >> 31);
  return (v ^ s) - s;
}
__device__ __forceinline__ fx fx_of_double(double x, unsigned& mag) { return fx_of_bits(fx_bits_of_double(x, mag)); }
// Whether the largest magnitude seen is below FX_BOUND (false for NaN and Inf).
__device__ __forceinline__ bool fx_mag_ok(unsigned mag) { return mag < 0x3FF70000u; }  // 1.4375

// x 2^n on the integer pipe; zero below the smallest normal number.
__device__ __forceinline__ double fx_pow2(double x, int n) {
  const int hi = __double2hiint(x), e = (hi >> 20) & 0x7ff;
  if (e == 0x7ff) return x;
  if (e == 0 || e + n <= 0) return 0.0;
  return e + n >= 0x7ff ? __hiloint2double((hi & 0x80000000) | 0x7ff00000, 0) : __hiloint2double(hi + n * (1 << 20), __double2loint(x));
}
// A complex constant below one, times 2^t so that its larger part is in [1/2, 1):
// a small one keeps its 53 bits (down to 2^-32; what it multiplies is then below
// the numbers' resolution).
struct fx_cscale {
  fx_cleft m;
  int t;
  bool imag;  // real part zero
  // (re + i im) 2^up
  __device__ __forceinline__ fx_cscale(double re, double im, int up, unsigned& mag) {
    const int e = max((__double2hiint(re) >> 20) & 0x7ff, (__double2hiint(im) >> 20) & 0x7ff);
    t = max(0, min(31, 1022 - up - e));
    imag = re == 0.0;
    m = fx_lhs(cx<fx>{fx_of_double(fx_pow2(re, up + t), mag), fx_of_double(fx_pow2(im, up + t), mag)});
  }
};
// a <- s a
template <int B>
__device__ __forceinline__ void fx_cscaled(mat<fx>& a, const fx_cscale& s, fx_chk& ck) {
  const long long up = (1ll << 29) - (1ll << (29 - min(s.t, 29)));
  const auto get = [&](const fx_acc& x, bool see) {
    const long long r = fx_sum(x);  // offset by 2^29
    const int hi = (int)(r >> 32), w = hi >> s.t;
    if (see) ck.see<B>(w);
    return fx_split((long long)(((unsigned long long)(unsigned)w << 32) | __funnelshift_r((unsigned)r, (unsigned)hi, s.t)) + up);
  };
  if (s.imag) {  // theta real
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      fx_acc re = fx_zero(), im = fx_zero();
      fx_mac(re, s.m.nim, fx_rhs(a.e[k].im));
      fx_mac(im, s.m.im, fx_rhs(a.e[k].re));
      a.e[k] = cx<fx>{get(re, false), get(im, false)};  // no larger than a
    }
  } else {
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      fx_acc re = fx_zero(), im = fx_zero();
      fx_cmac(re, im, s.m, fx_rhs(a.e[k]));
      a.e[k] = cx<fx>{get(re, true), get(im, true)};
    }
  }
}

// v 2^(e - 60) as a double, rounded to nearest even.
__device__ __forceinline__ double fx_bits_to_double(long long v, int e = 0) {
  const unsigned long long s = (unsigned long long)(v >> 63);
  const unsigned long long m = ((unsigned long long)v ^ s) - s;
  const int lz = __clzll((long long)m);
  const unsigned long long n = m << (lz & 63);
  unsigned long long q = n >> 11;
  const unsigned rem = (unsigned)n & 0x7ffu;
  q += (rem + ((unsigned)q & 1u)) > 0x400u ? 1u : 0u;
  q += (unsigned long long)(1023 + 63 - 60 - 1 + e - lz) << 52;
  q = m ? q : 0ull;
  return __longlong_as_double((long long)(q | (s << 63)));
}
__device__ __forceinline__ double fx_to_double(fx a, int e = 0) { return fx_bits_to_double(fx_bits(a), e); }

// The power of two k that the clover field is kept at: the largest with 2^k times
// the lattice's largest D / 2 below the bound.  (top: its high limb, which the
// plaquette pass has left.)  The field's sums then add little to the error that D
// itself has as a difference of P and P^{-1}, for smooth links too: with k = 0 the
// charge density of links within 0.03 of one is off by 2.6e-15, within 1e-3 by
// 6.1e-13; so by 1.2e-15 and 2.7e-14; FP64 arithmetic 1.4e-15 and 4.8e-14.
__device__ __forceinline__ int fx_field_shift(const unsigned* top) {
  const unsigned m = *top;
  const int k = max(0, __clz((int)m) - 2);
  return min(24, k + (m << k < 0x2E000000u ? 1 : 0));  // 1.4375 / 2
}

// -------------------------------------------------- stored 64-bit words
// A matrix is stored as fixed-point words (l, h) or, all 18 of them, as
// doubles.  Which one it is shows in its first word alone: l of a stored
// number is below 2^31 in magnitude; the first double is stored times 2^400,
// its high word first, which read as a float is above.  Doubles outside
// 2^-150 .. 2^500 are stored there as 2^-150 and NaN (one has lost all meaning
// next to the entries of a matrix of determinant one, the other overflows in
// the next product).
__device__ __forceinline__ bool fx_is_raw(float l) { return (__float_as_uint(l) & 0x7fffffffu) >= 0x4F000000u; }
__device__ __forceinline__ float fx_raw_mark() { return __uint_as_float(0x7ff80000u); }

__device__ __forceinline__ void fx_load(mat<fx>& a, const int4* __restrict__ f, int plane, int site, int V, fx_chk& ck) {
  load<fx>(a, f, plane, site, V);
  if (fx_is_raw(a.e[0].re.l)) ck.fail();
}

// Matrices on their way from memory: each thread copies those that it will need
// next into slots of shared memory (cp.async) while it works on the last one.
// Three warps per scheduler do not hide a load of 144 bytes (a quarter of a
// warp's time), and registers to load ahead are not there.  A slot is a
// thread's own: element k of slot q at sm[(9 q + k) FX_PIPE_THREADS + thread],
// no barrier.  With two slots `in` and `out` are constants of unrolled code.
const int FX_PIPE_THREADS = 128;
template <int SLOTS>
struct fx_pipe {
  static const int WORDS = SLOTS * 9 * FX_PIPE_THREADS;  // int4
  int4* sm;
  int in, out;  // matrices asked for and taken
  __device__ __forceinline__ explicit fx_pipe(int4* s) : sm(s + threadIdx.x), in(0), out(0) {}
  __device__ __forceinline__ void ask(const int4* f, int plane, int site, int V) {
    const int4* p = f + (size_t)plane * 9 * V + site;
    const unsigned d = (unsigned)__cvta_generic_to_shared(sm + (in & (SLOTS - 1)) * 9 * FX_PIPE_THREADS);
#pragma unroll
    for (int k = 0; k < 9; ++k)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d + k * FX_PIPE_THREADS * 16), "l"(p + (size_t)k * V) : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
    ++in;
  }
  __device__ __forceinline__ void take(mat<fx>& a, fx_chk& ck) {
    if (SLOTS > 1 && in - out > 1)
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    else
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    const int4* p = sm + (out & (SLOTS - 1)) * 9 * FX_PIPE_THREADS;
#pragma unroll
    for (int k = 0; k < 9; ++k) a.e[k] = unpack(p[k * FX_PIPE_THREADS]);
    if (fx_is_raw(a.e[0].re.l)) ck.fail();
    ++out;
  }
};

// One matrix of a thread set aside in shared memory, laid out as a slot.
struct fx_park {
  static const int WORDS = 9 * FX_PIPE_THREADS;  // int4
  int4* sm;
  __device__ __forceinline__ explicit fx_park(int4* s) : sm(s + threadIdx.x) {}
  __device__ __forceinline__ void put(const mat<fx>& a) const {
#pragma unroll
    for (int k = 0; k < 9; ++k) sm[k * FX_PIPE_THREADS] = pack(a.e[k]);
  }
  __device__ __forceinline__ void get(mat<fx>& a) const {
#pragma unroll
    for (int k = 0; k < 9; ++k) a.e[k] = unpack(sm[k * FX_PIPE_THREADS]);
  }
};

// Plain (coherent) load, for words this kernel also writes; |v| < 1 for a 60-bit integer.
__device__ __forceinline__ void fx_load_plain(mat<fx>& a, const int4* f, int plane, int site, int V) {
  const int4* p = f + (size_t)plane * 9 * V + site;
#pragma unroll
  for (int k = 0; k < 9; ++k) a.e[k] = unpack(p[(size_t)k * V]);
}
__device__ __forceinline__ bool fx_below_one(long long v) { return (unsigned)((int)(v >> 32) + (1 << 28)) < (1u << 29); }

// The first double of a raw matrix, to and from its stored words.
__device__ __forceinline__ int2 fx_raw_first(double x) {
  const double ax = fabs(x);
  if (ax < 0x1p-150) x = 0x1p-150;
  x = ax < 0x1p500 ? x * 0x1p400 : __longlong_as_double(0x7ff8000000000000ll);
  return make_int2(__double2hiint(x), __double2loint(x));
}
__device__ __forceinline__ double fx_raw_first(int2 v) { return __hiloint2double(v.x, v.y) * 0x1p-400; }

// The general path's view of such a field; its numbers are the field's times 2^ex.
// (As a factor in FP64 that power cost as much as a sixth of a product for every
// matrix read or written.)
struct tagged {
  int4* p;
  int ex;
  unsigned lim = 0x3FF70000u;  // stored as words below this (high word of a double; 1.4375)
};
__device__ __forceinline__ void load(mat<double>& a, tagged f, int plane, int site, int V) {
  const int4* p = f.p + (size_t)plane * 9 * V + site;
  const bool raw = fx_is_raw(__int_as_float(p[0].x));
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const int4 v = p[(size_t)k * V];
    if (raw) {
      const double re = k == 0 ? fx_raw_first(make_int2(v.x, v.y)) : __hiloint2double(v.y, v.x), im = __hiloint2double(v.w, v.z);
      a.e[k] = f.ex ? cx<double>{fx_pow2(re, f.ex), fx_pow2(im, f.ex)} : cx<double>{re, im};
    } else {
      const cx<fx> w = unpack(v);
      a.e[k] = cx<double>{fx_to_double(w.re, f.ex), fx_to_double(w.im, f.ex)};
    }
  }
}
// The same times a complex factor (the clover field in the force).
struct tagged_c {
  tagged f;
  cx<double> sc;
};
__device__ __forceinline__ void load(mat<double>& a, tagged_c f, int plane, int site, int V) {
  load(a, f.f, plane, site, V);
#pragma unroll
  for (int k = 0; k < 9; ++k) a.e[k] = cmul(a.e[k], f.sc);
}
// In fixed point where it fits, so that one number out of range does not send
// its readers the same way.
__device__ __forceinline__ void store(tagged f, int plane, int site, int V, const mat<double>& a) {
  int4* p = f.p + (size_t)plane * 9 * V + site;
  unsigned mag = 0;
#pragma unroll
  for (int k = 0; k < 9; ++k)
    mag = max(mag, max((unsigned)__double2hiint(a.e[k].re) & 0x7fffffffu, (unsigned)__double2hiint(a.e[k].im) & 0x7fffffffu));
  const bool fits = (int)(mag >> 20) < 0x7ff && (int)mag - f.ex * (1 << 20) < (int)f.lim;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const double re = f.ex ? fx_pow2(a.e[k].re, -f.ex) : a.e[k].re, im = f.ex ? fx_pow2(a.e[k].im, -f.ex) : a.e[k].im;
    if (fits) {
      p[(size_t)k * V] = pack(cx<fx>{fx_of_double(re, mag), fx_of_double(im, mag)});
    } else {
      const int2 w = k == 0 ? fx_raw_first(re) : make_int2(__double2loint(re), __double2hiint(re));
      p[(size_t)k * V] = make_int4(w.x, w.y, __double2loint(im), __double2hiint(im));
    }
  }
}

}  // namespace clgc
